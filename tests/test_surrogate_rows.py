"""Surrogate predictions for row counts and shapes at the edge of what they take."""
import ctypes

import pytest

torch = pytest.importorskip("torch")


def test_no_rows_need_no_row_pointers():
    """An empty tensor's address is NULL; nothing is read or launched for it (no GPU)."""
    from paper_2401_11882_gb300 import _lib
    lib = _lib.load()
    p = ctypes.c_void_p(256)   # never read: n is 0, or the call is refused

    def predict(params, x, n, y):
        return _lib.STATUS[lib.drt_mlp_predict(params, p, p, x, n, y, None)]

    assert predict(p, None, 0, None) == "DRT_OK"
    assert predict(None, None, 0, None) == "DRT_ERR_INVALID_ARG"
    assert predict(p, p, -1, p) == "DRT_ERR_INVALID_ARG"
    assert predict(p, None, 1, p) == "DRT_ERR_INVALID_ARG"


@pytest.mark.gpu
def test_predicting_no_rows_gives_an_empty_tensor():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_11882_gb300.surrogate import SurrogateMLP
    m = SurrogateMLP("cuda", batch=64)
    for x in (torch.empty(0, 2, device="cuda"), torch.empty(0, 2)):
        y = m.forward(x)
        assert y.shape == (0,) and y.dtype == torch.float32 and y.is_cuda
