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


class RowReader:
    """Stands in for the library on the CPU: y[i] = 1000 x[i][0] + x[i][1], read from the addresses
    the kernel would read."""

    def __init__(self):
        self.calls = 0

    def drt_mlp_predict(self, params, shadow, freqs, x, n, y, stream):
        self.calls += 1
        rows = (ctypes.c_float * (2 * n)).from_address(x.value)
        out = (ctypes.c_float * n).from_address(y.value)
        for i in range(n):
            out[i] = 1000.0 * rows[2 * i] + rows[2 * i + 1]
        return 0


@pytest.fixture
def surrogate(monkeypatch):
    from paper_2401_11882_gb300 import surrogate as sur
    lib = RowReader()
    monkeypatch.setattr(sur._lib, "load", lambda: lib)
    monkeypatch.setattr(sur, "_stream", lambda device: None)
    m = object.__new__(sur.SurrogateMLP)
    m.device = torch.device("cpu")
    m.params = m.shadow = m.freqs = torch.zeros(4)
    return m, lib


def test_rows_of_two_are_read_where_they_are(surrogate):
    m, _ = surrogate
    base = torch.arange(24, dtype=torch.float32).reshape(6, 4)
    for x in (base[:, :2], base[:, 1:3], base[::2, :2].double(), base.t()[:2].t()):
        assert m.forward(x).tolist() == [1000.0 * a + b for a, b in x.tolist()]


def test_other_shapes_are_broadcast_to_rows_of_two_or_refused(surrogate):
    """The kernel reads two floats a row: a column is spread over both, as assignment to rows of
    two does it; what does not fit raises before any launch.  (x's memory goes on past its rows.)"""
    m, lib = surrogate
    long = torch.arange(64, dtype=torch.float32)
    assert m.forward(long[:5].reshape(5, 1)).tolist() == [1001.0 * i for i in range(5)]
    assert m.forward(long[3:5]).tolist() == [3004.0, 3004.0]   # [2]: one row, for both
    calls = lib.calls
    for bad in (long[:15].reshape(5, 3), long[:5], long[:20].reshape(5, 2, 2)):
        with pytest.raises((RuntimeError, ValueError)):
            m.forward(bad)
    assert lib.calls == calls
