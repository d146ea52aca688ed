"""drt_forward_noalloc takes drt_forward's own units where their partial sums fit its fixed scratch
array, so the powers are the same bit for bit; scenes that need larger ones stay within tolerance."""
import ctypes

import numpy as np
import pytest

from parity import assert_power_close
from paper_2401_11882_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def powers(W, R, K, alpha, smoothing):
    """(drt_forward_noalloc's, drt_forward's, workspace bytes of the default units)"""
    from paper_2401_11882_gb300 import _lib, ops
    rng = np.random.default_rng([W, R])
    d = dict(device="cuda", dtype=torch.float32)
    w, t, r = (torch.tensor(a, **d) for a in (scenes.random_segments(rng, W), [0.4, 0.6],
                                              rng.uniform(0.02, 0.98, (R, 2))))
    sc, keep = ops.make_scene(w, t, r, K, alpha, smoothing, 0.5)
    need = ctypes.c_size_t()
    _lib.call("drt_forward_workspace_size", ctypes.byref(sc), None, ctypes.byref(need))
    out = torch.full((R,), float("nan"), device="cuda")
    _lib.call("drt_forward_noalloc", ctypes.byref(sc), out.data_ptr(),
              torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy(), ops.forward(w, t, r, K, alpha, smoothing).cpu().numpy(), need.value


@pytest.fixture(scope="module", autouse=True)
def device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("smoothing", ["hard_sigmoid", "step", "sigmoid"])
@pytest.mark.parametrize("W,R,K", [(5, 16, 1), (40, 33, 2), (1000, 300, 1), (1500, 65, 1), (6, 1, 3)])
def test_same_units_where_they_fit(W, R, K, smoothing):
    got, want, need = powers(W, R, K, 60.0, smoothing)
    assert need <= 8 << 20
    np.testing.assert_array_equal(got, want)


def test_fewer_units_where_they_do_not_fit():
    got, want, need = powers(100, 65600, 2, 60.0, "hard_sigmoid")   # 40 sums a receiver: 10.5 MB
    assert need > 8 << 20
    assert_power_close(got, want)
