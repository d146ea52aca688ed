"""The default units of a scene that fills the chip are not slower than given ones: the sigmoid's
forward once took 256 candidates a unit, 1.07 times the time of 64 (its last units left SMs idle); now
1.00.  The limit lies between, on the best of many repetitions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def milliseconds(fn, rounds=8):
    fn()
    best = float("inf")
    for _ in range(rounds):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_sigmoid_forward():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_11882_gb300 import ops, scenes
    rng = np.random.default_rng([3, 128, 16384])
    d = dict(device="cuda", dtype=torch.float32)
    w = torch.tensor(np.concatenate([scenes.unit_square_walls(), scenes.random_segments(rng, 124)]), **d)
    x = np.linspace(0.02, 0.98, 128)
    t = torch.tensor(rng.uniform(0.3, 0.7, 2), **d)
    r = torch.tensor(np.stack(np.meshgrid(x, x), -1).reshape(-1, 2), **d)
    s, given = (2, 100.0, "sigmoid"), ops.TileConfig(cands_per_unit=64)
    assert (milliseconds(lambda: ops.forward(w, t, r, *s))
            < 1.035 * milliseconds(lambda: ops.forward(w, t, r, *s, tile=given)))
