"""A line-of-sight map (no reflections) tests its walls once.  The reflection coefficient does not
enter it; a negative one has no floors of negligible paths, whose own line-of-sight sweep once
doubled the sigmoid's work, so the two signs take the same time.  Measured ratios: 2.0 with the
second sweep, 1.0 without; the limit lies between them, on the best of many repetitions."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def microseconds(fn, reps=20, rounds=5):
    for _ in range(3):
        fn()
    best = float("inf")
    for _ in range(rounds):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / reps * 1e3)
    return best


@pytest.mark.parametrize("call", ["forward", "single_rx", "save", "vjp_tx", "forward3"])
def test_floors_cost_nothing_without_reflections(call):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np
    from paper_2401_11882_gb300 import ops, scenes
    rng = np.random.default_rng(0)
    d = dict(device="cuda", dtype=torch.float32)
    w = scenes.random_segments(rng, 1024)
    walls = torch.tensor(w, **d)
    tx, rx = torch.tensor([0.4, 0.6], **d), torch.tensor(rng.uniform(0, 1, (16384, 2)), **d)
    g = torch.ones(16384, **d)
    tris = torch.tensor(scenes.extrude(w[:256], 0.0, 1.0), **d)
    tx3, rx3 = torch.tensor([0.4, 0.6, 0.5], **d), torch.cat([rx, torch.full_like(rx[:, :1], 0.4)], 1)
    s = (0, 100.0, "sigmoid")
    run = {
        "forward": lambda c: ops.forward(walls, tx, rx, *s, c),
        "single_rx": lambda c: ops.forward(walls, tx, rx, *s, c, tile=ops.TileConfig(single_rx=True)),
        "save": lambda c: ops.forward_save(walls, tx, rx, *s, c),
        "vjp_tx": lambda c: ops.vjp(walls, tx, rx, *s, g, c, wall_grad=False),
        "forward3": lambda c: ops.forward3(tris, tx3, rx3, *s, c),
    }[call]
    assert microseconds(lambda: run(0.5)) < 1.25 * microseconds(lambda: run(-0.5))
