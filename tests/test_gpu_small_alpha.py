"""Small alphas, where every path counts.  The hard sigmoid's dense adjoint, whose walls all have an
adjoint from every leg: against the oracle, at walls around the sweeps' blocks of 8 and their split at
a quarter of the walls, and around one tile of receivers; and its time."""
import numpy as np
import pytest

from parity import assert_grad_close
from paper_2401_11882_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def cuda(*arrays):
    return tuple(torch.tensor(np.asarray(a, np.float32), device="cuda") for a in arrays)


@pytest.mark.parametrize("W,R,K,alpha", [(1, 40, 1, 1.0), (3, 33, 2, 1.0), (8, 32, 2, 3.0), (9, 65, 2, 1.0),
                                         (33, 31, 1, 2.0), (5, 1, 3, 1.0), (4, 34, 3, 0.5)])
def test_gradients(oracle_mod, W, R, K, alpha):
    from paper_2401_11882_gb300 import ops
    rng = np.random.default_rng([W, R, K])
    sc = scenes.random_small_scene(rng, W, R, K, alpha, "hard_sigmoid")
    g = rng.normal(size=sc.n_rx).astype(np.float32)
    w, t, r, gd = cuda(sc.walls, sc.tx, sc.rx, g)
    s = (K, alpha, "hard_sigmoid")
    ref = oracle_mod.gradient(sc.walls, sc.tx, sc.rx, *s, g, "all")
    runs = [ops.vjp(w, t, r, *s, gd, tile=x) for x in (None, ops.TileConfig(cands_per_unit=1000))]
    for gtx, gw in runs:
        assert_grad_close(gtx.cpu().numpy(), ref[:2], "grad_tx")
        assert_grad_close(gw.cpu().numpy(), ref[2:], "grad_walls")
    again = ops.vjp(w, t, r, *s, gd)   # the TX gradient's bits do not depend on the run
    np.testing.assert_array_equal(again[0].cpu().numpy(), runs[0][0].cpu().numpy())
    # a wavelength above the paths' lengths (at a small alpha reflection points far along a wall's
    # line count, and FP32 lengths of many wavelengths would be most of the difference)
    E, _ = ops.field(w, t, r, *s, 1000.0, 4.0)
    fref = oracle_mod.field_gradient(sc.walls, sc.tx, sc.rx, *s, 1000.0, 4.0, g, "all")
    ftx, fw = ops.field_vjp(w, t, r, *s, 1000.0, 4.0, E, gd)
    assert_grad_close(ftx.cpu().numpy(), fref[:2], "field grad_tx")
    assert_grad_close(fw.cpu().numpy(), fref[2:], "field grad_walls")


def microseconds(fn, rounds=10):
    for _ in range(2):
        fn()
    best = float("inf")
    for _ in range(rounds):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


def test_the_adjoint_of_every_path_takes_under_twelve_forwards():
    """11 forwards before paths were queued, 17 with a sum per leg and wall, 8 with one per wall."""
    from paper_2401_11882_gb300 import ops
    rng = np.random.default_rng(0)
    w, t, r, g = cuda(np.concatenate([scenes.unit_square_walls(), scenes.random_segments(rng, 6)]),
                      [0.4, 0.6], rng.uniform(0.02, 0.98, (20000, 2)), np.ones(20000))
    s = (2, 1.0, "hard_sigmoid")
    forward = microseconds(lambda: ops.forward(w, t, r, *s))
    assert microseconds(lambda: ops.vjp(w, t, r, *s, g)) < 12 * forward


@pytest.mark.parametrize("W,nx,ny,K,alpha", [(1, 1, 1, 1, 1.0), (7, 9, 7, 2, 1.0), (8, 8, 8, 2, 10.0), (9, 5, 13, 3, 10.0),
                                             (17, 26, 25, 2, 30.0), (12, 64, 40, 2, 100.0), (6, 11, 6, 2, 0.0)])
def test_sigmoid_paths_evaluated_without_stages_have_the_same_powers(oracle_mod, W, nx, ny, K, alpha):
    """Tiles near the transmitter for their alpha evaluate every path, the others queue the ones that
    count; the forward that saves visibilities always queues.  Same bits, also where a scene has tiles
    of both kinds (alpha 30 and 100), and the oracle's powers."""
    from parity import assert_power_close
    from paper_2401_11882_gb300 import ops
    rng = np.random.default_rng([W, nx])
    gx, gy = np.meshgrid(np.linspace(0.03, 0.97, nx), np.linspace(0.05, 0.93, ny))
    walls, tx, rx = (np.asarray(a, np.float32) for a in (
        scenes.random_segments(rng, W), [0.41, 0.52], np.stack([gx.ravel(), gy.ravel()], 1)))
    w, t, r = cuda(walls, tx, rx)
    s = (K, alpha, "sigmoid")
    for tile in (dict(), dict(cands_per_unit=7)):
        P = ops.forward(w, t, r, *s, tile=ops.TileConfig(**tile))
        saved = ops.forward_save(w, t, r, *s, tile=ops.TileConfig(save_counting=True, **tile))[0]
        np.testing.assert_array_equal(P.cpu().numpy(), saved.cpu().numpy())
        E, _ = ops.field(w, t, r, *s, 0.3, 4.0, tile=ops.TileConfig(**tile))
        Es, _, _ = ops.field_save(w, t, r, *s, 0.3, 4.0, tile=ops.TileConfig(save_counting=True, **tile))
        np.testing.assert_array_equal(E.cpu().numpy(), Es.cpu().numpy())
    assert_power_close(P.cpu().numpy(), oracle_mod.power(walls, tx, rx, *s))
