"""A negative reflection coefficient (paths of one and three reflections count negative) in every
kernel that leaves out negligible paths, against the oracle.

Tolerances: the kernels' error is relative to each path, and the paths' magnitudes are those of the
positive coefficient, so the plain bounds of parity.py are taken of the positive coefficient's
powers (which no cancellation between the orders makes small) and gradients."""
import numpy as np
import pytest

from parity import GRAD_RTOL, POWER_FLOOR, POWER_RTOL
from paper_2401_11882_gb300 import scenes

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GAMMA = -0.5
SIZES = [(1, 6, 70, 30.0), (2, 8, 45, 100.0), (3, 5, 33, 20.0)]   # K, walls, receivers, alpha


@pytest.fixture(scope="module")
def drt():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2401_11882_gb300 as m
    return m


def cuda(*arrays):
    return tuple(torch.tensor(np.asarray(a, np.float32), device="cuda") for a in arrays)


def power_tol(magnitude):
    return POWER_RTOL * (magnitude + POWER_FLOOR * magnitude.max())


def check_power(got, ref, pos):
    # the odd orders are in the sums: without them the powers were (ref + pos) / 2
    assert (np.abs(pos - ref) / 2 > 10 * power_tol(pos)).mean() > 0.5
    np.testing.assert_array_less(np.abs(got.cpu().numpy() - ref), power_tol(pos))


def check_grad(got, ref, pos):
    for i, (a, b, c) in enumerate(zip(got, ref, pos)):
        a, b, c = (np.asarray(x, np.float64).ravel() for x in (a.cpu(), b, c))
        tol = GRAD_RTOL * max(np.linalg.norm(b), np.linalg.norm(c))
        # as above (the transmitter's is that of the nearest lines of sight)
        assert i == 0 or np.linalg.norm(c - b) / 2 > 10 * tol
        assert np.linalg.norm(a - b) <= tol, ("tx", "walls")[i]


def scene2(K, W, R, alpha, smoothing):
    sc = scenes.random_small_scene(np.random.default_rng(10 + K), W, R, K, alpha, smoothing, True)
    return sc, cuda(sc.walls, sc.tx, sc.rx)


@pytest.mark.parametrize("smoothing", ["sigmoid", "hard_sigmoid"])
@pytest.mark.parametrize("K,W,R,alpha", SIZES)
def test_power(drt, oracle_mod, K, W, R, alpha, smoothing):
    from paper_2401_11882_gb300 import ops
    sc, (w, t, r) = scene2(K, W, R, alpha, smoothing)
    ref, pos = (oracle_mod.power(sc.walls, sc.tx, sc.rx, K, alpha, smoothing, c)
                for c in (GAMMA, -GAMMA))
    s = (K, alpha, smoothing, GAMMA)
    for tile in (None, ops.TileConfig(single_rx=True), ops.TileConfig(cands_per_unit=5)):
        check_power(ops.forward(w, t, r, *s, tile=tile), ref, pos)
    if smoothing == "sigmoid":
        for tile in (None, ops.TileConfig(save_counting=True)):
            check_power(ops.forward_save(w, t, r, *s, tile=tile)[0], ref, pos)


@pytest.mark.parametrize("smoothing", ["sigmoid", "hard_sigmoid"])
@pytest.mark.parametrize("K,W,R,alpha", SIZES)
def test_dense_adjoint(drt, oracle_mod, K, W, R, alpha, smoothing):
    from paper_2401_11882_gb300 import ops
    sc, (w, t, r) = scene2(K, W, R, alpha, smoothing)
    g = np.random.default_rng(K).normal(size=sc.n_rx).astype(np.float32)
    ref, pos = (np.split(oracle_mod.gradient(sc.walls, sc.tx, sc.rx, K, alpha, smoothing, g, "all",
                                             c), [2]) for c in (GAMMA, -GAMMA))
    s = (K, alpha, smoothing)
    gd = torch.tensor(g, device="cuda")
    for tile in (None, ops.TileConfig(single_rx=True), ops.TileConfig(cands_per_unit=5)):
        check_grad(ops.vjp(w, t, r, *s, gd, GAMMA, tile=tile), ref, pos)
    check_grad(ops.vjp(w, t, r, *s, gd, GAMMA, wall_grad=False)[:1], ref, pos)
    if smoothing == "sigmoid":
        for tile in (None, ops.TileConfig(save_counting=True)):
            saved = ops.forward_save(w, t, r, *s, GAMMA, tile=tile)[1]
            check_grad(ops.vjp(w, t, r, *s, gd, GAMMA, tile=tile, saved=saved), ref, pos)


@pytest.mark.parametrize("smoothing", ["sigmoid", "hard_sigmoid"])
@pytest.mark.parametrize("K,W,R,alpha", SIZES)
def test_triangles(drt, oracle_mod, K, W, R, alpha, smoothing):
    from paper_2401_11882_gb300 import ops
    if K < 3:   # a room: reflections reach every receiver
        tris = scenes.extrude(np.concatenate([scenes.unit_square_walls(),
                                              [[0.3, 0.2, 0.5, 0.45]]]), 0.0, 1.0)
    else:       # the square's four walls
        tris = scenes.extrude(scenes.unit_square_walls(), 0.0, 1.0)
    rng = np.random.default_rng(K)
    tris, tx, rx, g = (np.asarray(a, np.float32) for a in (
        tris, [0.31, 0.62, 0.45], rng.uniform([0.1, 0.1, 0.2], [0.9, 0.9, 0.8], (R, 3)),
        rng.normal(size=R)))
    w, t, r, gd = cuda(tris, tx, rx, g)
    s = (K, alpha, smoothing)
    ref, pos = (oracle_mod.power3(tris, tx, rx, *s, c) for c in (GAMMA, -GAMMA))
    check_power(ops.forward3(w, t, r, *s, GAMMA), ref, pos)
    gref, gpos = (oracle_mod.gradient3(tris, tx, rx, *s, g, c) for c in (GAMMA, -GAMMA))
    check_grad(ops.vjp3(w, t, r, *s, gd, GAMMA), gref, gpos)
    check_grad([ops.vjp3_tx(w, t, r, *s, gd, GAMMA)], gref, gpos)


@pytest.mark.parametrize("dim", [2, 3])
def test_batch(drt, oracle_mod, dim):
    from paper_2401_11882_gb300.batched import BatchedDescent
    batch = (scenes.scene_batch(4, 1, walls_range=(5, 16), rx_range=(33, 100), orders=(1, 2),
                                n_tx=2, smoothing="sigmoid") if dim == 2 else
             scenes.scene_batch3(4, 1, segments_range=(2, 4), rx_range=(33, 70), orders=(1, 2),
                                 n_tx=2, smoothing="sigmoid"))
    batch.refl_coef = GAMMA
    bd = BatchedDescent(batch)
    lowest = -bd.evaluate().cpu().numpy().astype(np.float64).reshape(batch.n_scenes, 2)
    bd.close()
    power = oracle_mod.power if dim == 2 else oracle_mod.power3
    for i in range(batch.n_scenes):
        for j in range(2):
            sc = batch.scene(i, j)
            walls = sc.walls if dim == 2 else sc.tris
            ref, pos = (power(walls, sc.tx, sc.rx, sc.max_order, 100.0, "sigmoid", c)
                        for c in (GAMMA, -GAMMA))
            tol = power_tol(pos)
            assert (ref - tol).min() <= lowest[i, j] <= (ref + tol).min()
