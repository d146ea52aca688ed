"""The forward's autotuner offers the library's own units, and its cache does not outlive the kernels
that its times were taken on (no GPU: the timer and the device name are stand-ins)."""
import json
from types import SimpleNamespace

import pytest

from paper_2401_11882_gb300 import _build, autotune, ops
from paper_2401_11882_gb300.ops import TileConfig

torch = pytest.importorskip("torch")


@pytest.fixture
def tune(tmp_path, monkeypatch):
    """tune(ms): the tile tune_forward picks when ms(tile) is each tile's time."""
    monkeypatch.setenv("DRT_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda device: "GB300")
    monkeypatch.setattr(ops, "forward", lambda *a, tile=None: tile)
    walls, rx = SimpleNamespace(device="cuda", shape=(64, 4)), SimpleNamespace(shape=(4096, 2))

    def run(ms):
        return autotune.tune_forward(walls, None, rx, 2, 100.0, "hard_sigmoid",
                                     timer=lambda fn, reps: ms(fn()))
    return run


def test_the_default_units_are_a_candidate(tune):
    best = tune(lambda t: 1.0 if t.cands_per_unit == 0 else 2.0)
    assert best.cands_per_unit == 0
    # the library's defaults in every field: 8 warps per CTA, CTAs by occupancy, two receivers a lane
    assert TileConfig(warps_per_cta=8) in autotune.FORWARD_CANDIDATES


def test_cached_tiles_are_reused_until_the_kernels_change(tune, monkeypatch, tmp_path):
    first = tune(lambda t: abs(t.cands_per_unit - 32) + t.ctas_per_sm + t.single_rx)
    assert first.cands_per_unit == 32

    def fail(t):
        raise AssertionError("timed again")
    assert tune(fail) == first
    source = tmp_path / "kernel.cu"
    source.write_text("// another kernel")
    monkeypatch.setattr(_build, "_inputs", lambda: [str(source)])
    autotune.kernels.cache_clear()
    assert tune(lambda t: abs(t.cands_per_unit - 64) + t.ctas_per_sm + t.single_rx).cands_per_unit == 64
    autotune.kernels.cache_clear()


def test_a_cache_without_the_kernels_version_is_not_taken(tune, tmp_path):
    old = {"fwd|GB300|hard_sigmoid|K2|W64|R4096": {"tile": {"warps_per_cta": 4, "cands_per_unit": 16}}}
    (tmp_path / "tune.json").write_text(json.dumps(old))
    best = tune(lambda t: abs(t.cands_per_unit - 64) + t.ctas_per_sm + t.single_rx)
    assert best.cands_per_unit == 64
