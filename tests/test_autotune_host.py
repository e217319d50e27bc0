"""Host logic of the autotuner (paper_2104_00537_gb300/autotune.py) on CPU,
with a fake engine whose step time is a known function of the launch choices:
the search takes the fastest (cell size, pair loop), then the fastest block
size of its list walk, restores the cases' cell size, and caches the result
per (GPU, case-count bucket, particle-count bucket)."""
import json

import pytest

from paper_2104_00537_gb300 import autotune


class FakeCase:
    def __init__(self, n):
        self.n = n
        self.params = {"cell_mode": 0}


def cost(cm, var, block):
    base = {(1, 5): 10.0, (1, 4): 12.0, (2, 5): 11.0}.get((cm, var), 20.0 + cm + var)
    return base * {0: 1.0, 128: 1.0, 256: 0.9, 512: 0.95}[block]


class FakeEngine:
    made = []

    def __init__(self, cases):
        self.cm = cases[0].params["cell_mode"]
        self.var, self.block, self.ms = 0, 0, 0.0
        FakeEngine.made.append((self.cm,))

    def set_options(self, pi_variant=-1, pi_block=0, timing=0, **kw):
        self.var, self.block = pi_variant, pi_block

    def step(self, n):
        self.ms += n * cost(self.cm, self.var, self.block)

    def timing(self, reset=False):
        t = {"step_ms": self.ms}
        if reset:
            self.ms = 0.0
        return t

    def destroy(self):
        pass


def test_tune_picks_fastest_configuration_and_block(tmp_path, monkeypatch):
    monkeypatch.setenv("SPH_AUTOTUNE_CACHE", str(tmp_path / "cache.json"))
    cases = [FakeCase(5000), FakeCase(70000)]
    best, times = autotune.tune(cases, FakeEngine, "GB300")
    assert best == (1, 5, 256)
    assert times["1,5,128"] == 10.0 and abs(times["1,5,256"] - 9.0) < 1e-12
    assert all(c.params["cell_mode"] == 0 for c in cases)  # restored
    cached = json.load(open(tmp_path / "cache.json"))
    key = autotune.bucket_key("GB300", cases)
    assert cached[key]["best"] == [1, 5, 256]
    # a second call is served from the cache without building an engine
    FakeEngine.made.clear()
    best2, _ = autotune.tune(cases, FakeEngine, "GB300")
    assert best2 == (1, 5, 256) and FakeEngine.made == []


def test_tune_without_list_skips_block_search(tmp_path, monkeypatch):
    monkeypatch.setenv("SPH_AUTOTUNE_CACHE", str(tmp_path / "cache.json"))
    cases = [FakeCase(1000)]
    best, times = autotune.tune(cases, FakeEngine, "GB300", candidates=[(1, 0), (2, 0)],
                                use_cache=False)
    assert best == (1, 0, 128)
    assert set(times) == {"1,0,128", "2,0,128"}


class FailingEngine(FakeEngine):
    def __init__(self, cases):
        if cases[0].params["cell_mode"] == 2:
            raise RuntimeError("list overflow")
        super().__init__(cases)


def test_configuration_that_cannot_run_is_skipped(tmp_path, monkeypatch):
    monkeypatch.setenv("SPH_AUTOTUNE_CACHE", str(tmp_path / "cache.json"))
    best, times = autotune.tune([FakeCase(1000)], FailingEngine, "GB300",
                                candidates=[(2, 5), (1, 4)], use_cache=False)
    assert times["2,5,128"] == float("inf")
    assert best[:2] == (1, 4)


class RecordingEngine(FakeEngine):
    """Notes the block size of every run under (cell mode, variant)."""
    ran = []

    def step(self, n):
        RecordingEngine.ran.append((self.cm, self.var, self.block))
        super().step(n)


def test_every_entry_is_timed_at_its_own_block(tmp_path, monkeypatch):
    monkeypatch.setenv("SPH_AUTOTUNE_CACHE", str(tmp_path / "cache.json"))
    RecordingEngine.ran.clear()
    _, times = autotune.tune([FakeCase(5000)], RecordingEngine, "GB300")
    assert {"%d,%d,%d" % r for r in RecordingEngine.ran} == set(times)
    assert {"1,5,128", "1,5,256", "1,5,512"} <= set(times)


@pytest.mark.parametrize("pair_once,params", [(1, {}), (0, {"visc_mode": 1}),
                                              (0, {"ddt_mode": 2})])
def test_no_block_search_where_the_walk_has_its_own(tmp_path, monkeypatch, pair_once, params):
    """pi_block is for the default physics' walk of each target's own pairs."""
    monkeypatch.setenv("SPH_AUTOTUNE_CACHE", str(tmp_path / "cache.json"))
    case = FakeCase(5000)
    case.params.update(params)
    best, times = autotune.tune([case], FakeEngine, "GB300", pair_once=pair_once)
    assert best == (1, 5, 128)
    assert all(k.endswith(",128") for k in times)


def test_entries_of_an_earlier_search_are_not_reused(tmp_path, monkeypatch):
    """A cached entry that does not say which block size its first stage ran with."""
    monkeypatch.setenv("SPH_AUTOTUNE_CACHE", str(tmp_path / "cache.json"))
    cases = [FakeCase(5000)]
    key = autotune.bucket_key("GB300", cases)
    (tmp_path / "cache.json").write_text(json.dumps({key: {"best": [0, 4, 128], "times": {}}}))
    best, _ = autotune.tune(cases, FakeEngine, "GB300")
    assert best == (1, 5, 256)
