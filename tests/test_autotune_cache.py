"""CPU: the autotuner's cache belongs to the kernels it was measured on, and the library's defaults are candidates."""
import json

import numpy as np
import pytest
import torch

from paper_2310_03568_gb300 import autotune, build


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    """A cache file, a device name, and timings that a test sets: cost(candidate) of what was selected last."""
    class Tuner:
        path = tmp_path / "tune.json"
        scan, strategy, items, timed = None, None, None, 0
        cost = staticmethod(lambda t: 1.0)

        def restart(self):  # another process: nothing in memory
            autotune._cache = None

    t = Tuner()

    def timed(fn, reps=3):
        t.timed += 1
        return t.cost(t)

    monkeypatch.setenv("ADC_AUTOTUNE_CACHE", str(t.path))
    monkeypatch.setattr(autotune, "_cache", None)
    monkeypatch.setattr(autotune, "_digest", None)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "a GPU")
    monkeypatch.setattr(autotune, "_time", timed)
    monkeypatch.setattr(autotune, "apply_scan", lambda c: setattr(t, "scan", (c["engine"], c["range_tiles"])))
    monkeypatch.setattr(autotune.adcomb, "scan_fwd", lambda op, x, *a: x)
    monkeypatch.setattr(autotune.adcomb, "hist_fwd", lambda *a: (None, None))
    monkeypatch.setattr(autotune.adcomb, "debug_force_hist_strategy", lambda s: setattr(t, "strategy", s))
    monkeypatch.setattr(autotune.adcomb, "debug_set_batched_items", lambda i: setattr(t, "items", i))
    return t


class Problem:
    chunk, smem_bins = 1 << 16, 0
    desc_h = {"n": np.array([1000, 2000]), "m": np.array([10, 20])}

    def set_plan(self, chunk):
        self.chunk = chunk


def test_entries_of_other_kernels_do_not_answer(tuner, monkeypatch):
    x, k, v = torch.zeros(1000), torch.zeros(1000, dtype=torch.int32), torch.zeros(1000)
    # what a cache file held before the keys named the kernels
    tuner.path.write_text(json.dumps({
        "scan|a GPU|lin|torch.float32|n=10": {"engine": 2, "range_tiles": 16},
        "hist|a GPU|max|torch.float32|n=10|m=5": {"strategy": 3},
        "batched|a GPU|count=1|n=12|mmean=4": {"chunk": 1 << 14, "smem_bins": 4096, "items": 1}}))
    tuner.cost = lambda t: 1.0 if t.scan == (0, 0) else 2.0
    assert autotune.tune_scan("lin", x)["engine"] == 0 and tuner.timed == len(autotune.SCAN_CANDIDATES)
    tuner.cost = lambda t: 1.0 if t.strategy == 1 else 2.0
    assert autotune.tune_hist("max", 31, k, v)["strategy"] == 1
    p = Problem()
    tuner.cost = lambda t: 1.0 if (p.chunk, p.smem_bins, t.items) == (1 << 16, 0, 8) else 2.0
    assert autotune.tune_batched(p)["smem_bins"] == 0
    # the same kernels, another process: the entries answer
    done = tuner.timed
    tuner.restart()
    assert autotune.tune_scan("lin", x)["engine"] == 0
    assert autotune.tune_hist("max", 31, k, v)["strategy"] == 1
    autotune.tune_batched(Problem())
    assert tuner.timed == done
    # other kernels: they do not
    tuner.restart()
    monkeypatch.setattr(autotune, "_digest", "other")
    tuner.cost = lambda t: 1.0 if t.scan == (1, 0) else 2.0
    assert autotune.tune_scan("lin", x)["engine"] == 1 and tuner.timed > done


def test_defaults_are_candidates():
    assert 0 in autotune.BATCHED_SMEM_BINS and 1 << 16 in autotune.BATCHED_CHUNKS and 8 in autotune.BATCHED_ITEMS
    assert (0, 0) in autotune.SCAN_CANDIDATES


def test_digest_follows_the_sources(tmp_path, monkeypatch):
    src = tmp_path / "csrc"
    src.mkdir()
    (src / "a.cu").write_text("1")
    (src / "b.cuh").write_text("2")
    monkeypatch.setattr(build, "CSRC", str(src))
    seen = {build.source_digest()}
    (src / "b.cuh").write_text("3")
    seen.add(build.source_digest())
    (src / "c.h").write_text("")
    seen.add(build.source_digest())
    assert len(seen) == 3 and build.source_digest() in seen
