"""The tuners time calls that read their knobs, and leave the others alone."""
import json

import numpy as np
import pytest
import torch

import paper_1907_01063_gb300 as gp
from paper_1907_01063_gb300 import autotune
from test_gpu_batched import make_batch

FP64_IDS = [gp.GPC_TUNE_BLOCK, gp.GPC_TUNE_SPLITK_MIN, gp.GPC_TUNE_F64_SMALL_TILE]


@pytest.fixture
def cache(tmp_path, monkeypatch):
    monkeypatch.setenv("GPCHOL_TUNE_CACHE", str(tmp_path / "tune.json"))
    return tmp_path / "tune.json"


@pytest.fixture
def knobs():
    ids = FP64_IDS + [gp.GPC_TUNE_BATCH_BLOCK]
    saved = [gp.get_tuning(k) for k in ids]
    yield
    for k, v in zip(ids, saved):
        gp.set_tuning(k, v)


def test_records_of_other_routes_are_not_applied(cache, knobs, monkeypatch):
    monkeypatch.setattr(autotune, "_device_key", lambda: "dev")
    cache.write_text(json.dumps({"dev/fp64_block/4096": {"best": 96},
                                 "dev/fp64/8192": {"best": {"fp64_block": 96, "splitk_min": 128, "f64_small_tile": 0}}}))
    before = [gp.get_tuning(k) for k in FP64_IDS]
    assert autotune.apply_cached() == {}
    assert [gp.get_tuning(k) for k in FP64_IDS] == before
    cache.write_text(json.dumps({"dev/fp64_kernels_block/4096": {"best": 64},
                                 "dev/fp64_schedule/8192": {"best": {"splitk_min": 128, "f64_small_tile": 0}}}))
    assert autotune.apply_cached() == {"fp64_block": 64, "splitk_min": 128, "f64_small_tile": 0}
    assert [gp.get_tuning(k) for k in FP64_IDS] == [64, 128, 0]


@pytest.mark.gpu
def test_the_fp64_block_is_timed_on_the_kernels_that_read_it(cache, knobs, monkeypatch):
    seen = []

    def timed(fn, reps=2):
        torch.cuda.synchronize()
        gp.trace_enable(True, timeline=True)
        fn()
        torch.cuda.synchronize()
        gp.trace_enable(False)
        names = [s["kernel"] for s in gp.trace_timeline()]
        seen.append((gp.get_tuning(gp.GPC_TUNE_BLOCK), len(names), any("f64x" in k for k in names)))
        return float(len(seen))

    monkeypatch.setattr(autotune, "_time", timed)
    assert autotune.tune_fp64_block(600, force=True)["best"] == 64  # the first one timed
    assert [b for b, _, _ in seen] == [64, 96, 128] and not any(s for _, _, s in seen)
    assert seen[0][1] != seen[2][1]  # more blocks, more launches
    seen.clear()
    rec = autotune.tune_fp64(1000, force=True)
    assert rec["n"] == 1024 and set(rec["best"]) == {"fp64_block", "splitk_min", "f64_small_tile"}
    assert [s for _, _, s in seen] == [False] * 5 + [True] * 4
    assert autotune.tune_fp64(1000)["when"] == rec["when"]  # from the cache


@pytest.mark.gpu
def test_the_batch_block_is_left_alone_in_lockstep(cache, knobs):
    gp.set_tuning(gp.GPC_TUNE_BATCH_BLOCK, 32)
    for sizes, lockstep in (([300, 140], True), ([40 + i % 30 for i in range(200)], False)):
        Xs, ys, hyps = make_batch(sizes, seed=2)
        b = gp.Batch(sizes)
        X, y = (torch.as_tensor(np.concatenate(v), device="cuda").contiguous() for v in (Xs, ys))
        rec = autotune.tune_batch_block(b, X, y, torch.as_tensor(hyps))
        assert bool(rec.get("lockstep")) == lockstep and cache.exists() != lockstep
        assert gp.get_tuning(gp.GPC_TUNE_BATCH_BLOCK) == rec["best"] and (rec["best"] == 32 or not lockstep)
