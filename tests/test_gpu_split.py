"""Launches that hand out chunks by accumulation blocks: the records are those of
whole chunks bit for bit, at the edges of lanes, steps, blocks and chunks, and a
plan's scratch goes back to the arena when another table needs the room."""
import numpy as np
import pytest

from paper_2104_10073_gb300 import workloads as W
from paper_2104_10073_gb300 import zmc

pytestmark = pytest.mark.gpu


def _edges(q):
    """Sizes around quints, steps (160 samples), blocks (13 steps) and chunks."""
    base = [1, 5, 160, 160 * 13, 160 * 13 * max(1, q // 13 - 1), 160 * q, 320 * q]
    return sorted({max(1, b + d) for b in base for d in (-1, 0, 1, 7)})


@pytest.mark.parametrize("q", [14, 26, 104, 208])
def test_split_records_equal_whole_ones(q):
    rng = np.random.default_rng(q)
    sizes = _edges(q)
    t = W.random_table(28 * len(sizes), rng)  # families and dimensions differ: always split
    t["n_samples"] = np.resize(sizes, len(t))
    with zmc.Context(arena_bytes=256 << 20, quints_per_lane=q) as c:
        split = zmc.zmc_integrate(c.handle, t)
    # a serving launch keeps chunks whole
    with zmc.Context(arena_bytes=512 << 20, serving=True, quints_per_lane=q) as c:
        st, whole = zmc.zmc_poll(c.handle, zmc.zmc_submit(c.handle, t), len(t))
    assert st == zmc.ZMC_OK
    for k in ("estimate", "stderr", "n", "status"):
        assert np.array_equal(split[k], whole[k], equal_nan=k == "stderr"), k


def test_one_row_alone_equals_the_row_among_many(zctx):
    """A single row splits, the same row in a table of several waves does not."""
    t = np.repeat(W.abslin_eq2(50003)[60:61], 3000)
    one = zmc.zmc_integrate(zctx.handle, t[:1])
    many = zmc.zmc_integrate(zctx.handle, t)
    assert np.all(many["estimate"] == one["estimate"])
    assert np.all(many["stderr"] == one["stderr"])


def test_scratch_returns_to_the_arena():
    rng = np.random.default_rng(3)
    a = W.random_table(40, rng, families=(W.GAUSS,), dims=(1, 7))
    a["n_samples"] = 16640 * 15  # 600 chunks, 1.2 MB of scratch
    b = W.random_table(3000, rng, n_lo=10, n_hi=20, families=(W.POLY,))  # 1.2 MB of descriptors
    with zmc.Context(arena_bytes=2 << 20) as c:
        pa = zmc.zmc_plan_create(c.handle, a)
        zmc.zmc_plan_run(pa)
        first = zmc.zmc_plan_results(pa, len(a))
        pb = zmc.zmc_plan_create(c.handle, b)
        for p, t in ((pa, a), (pb, b), (pa, a)):
            zmc.zmc_plan_run(p)
            got = zmc.zmc_plan_results(p, len(t))
            assert np.all(got["status"] == 0)
        assert np.array_equal(first["estimate"], got["estimate"])
        assert np.array_equal(first["stderr"], got["stderr"])
        zmc.zmc_plan_destroy(pa)
        zmc.zmc_plan_destroy(pb)


def test_scratch_taken_back_between_the_stages():
    """A sampling stage whose merge comes after another table took the scratch; and
    stages repeated by themselves."""
    rng = np.random.default_rng(4)
    a = W.random_table(40, rng, families=(W.GAUSS,), dims=(1, 7))
    a["n_samples"] = 16640 * 15
    b = W.random_table(3000, rng, n_lo=10, n_hi=20, families=(W.POLY,))
    with zmc.Context(arena_bytes=2 << 20) as c:
        want = zmc.zmc_integrate(c.handle, a)
        pa = zmc.zmc_plan_create(c.handle, a)
        zmc.zmc_plan_run(pa, zmc.ZMC_STAGE_SAMPLE)
        zmc.zmc_plan_run(pa, zmc.ZMC_STAGE_SAMPLE)
        pb = zmc.zmc_plan_create(c.handle, b)
        for stages in ((zmc.ZMC_STAGE_MERGE,), (zmc.ZMC_STAGE_MERGE,), (zmc.ZMC_STAGE_ALL,),
                       (zmc.ZMC_STAGE_SAMPLE, zmc.ZMC_STAGE_ALL)):
            for stage in stages:
                zmc.zmc_plan_run(pa, stage)
            got = zmc.zmc_plan_results(pa, len(a))
            assert np.array_equal(got["estimate"], want["estimate"]), stages
            assert np.array_equal(got["stderr"], want["stderr"]), stages
        zmc.zmc_plan_destroy(pa)
        zmc.zmc_plan_destroy(pb)
