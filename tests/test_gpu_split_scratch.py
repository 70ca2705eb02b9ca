"""Scratch of split chunks that a later table takes: the plan's results stay what the
caller last asked for."""
import numpy as np
import pytest

from paper_2104_10073_gb300 import workloads as W
from paper_2104_10073_gb300 import zmc

pytestmark = pytest.mark.gpu


def _tables():
    rng = np.random.default_rng(5)
    a = W.random_table(40, rng, families=(W.GAUSS,), dims=(1, 7))
    a["n_samples"] = 16640 * 15  # 600 chunks, 1.2 MB of scratch
    b = W.random_table(3000, rng, n_lo=10, n_hi=20, families=(W.POLY,))  # 1.2 MB of descriptors
    return a, b


def test_taking_scratch_back_writes_no_result():
    """A plain run's results, read after another table took the scratch of the sampling
    stage that followed it."""
    a, b = _tables()
    with zmc.Context(arena_bytes=2 << 20) as c:
        pa = zmc.zmc_plan_create(c.handle, a)
        zmc.zmc_plan_run_plain(pa)
        plain = zmc.zmc_plan_results(pa, len(a))
        zmc.zmc_plan_run(pa, zmc.ZMC_STAGE_SAMPLE)
        pb = zmc.zmc_plan_create(c.handle, b)
        got = zmc.zmc_plan_results(pa, len(a))
        assert np.array_equal(got["estimate"], plain["estimate"])
        zmc.zmc_plan_run(pa, zmc.ZMC_STAGE_MERGE)
        batched = zmc.zmc_plan_results(pa, len(a))
        want = zmc.zmc_integrate(c.handle, a)
        assert np.array_equal(batched["estimate"], want["estimate"])
        assert np.array_equal(batched["stderr"], want["stderr"])
        zmc.zmc_plan_destroy(pa)
        zmc.zmc_plan_destroy(pb)
