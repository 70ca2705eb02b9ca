"""Scratch of split chunks: a plan says how many chunks it splits, loses its scratch to a
table that needs the room and takes it again, with the results that the caller last
asked for; and user code splits its chunks with the records of whole ones."""
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


def test_plan_info_tells_what_is_split():
    a, b = _tables()
    with zmc.Context(arena_bytes=2 << 20) as c:
        pa = zmc.zmc_plan_create(c.handle, a)
        split, res = [zmc.zmc_plan_info_get(pa)["split_chunks"]], []

        def run():
            zmc.zmc_plan_run(pa)
            res.append(zmc.zmc_plan_results(pa, len(a)))
            split.append(zmc.zmc_plan_info_get(pa)["split_chunks"])

        run()
        pb = zmc.zmc_plan_create(c.handle, b)
        run()
        zmc.zmc_plan_destroy(pb)
        run()
        run()
        assert split == [600, 600, 0, 600, 600]
        for r in res[1:]:
            assert np.array_equal(r["estimate"], res[0]["estimate"])
            assert np.array_equal(r["stderr"], res[0]["stderr"])
        zmc.zmc_plan_destroy(pa)


def test_callers_graph_of_the_stages_replays():
    """Both stages in a graph of the caller's: each replay samples and merges anew."""
    import torch

    a, _ = _tables()
    with zmc.Context(arena_bytes=16 << 20) as c:
        want = zmc.zmc_integrate(c.handle, a)
        pa = zmc.zmc_plan_create(c.handle, a)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=c.stream):
            zmc.zmc_plan_run(pa, zmc.ZMC_STAGE_SAMPLE)
            zmc.zmc_plan_run(pa, zmc.ZMC_STAGE_MERGE)
        for _ in range(2):
            zmc.zmc_plan_run_plain(pa)  # other results in between
            c.stream.synchronize()
            with torch.cuda.stream(c.stream):
                g.replay()
            got = zmc.zmc_plan_results(pa, len(a))
            assert np.array_equal(got["estimate"], want["estimate"])
            assert np.array_equal(got["stderr"], want["stderr"])
        zmc.zmc_plan_run(pa)
        got = zmc.zmc_plan_results(pa, len(a))
        assert np.array_equal(got["estimate"], want["estimate"])
        del g
        zmc.zmc_plan_destroy(pa)


SUM = {zmc.ZMC_UDF_F32: "__device__ float zmc_user_f(const float *x, const float *p) {\n"
                        "  float s = p[0];\n"
                        "  for (int i = 0; i < ZMC_UDF_DIM; ++i) s = fmaf(x[i], x[i], s);\n"
                        "  return s;\n}\n",
       zmc.ZMC_UDF_F64: "__device__ double zmc_user_f(const double *x, const double *p) {\n"
                        "  double s = p[0];\n"
                        "  for (int i = 0; i < ZMC_UDF_DIM; ++i) s = fma(x[i], x[i], s);\n"
                        "  return s;\n}\n"}


def _user_rows(n, dim, samples, func=0):
    t = W.empty(n)
    for i in range(n):
        W.gauss(t[i], 0.25, 1.0, np.zeros(dim), np.full(dim, -0.5), np.full(dim, 1.5), samples,
                77, i)
        t[i]["family"], t[i]["deg"] = W.USER, func
    return t


@pytest.mark.parametrize("precision", [zmc.ZMC_UDF_F32, zmc.ZMC_UDF_F64])
@pytest.mark.parametrize("dim", [1, 5])
def test_user_rows_split_and_whole(zctx, precision, dim):
    """A row alone is split; among 3000 alike rows (12000 chunks, more than the chip keeps
    warps) it is whole."""
    u = zmc.Udf(SUM[precision], dim, precision)
    t = _user_rows(3000, dim, 50003)
    many = u.integrate(zctx.handle, t)
    for i in (0, 1234, 2999):
        one = u.integrate(zctx.handle, t[i:i + 1])
        assert one["estimate"][0] == many["estimate"][i] and one["stderr"][0] == many["stderr"][i]
    u.close()


@pytest.mark.parametrize("precision", [zmc.ZMC_UDF_F32, zmc.ZMC_UDF_F64])
def test_user_row_with_split_and_whole_chunks(zctx, precision):
    """Unlike functions split a launch's last chunks only, here some of the second row's;
    that row alone (12000 alike chunks and more) is whole."""
    u = zmc.Udf([SUM[precision]] * 2, [1, 2], precision)
    n = 16640 * 12000 + 4321
    t = np.concatenate([_user_rows(1, 1, 50003), _user_rows(1, 2, n, 1)])
    both = u.integrate(zctx.handle, t)
    for i in range(2):
        one = u.integrate(zctx.handle, t[i:i + 1])
        assert one["estimate"][0] == both["estimate"][i] and one["stderr"][0] == both["stderr"][i]
    u.close()


def test_fp64_user_samples_are_the_generators_fields(zctx):
    """x of [0, 1) is the 23-bit field over 2^23, exactly."""
    u = zmc.Udf("__device__ double zmc_user_f(const double *x, const double *p) "
                "{ return x[0]; }", 1, zmc.ZMC_UDF_F64)
    t = W.empty(1)
    W.gauss(t[0], 1.0, 1.0, [0.0], [0.0], [1.0], 10**6, 0x123456789ABCDEF0, 9)
    t["family"], t["deg"] = W.USER, 0
    got = u.eval_samples(zctx.handle, t[0], 0, 5000)
    ctr = np.zeros((1000, 4), dtype=np.uint32)
    ctr[:, 0], ctr[:, 1] = 9, np.arange(1000)
    key = np.tile(np.array([[0x9ABCDEF0, 0x12345678]], dtype=np.uint32), (1000, 1))
    w = zmc.zmc_philox4x32_10(zctx.handle, ctr, key).astype(np.uint64).T
    f = np.stack([w[0], (w[0] >> 23) | (w[1] << 9), (w[1] >> 14) | (w[2] << 18), w[2] >> 5,
                  (w[2] >> 28) | (w[3] << 4)], axis=-1) & 0x7FFFFF
    assert np.array_equal(got, (f.reshape(-1) / 2.0**23).astype(np.float32))
    u.close()
