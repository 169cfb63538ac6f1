"""The shared-memory GROUP BY table at its limits: values on both sides of a block's window (int64
ranges, float exponents), zeros, subnormals and extremes, blocks of more rows than the packed count
word holds, full tables; unpartitioned, partitioned and batched builds against the CPU oracle."""
import numpy as np
import pytest
import torch

import datagen as dg
import paper_2606_10030_gb300 as agg
from tests.test_gpu_groupby import check_groups, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    agg.build()
    agg.lib()


def values(kind, n, seed=0):
    rng = np.random.default_rng(seed)
    if kind == "i64_around_zero":
        return rng.integers(-1000, 1000, n)
    if kind == "i64_two_windows":
        return rng.integers(0, 2 ** 32, n) + (rng.integers(0, 8, n) == 0) * (np.int64(1) << 40)
    if kind == "i64_extremes":
        v = rng.integers(-(2 ** 63), 2 ** 63 - 1, n, dtype=np.int64)
        v[::5], v[1::7] = -(2 ** 63), 2 ** 63 - 1
        return v
    if kind == "i64_top":
        return np.int64(2 ** 63 - 1) - rng.integers(0, 2 ** 20, n)
    if kind == "i32_negative":
        return rng.integers(-(2 ** 31), 0, n, dtype=np.int64).astype(np.int32)
    if kind == "u32_large":
        return rng.integers(2 ** 31, 2 ** 32, n, dtype=np.uint64).astype(np.uint32)
    f = np.float32 if kind.startswith("f32") else np.float64
    x = rng.standard_normal(n)
    if kind.endswith("wide"):  # most rows outside any window
        return (x * 2.0 ** rng.integers(-60, 60, n)).astype(f)
    if kind.endswith("zeros"):
        x[::2] = 0.0
        x[1::8] = -0.0
        return x.astype(f)
    if kind.endswith("tiny"):  # subnormal float64, the smallest normal float32
        return (x * (2.0 ** -120 if f is np.float32 else 2.0 ** -1070)).astype(f)
    if kind.endswith("edge"):  # powers of two on both edges of the window, of both signs
        return (np.sign(x) * 2.0 ** rng.integers(-24, 4, n)).astype(f)
    raise ValueError(kind)


KINDS = ["i64_around_zero", "i64_two_windows", "i64_extremes", "i64_top", "i32_negative", "u32_large", "f32_wide",
         "f32_zeros", "f32_tiny", "f32_edge", "f64_wide", "f64_zeros", "f64_tiny", "f64_edge"]


@pytest.mark.parametrize("ops", [agg.AGG_ALL, agg.AGG_SUM | agg.AGG_AVG])
@pytest.mark.parametrize("keys", [1, 40, 900, 9000])
@pytest.mark.parametrize("kind", KINDS)
def test_windows_in_every_build(kind, keys, ops):
    n = 70_001
    k, v = dg.keys_uniform(n, keys, 3), values(kind, n)
    k[::1000] = 0xFFFFFFFF
    for kw in (dict(partition=-1), dict(partition=1, tile_rows=4096), dict(partition=-1, smem_slots=64)):
        res, _ = run(k, v, agg.AGG_STRAT_SMEM, ops, **kw)
        check_groups(res, k, v, ops)
    dev = [torch.from_numpy(a).cuda() for a in (k, v)]
    plan = agg.BatchPlan([(dev[0], dev[1], ops, agg.AGG_STRAT_SMEM)])
    plan.run()
    g = plan.result(0)
    check_groups(g.to_host(), k, v, ops)
    g.free()
    plan.free()


@pytest.mark.parametrize("kind", ["i64_two_windows", "i32_negative", "f32_edge", "f64_zeros"])
def test_blocks_of_more_rows_than_the_count_word(kind):
    """152 blocks of 64 threads fold about 80 thousand rows each: the packed words are settled twice."""
    n = 12_000_011
    k, v = dg.keys_uniform(n, 3, 5), values(kind, n)
    for off in (0, 1):  # vector loads; keys and values misaligned differently: scalar loads
        kd, vd = torch.from_numpy(k).cuda()[off:], torch.from_numpy(v).cuda()
        vd = vd[: n - off]
        g = agg.agg_groupby(kd, vd, agg.AGG_ALL,
                            agg.options(agg.AGG_STRAT_SMEM, partition=-1, block_threads=64, blocks_per_sm=1))
        check_groups(g.to_host(), k[off:], v[: n - off])
        g.free()
