"""Float sums where a lost low bit shows: groups of a few small negative values in a column of larger
ones."""
import math

import numpy as np
import pytest
import torch

import paper_2606_10030_gb300 as agg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    agg.build()
    agg.lib()


def small_negative_column(n, rows_a_group, dt, seed=0):
    """Every other row belongs to key 0xFFFFFFF0 and lies in [1, 2); the others form groups of
    rows_a_group rows in (-2^-p, -2^-p-1] for p of 10 to 23 (float32: to 20), all significand bits random:
    the lowest binades that a block's window of exponents above 1 still holds exactly."""
    rng = np.random.default_rng(seed)
    v = 1.0 + rng.random(n)
    k = np.full(n, 0xFFFFFFF0, dtype=np.uint32)
    m = n // 2
    v[1::2][:m] = -(1.0 + rng.random(m)) * np.exp2(-rng.integers(11, 24 if dt is np.float64 else 21, m).astype(float))
    k[1::2][:m] = np.arange(m, dtype=np.uint32) // rows_a_group
    return k, v.astype(dt)


@pytest.mark.parametrize("rows_a_group", [1, 3])
@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("how", ["plain", "full", "partitioned", "batch"])
def test_small_negative_groups_keep_their_bits(how, dt, rows_a_group):
    """A one-row group's sum is its value; of three rows, float64 additions of values of one sign
    lose at most two roundings of 2^-53 of the sum, and one more for the float64 of the sum."""
    n = 150_001 if how == "partitioned" else 6_001
    k, v = small_negative_column(n, rows_a_group, dt)
    dev = torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda()
    if how == "batch":
        plan = agg.BatchPlan([(*dev, agg.AGG_ALL, agg.AGG_STRAT_SMEM)])
        plan.run()
        g = plan.result(0)
    else:
        kw = dict(plain=dict(partition=-1, smem_slots=4096), full=dict(partition=-1, smem_slots=64),
                  partitioned=dict(partition=1))[how]
        g = agg.agg_groupby(*dev, agg.AGG_ALL, agg.options(agg.AGG_STRAT_SMEM, **kw))
    res = g.to_host()
    g.free()
    keys, inv = np.unique(k, return_inverse=True)
    assert np.array_equal(res["keys"], keys)
    small = np.arange(keys.size - 1)
    rows = [[] for _ in keys]
    for i, x in zip(inv, v.astype(np.float64)):
        if i < small.size:
            rows[i].append(x)
    want = np.array([math.fsum(rows[i]) for i in small])
    got = res["sum"][small]
    if rows_a_group == 1:
        assert np.array_equal(got, want)
        assert np.array_equal(res["avg"][small], want)
    else:
        assert np.all(np.abs(got - want) <= 3 * 2.0 ** -53 * np.abs(want))


def scan(x, host):
    if host:
        return agg.agg_reduce_host(torch.from_numpy(x).pin_memory(), agg.AGG_ALL)
    return agg.decode_scalar(agg.agg_reduce(torch.from_numpy(x).cuda(), agg.AGG_ALL))


@pytest.mark.parametrize("host", [False, True])
@pytest.mark.parametrize("small", ["ones", "normal"])
@pytest.mark.parametrize("dt,big", [(np.float32, 1e30), (np.float64, 2.0 ** 100), (np.float64, 1e35), (np.float64, 1e300)])
def test_scan_of_large_values_that_cancel(dt, big, small, host):
    """Rows far apart cancel and leave the other rows' sum. A thread folds at most 24 of these rows (2^22
    rows in at least 2^18 vectors' blocks). Of a thread that holds a large value, float64 rows lose what
    lies below 2^-147 of it, float32 rows nothing (TwoSum); what the merges shift below the unit is
    added in float64, at most 20 additions deep."""
    n = 1 << 22
    x = np.ones(n, dtype=dt)
    if small == "normal":
        x = np.random.default_rng(1).standard_normal(n).astype(dt)
    x[12_345], x[n - 77] = big, -big
    total = math.fsum(np.delete(x, [12_345, n - 77]).astype(np.float64))
    a = float(np.abs(np.delete(x, [12_345, n - 77]).astype(np.float64)).sum())
    lost = 0.0
    if dt is np.float64:
        lost = 48 * min(float(np.abs(x[np.abs(x) < big]).max()), big * 2.0 ** -146)
    r = scan(x, host)
    assert abs(r.sum_f - total) <= lost + (0.0 if small == "ones" else 20 * 2.0 ** -53 * a)
    assert abs(r.sum_f - total) <= r.err_bound
    assert np.isfinite(r.err_bound)


@pytest.mark.parametrize("span", [10, 40, 90, 140, 400, 2000])
def test_float64_scan_of_any_span_is_the_exact_sum(span):
    """Exponents uniform over span binades: the sum differs from the exact one by its own rounding and
    2^-100 of the largest rows, and the bound holds."""
    rng = np.random.default_rng(span)
    n = 1_000_003
    x = rng.standard_normal(n) * np.exp2(rng.integers(-span // 2, span // 2 + 1, n).astype(float))
    for y in (x, np.concatenate([x, -x[::-1][: n - 5]])):
        ref = math.fsum(y)
        r = scan(y, False)
        assert abs(r.sum_f - ref) <= 2.0 ** -53 * abs(ref) + y.size * 2.0 ** -120 * float(np.abs(y).max())
        assert abs(r.sum_f - ref) <= r.err_bound
