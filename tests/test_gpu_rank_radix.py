"""Results ordered by rank or by radix sort, and the sort's own passes, at the edges of their ranges:
group counts on both sides of a table size's limits with the sentinel keys among them, row counts
around a radix tile and beyond the tiles one block of the digit scan takes in one turn."""
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


def keyed_rows(n, distinct, seed):
    """n rows over exactly `distinct` keys, the extreme ones among them."""
    keys = dg.domain_keys(seed, np.arange(distinct)).astype(np.uint32)
    ends = np.array([0, 0xFFFFFFFF, 0xFFFFFFFE, 1], np.uint32)[:distinct]
    keys[:ends.size] = ends
    keys = np.unique(keys)
    rng = np.random.default_rng(seed)
    return np.concatenate([keys, rng.choice(keys, n - keys.size)])[rng.permutation(n)]


@pytest.mark.parametrize("strategy", ["global", "smem"])
@pytest.mark.parametrize("distinct", [1, 2047, 2048, 2049, 4095, 4096, 4098, 8193, 16383, 16385, 32767, 32768, 32769,
                                      32770, 70000])
def test_ordered_results_at_every_size(distinct, strategy):
    n = 150_000
    keys = keyed_rows(n, distinct, 5)
    vals = dg.values("i32", n, 6)
    res, _ = run(keys, vals, getattr(agg, "AGG_STRAT_" + strategy.upper()))
    check_groups(res, keys, vals, agg.AGG_ALL)


@pytest.mark.parametrize("strategy", ["global", "smem"])
@pytest.mark.parametrize("tail", [20, 6000, 60000])
def test_table_far_larger_than_its_groups(tail, strategy):
    """A heavy key and a thin tail: the table is sized from a sample that saw the tail only in part."""
    n = 1_000_003
    rng = np.random.default_rng(tail)
    keys = np.full(n, 0xFFFFFFFF, np.uint32)
    keys[rng.permutation(n)[:max(tail, n // 20)]] = rng.integers(0, tail, max(tail, n // 20)).astype(np.uint32)
    vals = dg.values("f32", n, 7)
    res, _ = run(keys, vals, getattr(agg, "AGG_STRAT_" + strategy.upper()))
    check_groups(res, keys, vals, agg.AGG_ALL)


@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097, 3 * 4096, 5 * 4096 - 1, 16 * 4096 + 1])
def test_sort_at_tile_edges(n):
    keys = keyed_rows(n, max(1, n // 2), 8)
    vals = dg.values("i64", n, 9)
    check_groups(run(keys, vals, agg.AGG_STRAT_SORT)[0], keys, vals, agg.AGG_ALL)


def test_sort_of_more_tiles_than_one_turn_of_the_digit_scan():
    n = 4096 * 4096 + 4096 + 1  # 4098 tiles, 4096 a turn
    keys = keyed_rows(n, 50_000, 10)
    vals = dg.values("i32", n, 11)
    check_groups(run(keys, vals, agg.AGG_STRAT_SORT)[0], keys, vals, agg.AGG_ALL)


@pytest.mark.parametrize("distinct,skew,strategy", [(1 << 20, 0.0, "SORT"), (4000, 0.0, "SMEM"), (20_000, 1.0, "SMEM")])
def test_auto_around_the_distinct_count(distinct, skew, strategy):
    """Columns that AUTO sorts without a distinct count, and that it builds in tables with one."""
    n = (1 << 22) + 5
    keys = dg.keys_zipf(n, distinct, skew, 12) if skew else keyed_rows(n, distinct, 12)
    vals = dg.values("f64", n, 13)
    res, (used, _, _) = run(keys, vals, agg.AGG_STRAT_AUTO)
    assert used == getattr(agg, "AGG_STRAT_" + strategy)
    check_groups(res, keys, vals, agg.AGG_ALL)


def test_runs_across_chunks_and_lanes():
    """Sorted runs of every length around a lane's 8 rows and a warp's 256, alone and in sequence."""
    lengths = np.concatenate([np.arange(1, 40), [255, 256, 257, 511, 512, 513, 2047, 2049], np.ones(300, int),
                              np.full(60, 8), [5000]]).astype(np.int64)
    keys = np.repeat(np.arange(lengths.size, dtype=np.uint32) * 7 + 3, lengths)
    for dt in ("i64", "f32", "f64", "u32"):
        vals = dg.values(dt, keys.size, 14)
        for ops in (agg.AGG_ALL, agg.AGG_SUM | agg.AGG_COUNT):
            check_groups(run(keys, vals, agg.AGG_STRAT_SORT, ops)[0], keys, vals, ops)
