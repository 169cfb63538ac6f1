"""Build options and planned sizes of GROUP BY: block sizes on every build, table sizes of host-fed
columns, the autotuner's choice as it is run, work items of a tuned batch."""
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


@pytest.mark.parametrize("dt", ["i32", "f64"])
@pytest.mark.parametrize("threads", [64, 512, 544, 1024])
@pytest.mark.parametrize("partition", [-1, 0, 1, 2])
def test_every_block_size_on_every_build(partition, threads, dt):
    """2^20 rows over 20 K keys: partition = 0 partitions them by itself."""
    n = 1 << 20
    k, v = dg.keys_uniform(n, 20_000, 1), dg.values(dt, n, 1)
    res, _ = run(k, v, agg.AGG_STRAT_SMEM, partition=partition, block_threads=threads)
    check_groups(res, k, v)


@pytest.mark.parametrize("threads", [512, 1024])
def test_every_block_size_on_host_fed_columns(threads):
    """More than one chunk of 8 Mi rows, hash-partitioned chunk by chunk."""
    n = (1 << 23) + 70_001
    k, v = dg.keys_uniform(n, 200_000, 1), dg.values("i64", n, 1)
    for partition in (-1, 1):
        g = agg.agg_groupby_host(torch.from_numpy(k), torch.from_numpy(v), agg.AGG_ALL,
                                 agg.options(agg.AGG_STRAT_SMEM, partition=partition, block_threads=threads))
        check_groups(g.to_host(), k, v)
        g.free()


def test_host_fed_column_keeps_its_planned_table():
    """Three chunks of 8 Mi rows run on the table that the whole column on the device runs on."""
    n = (1 << 24) + 1001
    k, v = dg.keys_uniform(n, 100, 2), dg.values("i32", n, 2)
    g = agg.agg_groupby(torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda(), agg.AGG_ALL,
                        agg.options(agg.AGG_STRAT_SMEM))
    h = agg.agg_groupby_host(torch.from_numpy(k), torch.from_numpy(v), agg.AGG_ALL,
                             agg.options(agg.AGG_STRAT_SMEM))
    assert h.smem_slots == g.smem_slots == 512
    check_groups(h.to_host(), k, v)
    g.free()
    h.free()


@pytest.mark.parametrize("keys", [100, 1000, 3000])
@pytest.mark.parametrize("dt", ["i32", "i64", "f64"])
def test_autotuned_call_runs_the_timed_build(dt, keys):
    """AUTOTUNE's table is the one timed; the shared-memory default among the candidates is AUTO's own."""
    agg.lib().agg_autotune_clear()
    n = 1 << 21
    k = torch.from_numpy(dg.keys_uniform(n, keys, 3)).cuda()
    v = torch.from_numpy(dg.values(dt, n, 3)).cuda()
    r = agg.agg_autotune(k, v, agg.AGG_ALL, reps=2)
    auto = agg.agg_groupby(k, v, agg.AGG_ALL, agg.options(agg.AGG_STRAT_SMEM))
    smem = [s for s, t in zip(r.smem_slots, list(r.strategy)[:r.ncand]) if t == agg.AGG_STRAT_SMEM]
    assert auto.smem_slots in smem
    g = agg.agg_groupby(k, v, agg.AGG_ALL, agg.options(agg.AGG_STRAT_AUTOTUNE))
    assert g.strategy == r.strategy[r.best]
    if g.strategy == agg.AGG_STRAT_SMEM:
        assert g.smem_slots == r.smem_slots[r.best]
    auto.free()
    g.free()


def _ms(f, reps=20):
    for _ in range(3):
        f()
    torch.cuda.synchronize()
    out = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            f()
        b.record()
        torch.cuda.synchronize()
        out.append(a.elapsed_time(b) / reps)
    return min(out)


def test_tuning_a_small_batch_does_not_slow_it_down():
    """131 K float64 rows over 64 K keys: a work item is a chain of atomics, so that 16 Ki rows an item
    take nearly twice the plan's own 8 Ki."""
    n = 1 << 17
    k, v = dg.keys_uniform(n, 1 << 16, 4), dg.values("f64", n, 4)
    plan = agg.BatchPlan([(torch.from_numpy(k).cuda(), torch.from_numpy(v).cuda(), agg.AGG_ALL, agg.AGG_STRAT_AUTO)])
    before = _ms(plan.run)
    assert plan.tune(5) in (16384, 32768, 65536)
    assert _ms(plan.run) <= 1.15 * before
    g = plan.result(0)
    check_groups(g.to_host(), k, v)
    g.free()
    plan.free()
