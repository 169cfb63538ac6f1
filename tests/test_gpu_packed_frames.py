"""Packed scans of every frame width class, whole and ragged, mixed in one column, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_10030_gb300 as agg
from tests.test_gpu_packed import same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    agg.build()
    agg.lib()


def column(widths, n, seed=0):
    """int64 values whose frames of 1024 need the given widths in turn, the extremes in every frame."""
    rng = np.random.default_rng(seed)
    x = np.empty(n, np.int64)
    for f, a in enumerate(range(0, n, 1024)):
        b = min(n, a + 1024)
        w = widths[f % len(widths)]
        off = rng.integers(0, 1 << min(w, 62), b - a) if w else np.zeros(b - a, np.int64)
        off[-1] = 0
        off[0] = (1 << min(w, 62)) - 1 if w else 0
        x[a:b] = off - (1 << 40) * (f % 3)
    return x


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1000, 1023, 1024, 1025, 3 * 1024 + 17, 70 * 1024 + 1])
@pytest.mark.parametrize("widths", [[1], [7], [17], [31], [32], [33], [0, 32, 5, 40, 16], [32, 33, 1, 0, 62, 8]])
def test_frame_widths(widths, n):
    x = column(widths, n)
    p = agg.agg_pack_for(torch.from_numpy(x))
    ref = oracle.reduce(x)
    dev = p.to("cuda")
    for ops in (agg.AGG_ALL, agg.AGG_SUM, agg.AGG_MIN | agg.AGG_MAX):
        same(agg.decode_scalar(agg.agg_reduce_packed(dev, ops)).as_dict(), ref, ops)
    same(agg.agg_reduce_packed_host(p, agg.AGG_ALL).as_dict(), ref, agg.AGG_ALL)
