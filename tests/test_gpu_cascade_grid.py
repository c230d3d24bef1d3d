"""The cascade's count commit on grids around its limit of 65,535 blocks."""
import numpy as np
import pytest
import torch

from paper_2301_07684_gb300 import cascade, sfq
from paper_2301_07684_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(ctx, grid):
    ctx.set_step_shape(1, 0, grid)
    d = W.config2(n=300, seed=5, a0=150.0, gamma0=1e4)
    run = cascade.CascadeRun(ctx, d, capacity=1 << 15, products_cap=1 << 15)
    run.run(0, 12)
    ctx.sort_products(run.out)
    a = run.alive()
    order = np.lexsort((a["flags"], a["id"]))
    return {k: v[order] for k, v in a.items()}, run.out.to_numpy(), sfq.counters_dict(run.counters), run.count()


def test_the_count_is_committed_on_any_grid():
    """The commit counts finished blocks in 16 bits; a larger grid is launched with as many."""
    ctx = sfq.Context(ref_len_m=W.REF_LEN, dt=W.DT, precision="fp32", seed=8)
    want = _run(ctx, 0)
    assert want[3] > 320 and want[2]["spawn_dropped"] == 0
    for grid in (1, 65534, 65535, 65536, 70000, 131072):
        got = _run(ctx, grid)
        assert got[2:] == want[2:], grid
        for a, b in zip(got[:2], want[:2]):
            for k in b:
                assert np.array_equal(a[k], b[k]), (grid, k)
