"""Batched probes in query order (all tables small) and grouped (a large table
in the wave) against the oracle: uneven and empty tables, waves that start at
any bucket."""
import numpy as np
import pytest

from paper_1907_02900_gb300 import datagen as dg
from gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,shift", [
    ([1, 0, 3, 5000, 2, 77_777, 1, 1], 0),
    ([10_000] * 50 + [0, 1, 2, 3], 0),
    ([30_000] * 40, 1),              # several waves
    ([2_500_000, 10, 300_000], 0),
    ([9_000_000, 10, 300_000], 0),   # a table above 64 MB: grouped
])
def test_counts_of_every_table(hg, orc, sizes, shift):
    import torch
    sizes = np.array(sizes)
    qsizes = sizes[::-1].copy() + 5
    plan = hg.BatchPlan(sizes, qsizes, seed=3)
    if shift:
        plan.set_config(bin_shift=shift)
        assert plan.config()["waves"] > 1
    keys = dg.batched_keys_u32(sizes, 5)
    queries = dg.batched_queries_u32(qsizes, keys, sizes, 0.5, 6)
    b = plan.alloc()
    b["keys"].view(torch.int32).copy_(to_dev(plan.pad_keys(keys)).view(torch.int32))
    b["queries"].view(torch.int32).copy_(to_dev(plan.pad_queries(queries)).view(torch.int32))
    b["counts"].view(torch.int32).fill_(-1)
    plan.run(b)
    kb, qb = np.concatenate([[0], np.cumsum(sizes)]), np.concatenate([[0], np.cumsum(qsizes)])
    for t in range(len(sizes)):
        got = to_np(plan.table(b, t)[3])
        assert np.array_equal(got, orc.multiplicity(keys[kb[t]:kb[t + 1]], queries[qb[t]:qb[t + 1]])), t
    assert hg.workspace_status(b["ws"]) == 0
