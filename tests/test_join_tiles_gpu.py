"""The join's tile walk at its edges: buckets of B of up to and above 32 edges
with some of their edges matching, edges of A spread over tiles, tiles with
more pairs than 32 bits count, small capacities, against the oracle."""
import numpy as np
import pytest

from paper_1907_02900_gb300 import datagen as dg
from gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kt", ["u32", "u64"])
@pytest.mark.parametrize("nA,nB,distinct,V", [
    (5000, 3000, 700, 1 << 14),     # whole buckets match
    (5000, 3000, 700, 256),         # buckets of about 12 edges, some matching
    (3000, 8000, 400, 256),         # 31 and more: on both sides of the mask
    (2047, 2048, 64, 7),            # long buckets only
    (6000, 6000, 6000, 1 << 13),    # few matches
    (4097, 1, 1, 5), (1, 4097, 3, 4096), (10_000, 10, 10, 1),
])
def test_count_and_pairs(hg, orc, kt, nA, nB, distinct, V):
    rng = np.random.default_rng(nA + V)
    dom = dg.uniform_keys_u32(distinct, 3) if kt == "u32" else dg.uniform_keys_u64(distinct, 3)
    ka, kb = dom[rng.integers(0, distinct, nA)], dom[rng.integers(0, distinct, nB)]
    A, B = hg.build(to_dev(ka), V), hg.build(to_dev(kb), V)
    # the pairs in canonical order: A's edges in table order, each with its matches in B's input order
    order_a = to_np(A.ids).astype(np.int64)
    sb = np.argsort(kb, kind="stable")
    lo, hi = np.searchsorted(kb[sb], ka[order_a], "left"), np.searchsorted(kb[sb], ka[order_a], "right")
    want_a = np.repeat(order_a, hi - lo)
    want_b = np.concatenate([sb[l:h] for l, h in zip(lo, hi)]) if nA else np.zeros(0, np.int64)
    total, per = hg.join_count(A, B)
    assert int(total.item()) == len(want_a) == orc.join_size_by_keys(ka, kb)
    bucket = orc.buckets(ka, V, 0).astype(np.int64)
    want_per = np.bincount(bucket[order_a], weights=(hi - lo).astype(np.float64), minlength=V).astype(np.int64)
    assert np.array_equal(to_np(per), want_per)
    for cap in (None, len(want_a) // 3 + 1):
        a, b = hg.join_materialize(A, B, capacity=cap)
        assert np.array_equal(to_np(a), want_a[:len(a)]) and np.array_equal(to_np(b), want_b[:len(b)])
        assert len(a) == (len(want_a) if cap is None else min(cap, len(want_a)))


def test_a_tile_of_more_pairs_than_31_bits(hg):
    """2050 equal keys against 2^20 + 3 equal ones: a tile alone has 2^31 pairs; only the capacity is written."""
    import torch
    nA, nB, cap = 2050, (1 << 20) + 3, 3 * ((1 << 20) + 3) + 1234
    A = hg.build(torch.full((nA,), 77, dtype=torch.int32, device="cuda").view(torch.uint32), 3)
    B = hg.build(torch.full((nB,), 77, dtype=torch.int32, device="cuda").view(torch.uint32), 3)
    assert int(hg.join_count(A, B, per_bucket=False)[0].item()) == nA * nB
    oa, ob = (torch.empty(cap, dtype=torch.int64, device="cuda") for _ in range(2))
    total = torch.empty(1, dtype=torch.int64, device="cuda")
    ws = torch.empty(hg.join_workspace_size(A.cfg, nA, nB), dtype=torch.uint8, device="cuda")
    hg.join_materialize_into(A, B, oa, ob, total, ws)
    assert int(total.item()) == nA * nB and hg.workspace_status(ws) == 3  # HG_ERR_OVERFLOW
    x = torch.arange(cap, device="cuda")
    assert torch.equal(oa, x // nB) and torch.equal(ob, x % nB)
