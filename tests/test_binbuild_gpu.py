"""The shared-memory bin build at its edges: every CTA size, buckets sorted one
by one or ranked slot by slot, both orders (by id, by bin position), bins at
and above a CTA's room, against the oracle byte for byte."""
import numpy as np
import pytest

from paper_1907_02900_gb300 import datagen as dg
from gpu_util import table_np, to_dev

pytestmark = pytest.mark.gpu


def _keys(kt, n, V, repeats, seed):
    """n uniform keys, of which some appear `repeats` times each, all over the input."""
    k = dg.uniform_keys_u32(n, seed) if kt == "u32" else dg.uniform_keys_u64(n, seed)
    rng = np.random.default_rng(seed)
    at = rng.permutation(n)
    i = 0
    for r in repeats:
        k[at[i:i + r]] = k[at[i]]
        i += r
    return k


# bins of 2^shift buckets: CTAs of 256 or 512 threads by the expected bin, of
# 1024 threads in builds of at most two bins per SM
@pytest.mark.parametrize("explicit", [False, True])
@pytest.mark.parametrize("kt", ["u32", "u64"])
@pytest.mark.parametrize("n,V,shift,repeats", [
    ((1 << 21) + 3, 1 << 21, 12, [2, 3, 4, 5, 6, 31, 32]),            # sorted one by one, up to a warp's bucket
    ((1 << 21) + 1, 1 << 21, 12, [33]),                               # one bin ranked slot by slot
    ((1 << 21) + 2, (1 << 21) - 5, 12, [255, 256, 257, 1000, 4000]),  # words' longest bucket, bins past a CTA's room
    ((1 << 22) + 5, 1 << 22, 13, [4, 5, 40, 9000, 17000]),            # 512 threads; second launch
    (1 << 19, 1 << 19, 13, [5] * 40),                                 # 1024 threads
    (5 << 19, 1 << 19, 10, [7]),                                      # load 5: every bin ranked slot by slot
    (1 << 21, 1 << 23, 14, [2, 33]),                                  # load 1/4, mostly empty buckets
    (700, 1 << 20, 12, []),                                           # bins of a few edges
])
def test_bin_build_edges(hg, orc, kt, n, V, shift, repeats, explicit):
    keys = _keys(kt, n, V, repeats, n + shift)
    ids = np.random.default_rng(1).integers(0, 1 << 32, n, dtype=np.uint32) if explicit else None
    t = hg.build(to_dev(keys), V, ids=None if ids is None else to_dev(ids), bin_shift=shift)
    got, ref = table_np(t), orc.build(keys, V, 0, ids=ids)
    for name, g, r in zip(("offsets", "keys", "ids"), got, ref):
        assert np.array_equal(g, r), name


@pytest.mark.parametrize("threads", [512, 1024])
def test_bin_build_threads_asked_for(hg, orc, threads):
    n = V = (1 << 20) + 9
    keys = _keys("u32", n, V, [300, 5000, 12000], threads)
    d = to_dev(keys)
    import torch
    cfg = hg.make_config(hg.KEY_U32, V)
    cfg.threads_per_bin = threads
    off = torch.empty(V + 1, dtype=torch.uint32, device="cuda")
    ck, ci = torch.empty_like(d), torch.empty(n, dtype=torch.uint32, device="cuda")
    ws = torch.empty(hg.build_workspace_size(cfg, n), dtype=torch.uint8, device="cuda")
    hg.build_into(cfg, d, None, off, ck, ci, ws)
    for g, r in zip(table_np(hg.Table(off, ck, ci, cfg)), orc.build(keys, V)):
        assert np.array_equal(g, r)
    assert hg.workspace_status(ws) == 0
