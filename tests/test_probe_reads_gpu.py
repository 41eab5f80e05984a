"""The direct probe's wide table reads at their edges: every position of a
bucket in its 32 bytes, buckets longer than one piece, the end of the arrays,
arrays that are not 32- or 16-byte aligned, against the oracle."""
import numpy as np
import pytest

from paper_1907_02900_gb300 import datagen as dg
from gpu_util import to_dev, to_np

pytestmark = pytest.mark.gpu


def _shifted(t, k):
    """A copy of a CUDA tensor that starts k elements into an allocation."""
    import torch
    a = torch.empty(t.numel() + k, dtype=t.dtype, device="cuda")[k:]
    a.copy_(t)
    return a


@pytest.mark.parametrize("kt", ["u32", "u64"])
@pytest.mark.parametrize("n,V", [(1, 1), (7, 3), (8, 8), (9, 15), (1000, 16), (1003, 1001), (5000, 4096), (300, 1 << 14)])
def test_every_bucket(hg, orc, kt, n, V):
    make, ask = (dg.uniform_keys_u32, dg.queries_u32) if kt == "u32" else (dg.uniform_keys_u64, dg.queries_u64)
    keys = make(n, 5)
    keys[n // 2:] = keys[:n - n // 2]  # every key about twice
    q = np.concatenate([keys, ask(4 * n + 50, keys, 0.3, 6)])
    t = hg.build(to_dev(keys), V)
    ref = orc.multiplicity(keys, q)
    for ko in (0, 1, 2, 3, 4):
        for oo in (0, 1, 4):
            s = hg.Table(_shifted(t.offsets, oo), _shifted(t.keys, ko), t.ids, t.cfg)
            assert np.array_equal(to_np(hg.probe(s, to_dev(q), binned=False)), ref), (ko, oo)


def test_learned_map_reads(hg, orc):
    keys = dg.lognormal_mixture_u64(20_001, 8)
    model, _ = hg.learned_train(to_dev(keys), 20_001, num_leaves=64)
    t = hg.build(to_dev(keys), 20_001, model=model)
    q = dg.queries_u64(30_000, keys, 0.5, 9)
    for ko in (0, 1):
        s = hg.Table(_shifted(t.offsets, ko), _shifted(t.keys, ko), t.ids, t.cfg, model)
        assert np.array_equal(to_np(hg.probe(s, to_dev(q), binned=False)), orc.multiplicity(keys, q))


def test_large_misaligned_batches_are_still_refused(hg):
    keys = dg.uniform_keys_u32(1000, 1)
    t = hg.build(to_dev(keys), 1000)
    q = to_dev(dg.uniform_keys_u32((1 << 20) + 4, 2))
    with pytest.raises(hg.HGError):
        hg.probe(t, q[1:])
    assert hg.probe(t, q[4:]).numel() == 1 << 20
