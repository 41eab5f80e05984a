"""The partitions in any order at their edges (tile remainders, empty and
crowded super-bins, ordered input), seen through the tables and counts they
lead to, against the oracle."""
import numpy as np
import pytest

from paper_1907_02900_gb300 import datagen as dg
from gpu_util import table_np, to_dev, to_np

pytestmark = pytest.mark.gpu


def _same_table(hg, orc, keys, V, shift):
    t = hg.build(to_dev(keys), V, bin_shift=shift)
    for name, g, r in zip(("offsets", "keys", "ids"), table_np(t), orc.build(keys, V)):
        assert np.array_equal(g, r), name
    return t


# tiles: pass A 12288 (uint32) and 5632 (uint64) keys, pass B 4608 and 4096
@pytest.mark.parametrize("kt", ["u32", "u64"])
@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097, 4608, 4609, 5632, 12287, 12288, 12289, 2 * 12288 + 513, 304 * 4096 + 17])
def test_tile_remainders(hg, orc, kt, n):
    keys = dg.uniform_keys_u32(n, n) if kt == "u32" else dg.uniform_keys_u64(n, n)
    _same_table(hg, orc, keys, 1 << 16, 4)  # 4096 bins: two passes
    _same_table(hg, orc, keys, 200, 1)      # 100 bins: one pass


@pytest.mark.parametrize("what", ["few super-bins", "by bucket", "one per super-bin"])
def test_crowded_and_empty_super_bins(hg, orc, what):
    V, shift = 1 << 20, 5  # 2^15 bins of 32 buckets, 256 super-bins of 4096 buckets
    pool = dg.uniform_keys_u32(1 << 21, 9)
    b = orc.buckets(pool, V, 0).astype(np.int64)
    if what == "few super-bins":  # the first, one in the middle, the last; nothing between
        keys = pool[np.isin(b >> 12, [0, 117, 255])]
    elif what == "by bucket":     # input already in table order: a tile falls into a few bins
        keys = pool[np.argsort(b, kind="stable")][:1 << 20]
    else:
        keys = pool[np.unique(b >> 12, return_index=True)[1]]
    _same_table(hg, orc, keys, V, shift)


@pytest.mark.parametrize("kt", ["u32", "u64"])
@pytest.mark.parametrize("q", [1, 4097, 8191, 8192, 8193, 3 * 8192, 32768 * 2 + 5, 304 * 8192 + 4099])
def test_query_blocks(hg, orc, kt, q):
    n, V = 40_000, 50_021
    keys = dg.uniform_keys_u32(n, 3) if kt == "u32" else dg.uniform_keys_u64(n, 3)
    queries = dg.queries_u32(q, keys, 0.5, 4) if kt == "u32" else dg.queries_u64(q, keys, 0.5, 4)
    t = hg.build(to_dev(keys), V)
    assert np.array_equal(to_np(hg.probe(t, to_dev(queries), binned=True)), orc.multiplicity(keys, queries))
