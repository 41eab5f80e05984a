"""Tables of more bins than one shared-memory histogram holds: the two-level
build with the late bin histogram (implicit ids) and the slab build (explicit
ids) are different paths to the same table; so are the binned probe, with 256
groups and several launches, and the direct one."""
import pytest

from paper_1907_02900_gb300 import datagen as dg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,V,hot", [
    ((1 << 29) + 12345, 1 << 29, 0),           # 2^16 bins
    (3 << 28, (1 << 29) + (1 << 28) + 99, 0),  # more than 2^16 bins, 512-way pass A, V no power of two
    ((1 << 29) + 77, 1 << 29, 15_000),         # a bin for the bin build's second launch
    ((1 << 29) + 77, 1 << 29, 50_000),         # a bin too large for shared memory: the slabs take over
])
def test_wide_build_equals_slab_build(hg, n, V, hot):
    import torch
    import paper_1907_02900_gb300.datagen_gpu as dgg
    torch.cuda.empty_cache()
    keys = dgg.uniform_keys_u32(n, dg.SEED_SCALE + hot)
    if hot:
        keys.view(torch.int32)[5:5 + hot] = 123456789
    t = hg.build(keys, V)
    ids = torch.arange(n, dtype=torch.int32, device="cuda").view(torch.uint32)
    s = hg.build(keys, V, ids=ids)
    for name in ("offsets", "keys", "ids"):
        assert torch.equal(getattr(t, name).view(torch.int32), getattr(s, name).view(torch.int32)), name
    del s, ids
    torch.cuda.empty_cache()
    if hot == 0:
        q = dgg.queries_u32((1 << 27) + 4099, keys, 0.5, 7)
        a, b = hg.probe(t, q, binned=True), hg.probe(t, q, binned=False)
        assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    del t, keys
    torch.cuda.empty_cache()
