"""Builds at the edges of the small paths: the fused scan (up to 64 chunks of
4096 keys in one pass), sizes below which no bin can overflow, bins too large
for shared memory in small builds, against the oracle."""
import numpy as np
import pytest

from paper_1907_02900_gb300 import datagen as dg
from gpu_util import table_np, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("explicit", [False, True])
@pytest.mark.parametrize("kt", ["u32", "u64"])
@pytest.mark.parametrize("n,V", [
    (1, 7), (18432, 18432), (18433, 18433), (14336, 1), (14337, 2), (64 * 4096, 1 << 18), (64 * 4096 + 1, 1 << 18),
    (64 * 4096, 3), (200_000, 129), (100_000, 1 << 20), (1 << 20, 1 << 14),
])
@pytest.mark.parametrize("hot", [0, 30_000])
def test_small_build(hg, orc, kt, n, V, hot, explicit):
    keys = dg.uniform_keys_u32(n, n) if kt == "u32" else dg.uniform_keys_u64(n, n)
    at = np.random.default_rng(n).permutation(n)[:hot]
    keys[at] = keys[0]  # a bin too large for shared memory, where the build is large enough
    ids = np.random.default_rng(V).permutation(n).astype(np.uint32) if explicit else None
    import torch
    ws = torch.full((hg.build_workspace_size(hg.make_config(hg.KEY_U32 if kt == "u32" else hg.KEY_U64, V), n),), 255,
                    dtype=torch.uint8, device="cuda")  # nothing may rely on what a workspace held
    t = hg.build(to_dev(keys), V, ids=None if ids is None else to_dev(ids), ws=ws)
    for name, g, r in zip(("offsets", "keys", "ids"), table_np(t), orc.build(keys, V, 0, ids=ids)):
        assert np.array_equal(g, r), name
    assert hg.workspace_status(ws) == 0
