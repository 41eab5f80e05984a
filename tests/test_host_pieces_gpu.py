"""The host-buffer call with its queries in pieces (2^22 and more queries, a
ragged last piece, both key widths, direct and binned, pinned and not) against
the oracle's counts."""
import numpy as np
import pytest

from paper_1907_02900_gb300 import datagen as dg

pytestmark = pytest.mark.gpu

P = 1 << 22


@pytest.mark.parametrize("n,q,u64,binned,pinned", [
    (1000, P, False, True, True),            # one piece
    (1000, P + 1, False, True, True),        # a last piece of one query
    (100_000, 4 * P, False, True, False),
    (100_000, 4 * P + 4097, True, True, True),
    (100_000, 2 * P + 3, True, False, True),  # direct
    (5 * P, 2 * P + 77, False, True, True),  # pieces from the table's size
    (0, P + 5, False, True, True),
])
def test_counts(hg, orc, n, q, u64, binned, pinned):
    import torch
    keys = (dg.uniform_keys_u64 if u64 else dg.uniform_keys_u32)(n, 3)
    rng = np.random.default_rng(q)
    queries = rng.integers(0, 1 << 32, q, dtype=keys.dtype)
    if n:
        queries[::2] = keys[rng.integers(0, n, len(queries[::2]))]
    V = max(1, n)
    cfg = hg.make_config(hg.KEY_U64 if u64 else hg.KEY_U32, V)
    dev = lambda m, t: torch.empty(m, dtype=t, device="cuda")  # noqa: E731
    kt = torch.uint64 if u64 else torch.uint32
    t = hg.Table(dev(V + 1, torch.uint32), dev(n, kt), dev(n, torch.uint32), cfg)
    hk, hq = torch.from_numpy(keys.copy()), torch.from_numpy(queries)
    hc = torch.full((q,), -1, dtype=torch.int32)
    if pinned:
        hk, hq, hc = hk.pin_memory(), hq.pin_memory(), hc.pin_memory()
    ws = dev(hg.build_workspace_size(cfg, n), torch.uint8)
    pws = dev(hg.probe_workspace_size(t, q), torch.uint8) if binned else None
    dc = dev(q, torch.uint32)
    hg.build_probe_host(cfg, hk, hq, hc, dev(n, kt), dev(q, kt), dc, t, ws, pws)
    torch.cuda.current_stream().synchronize()
    want = orc.multiplicity(keys, queries) if n else np.zeros(q, np.uint32)
    assert np.array_equal(hc.numpy().view(np.uint32), want)
    if binned:
        assert hg.workspace_status(pws) == 0
