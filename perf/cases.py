"""Timed cases of the HashGraph library: the calls a program makes, over the range of sizes it makes them at.

A case is a dict of plain values.  Kinds:
  build_probe   hg.build of n keys into v buckets, then hg.probe of q queries
  lookup        hg.probe of q queries in a table built beforehand
  host          hg.build_probe_host: keys and queries in pinned host memory, counts back to it
  join_count    hg.join_count (total and per bucket) of two tables built beforehand
  join_pairs    hg.join_count_into, then hg.join_materialize_into (every pair of ids) from that count, in kept buffers
  batched       hg.BatchPlan.run: many tables of uneven sizes built and probed together
  learned       hg.build and hg.probe with a learned bucket map trained beforehand
"""
import math

import numpy as np
import torch

import paper_1907_02900_gb300 as hg

M32 = 0xFFFFFFFF


def listed():
    return [
        # a service's lookup of a handful of keys: launch and latency are all there is
        {"name": "lookup_1k", "kind": "lookup", "key": "u32", "n": 1_000_000, "v": 1 << 20, "q": 1000, "hit": 0.9, "dup": 1},
        # a small build side and its probe (a dimension table), sizes off the powers of two
        {"name": "build_probe_60k", "kind": "build_probe", "key": "u32", "n": 60_001, "v": 1 << 16, "q": 60_001,
         "hit": 0.5, "dup": 1, "ids": False},
        # the plain workload: 2^20 keys at load 1, as many queries, half of them hits
        {"name": "build_probe_2e20", "kind": "build_probe", "key": "u32", "n": 1 << 20, "v": 1 << 20, "q": 1 << 20,
         "hit": 0.5, "dup": 1, "ids": False},
        # 8-byte keys that carry row ids of their own, load 2, a bucket count that is no power of two
        {"name": "build_probe_u64_ids", "kind": "build_probe", "key": "u64", "n": 20_000_003, "v": 10_000_019,
         "q": 30_000_001, "hit": 0.9, "dup": 1, "ids": True},
        # a foreign-key column: every key about eight times
        {"name": "build_probe_dup8", "kind": "build_probe", "key": "u32", "n": 50_000_017, "v": 50_000_017,
         "q": 50_000_017, "hit": 0.5, "dup": 8, "ids": False},
        # the headline: 2^28 keys at load 1, 2^28 queries at 50% hits
        {"name": "build_probe_2e28", "kind": "build_probe", "key": "u32", "n": 1 << 28, "v": 1 << 28, "q": 1 << 28,
         "hit": 0.5, "dup": 1, "ids": False},
        # more buckets than one two-level build holds
        {"name": "build_probe_2e30", "kind": "build_probe", "key": "u32", "n": 1 << 30, "v": 1 << 30, "q": 1 << 30,
         "hit": 0.5, "dup": 1, "ids": False},
        # size of an inner join and its split over the buckets, without the pairs (a planner's estimate, a semi-join)
        {"name": "join_count_u32", "kind": "join_count", "key": "u32", "n": 30_000_001, "v": 1 << 25, "q": 20_000_003,
         "hit": 0.5, "dup": 2},
        # the join workload: a Zipf side against a uniform side over the same keys, all pairs written
        {"name": "join_pairs_zipf", "kind": "join_pairs", "key": "u64", "n": 1 << 26, "v": 1 << 26, "q": 1 << 26,
         "ranks": 1 << 23},
        # many tables of uneven sizes in one call, sizes log-uniform as in the batched workload
        {"name": "batched_2500", "kind": "batched", "tables": 2500, "total": 1 << 28, "hit": 0.5},
        # the learned workload: clustered 8-byte keys under the learned map
        {"name": "learned_2e26", "kind": "learned", "key": "u64", "n": 1 << 26, "v": 1 << 26, "q": 1 << 26, "hit": 0.5},
        # keys and queries that arrive in host memory
        {"name": "host_2e25", "kind": "host", "key": "u32", "n": 1 << 25, "v": 1 << 25, "q": 1 << 25, "hit": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))


def draw(rng):
    kind = rng.choice(["build_probe"] * 5 + ["lookup", "host", "join_count", "join_pairs", "batched", "learned"])
    key = rng.choice(["u32", "u32", "u64"])
    load = rng.choice([0.25, 0.5, 1.0, 1.0, 1.0, 2.0, 4.0])
    hit = rng.choice([0.1, 0.5, 0.9])
    if kind == "batched":
        total = _log_int(rng, 1 << 18, 1 << 28)
        return {"kind": kind, "tables": max(4, int(total / _log_int(rng, 1 << 12, 1 << 17))), "total": total, "hit": hit}
    if kind == "learned":
        n = _log_int(rng, 1 << 17, 1 << 26)
        return {"kind": kind, "key": "u64", "n": n, "v": n, "q": _log_int(rng, n / 2, n), "hit": hit}
    if kind == "join_pairs":
        n = _log_int(rng, 1 << 14, 1 << 26)
        return {"kind": kind, "key": "u64", "n": n, "v": n, "q": _log_int(rng, n / 2, n), "ranks": max(1, n >> 3)}
    if kind == "join_count":
        n = _log_int(rng, 1 << 14, 1 << 26)
        return {"kind": kind, "key": key, "n": n, "v": max(1, int(n / load)), "q": _log_int(rng, n / 4, n), "hit": hit,
                "dup": rng.choice([1, 2, 4])}
    if kind == "lookup":
        n = _log_int(rng, 1 << 12, 1 << 26)
        return {"kind": kind, "key": key, "n": n, "v": max(1, int(n / load)), "q": _log_int(rng, 64, 1 << 24), "hit": hit,
                "dup": rng.choice([1, 1, 4])}
    if kind == "host":
        n = _log_int(rng, 1 << 16, 1 << 25)
        return {"kind": kind, "key": key, "n": n, "v": n, "q": _log_int(rng, n / 2, n), "hit": hit}
    n = _log_int(rng, 1 << 10, 1 << 29 if key == "u32" else 1 << 27)
    v = min(1 << 30, max(1, int(n / load)))
    if rng.random() < 0.5:
        v = 1 << (v.bit_length() - 1)
    return {"kind": kind, "key": key, "n": n, "v": v, "q": _log_int(rng, n / 4, n), "hit": hit,
            "dup": rng.choice([1, 1, 1, 2, 4, 8]), "ids": rng.random() < 0.25}


# ------------------------------------------------------------------ inputs
# Keys are scrambled preimages, as in the library's datagen module: a preimage in the lower half of the domain may
# be a key, one in the upper half never is, so a query drawn from there is a miss.
def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)


def _lsr(x, s):  # logical shift right of int64 words
    return (x >> s) & ((1 << (64 - s)) - 1)


def _scramble32(x):
    x = x ^ (x >> 15)
    x = (x * 0x7A1F3C9B) & M32
    x = x ^ (x >> 13)
    x = (x * 0x5C2E8D17) & M32
    return x ^ (x >> 16)


def _i64(c):
    return c - (1 << 64) if c >= 1 << 63 else c


def _scramble64(x):
    x = x ^ _lsr(x, 31)
    x = x * _i64(0x6A09E667F3BCC909)
    x = x ^ _lsr(x, 29)
    x = x * _i64(0xBB67AE8584CAA73B)
    return x ^ _lsr(x, 32)


def _narrow(x, key):  # int64 words -> a signed tensor of the key's bytes
    return torch.where(x > 0x7FFFFFFF, x - (1 << 32), x).to(torch.int32) if key == "u32" else x


def _unsigned(t):
    return t.view(torch.uint32 if t.dtype == torch.int32 else torch.uint64)


_CHUNK = 1 << 26


def _chunked(n, key, f):
    out = torch.empty(n, dtype=torch.int32 if key == "u32" else torch.int64, device="cuda")
    for a in range(0, n, _CHUNK):
        b = min(a + _CHUNK, n)
        out[a:b] = f(a, b - a)
    return out


def _keys(n, key, dup, seed, salt=1):
    """n keys: uniform over half the domain, or (dup > 1) over n / dup distinct ones."""
    g = _gen(seed, salt)
    top = max(1, n // dup) if dup > 1 else (1 << 31 if key == "u32" else (1 << 63) - 1)
    s = _scramble32 if key == "u32" else _scramble64
    return _chunked(n, key, lambda a, m: _narrow(s(torch.randint(0, top, (m,), generator=g, device="cuda")), key))


def _queries(q, keys, key, hit, seed, salt=2):
    """q queries: a share `hit` copies of random keys, the others keys that no table holds."""
    g = _gen(seed, salt)

    def some(a, m):
        if key == "u32":
            miss = _scramble32(torch.randint(1 << 31, 1 << 32, (m,), generator=g, device="cuda"))
        else:
            miss = _scramble64(torch.randint(-(1 << 63), 0, (m,), generator=g, device="cuda"))
        pick = torch.randint(0, keys.numel(), (m,), generator=g, device="cuda")
        return torch.where(torch.rand(m, generator=g, device="cuda") < hit, keys[pick], _narrow(miss, key))

    return _chunked(q, key, some)


def _zipf_keys(n, ranks, seed):
    g = _gen(seed, 3)
    cdf = torch.cumsum(1.0 / torch.arange(1, ranks + 1, dtype=torch.float64, device="cuda"), 0)

    def some(a, m):
        u = torch.rand(m, generator=g, dtype=torch.float64, device="cuda") * cdf[-1]
        return _scramble64(torch.clamp(torch.searchsorted(cdf, u, right=True), max=ranks - 1) + 1)

    return _chunked(n, "u64", some)


def _rank_keys(n, ranks, seed):
    g = _gen(seed, 4)
    return _chunked(n, "u64", lambda a, m: _scramble64(torch.randint(1, ranks + 1, (m,), generator=g, device="cuda")))


def _lognormal_keys(n, seed):
    """Clustered u64 keys: 64 lognormal clusters and a tenth of uniform words."""
    g = _gen(seed, 5)
    mu = 20.0 + 16.0 * torch.rand(64, generator=g, dtype=torch.float64, device="cuda")
    sigma = 0.5 + 1.5 * torch.rand(64, generator=g, dtype=torch.float64, device="cuda")

    def some(a, m):
        c = torch.randint(0, 64, (m,), generator=g, device="cuda")
        z = torch.randn(m, generator=g, dtype=torch.float64, device="cuda")
        x = torch.clamp(torch.exp(mu[c] + sigma[c] * z), max=2.0 ** 62).to(torch.int64)
        uni = torch.randint(-(1 << 63), (1 << 63) - 1, (m,), generator=g, device="cuda")
        return torch.where(torch.rand(m, generator=g, device="cuda") < 0.1, uni, x)

    return _chunked(n, "u64", some)


def _inputs(case, seed):
    """The case's keys and queries (join: the two sides' keys) as signed CUDA tensors."""
    kind, key = case["kind"], case.get("key", "u32")
    if kind == "join_pairs":
        return _zipf_keys(case["n"], case["ranks"], seed), _rank_keys(case["q"], case["ranks"], seed)
    if kind == "learned":
        k = _lognormal_keys(case["n"], seed)
    else:
        k = _keys(case["n"], key, case.get("dup", 1), seed)
    return k, _queries(case["q"], k, key, case["hit"], seed)


def _row_ids(n, seed):  # distinct ids in no order, as row numbers of a filtered column are
    g = _gen(seed, 6)
    return torch.randint(-(1 << 31), 1 << 31, (n,), generator=g, device="cuda").to(torch.int32)


def _capacity(case):
    """Room for a Zipf join's pairs: their expected number and seven standard deviations or so."""
    return int(1.4 * case["n"] * case["q"] / case["ranks"])


def _batch_sizes(case):  # the plan's shape belongs to the case; its keys and queries come from the seed
    u = np.random.default_rng(case["total"]).random(case["tables"])
    s = np.exp2(10.0 + 12.0 * u)
    return np.maximum(1, np.floor(s * (case["total"] / s.sum()))).astype(np.int64)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "batched":
        sizes = _batch_sizes(case)
        st["plan"] = plan = hg.BatchPlan(sizes, sizes, seed=0)
        st["bufs"] = b = plan.alloc()
        n = int(sizes.sum())
        table = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.from_numpy(sizes).cuda())
        first = torch.from_numpy(np.cumsum(sizes) - sizes).cuda()
        at = torch.arange(n, device="cuda") - first[table]
        where = torch.from_numpy(plan.key_begin[:-1].astype(np.int64)).cuda()[table] + at
        k = _keys(n, "u32", 1, seed)
        q = _queries(n, k, "u32", 0.0, seed)
        g = _gen(seed, 7)
        own = first[table] + (torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
                              * torch.from_numpy(sizes).cuda()[table]).to(torch.int64)
        q = torch.where(torch.rand(n, generator=g, device="cuda") < case["hit"], k[own], q)
        b["keys"].view(torch.int32)[where] = k
        b["queries"].view(torch.int32)[where] = q
        return st
    k, q = _inputs(case, seed)
    k, q = _unsigned(k), _unsigned(q)
    if kind == "build_probe":
        st.update(keys=k, queries=q, ids=_unsigned(_row_ids(case["n"], seed)) if case["ids"] else None)
    elif kind == "lookup":
        st.update(table=hg.build(k, case["v"]), queries=q)
    elif kind == "join_count":
        st.update(a=hg.build(k, case["v"]), b=hg.build(q, case["v"]))
    elif kind == "join_pairs":
        i64 = lambda size: torch.zeros(size, dtype=torch.int64, device="cuda")  # noqa: E731
        a, b, cap = hg.build(k, case["v"]), hg.build(q, case["v"]), _capacity(case)
        st.update(a=a, b=b, total=i64(1), per_bucket=i64(case["v"]), out_a=i64(cap), out_b=i64(cap),
                  ws=torch.zeros(hg.join_workspace_size(a.cfg, case["n"], case["q"]), dtype=torch.uint8, device="cuda"))
    elif kind == "learned":
        model, _ = hg.learned_train(k, case["v"])
        st.update(keys=k, queries=q, model=model)
    elif kind == "host":
        n, m, v = case["n"], case["q"], case["v"]
        cfg = hg.make_config(hg.KEY_U32 if case["key"] == "u32" else hg.KEY_U64, v)
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
        dev = lambda size, like: torch.empty(size, dtype=like, device="cuda")  # noqa: E731
        table = hg.Table(dev(v + 1, torch.uint32), dev(n, k.dtype), dev(n, torch.uint32), cfg)
        st.update(cfg=cfg, table=table, h_keys=pin(k), h_queries=pin(q),
                  h_counts=torch.empty(m, dtype=torch.uint32, pin_memory=True), d_keys=dev(n, k.dtype),
                  d_queries=dev(m, k.dtype), d_counts=dev(m, torch.uint32),
                  ws=dev(hg.build_workspace_size(cfg, n), torch.uint8),
                  probe_ws=dev(hg.probe_workspace_size(table, m), torch.uint8))
    else:
        raise ValueError(kind)
    return st


def _signed(**tensors):
    """The same bytes under the signed types, for which torch has every operation."""
    return {k: t.view(torch.int64 if t.element_size() == 8 else torch.int32) for k, t in tensors.items()}


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "build_probe":
        t = hg.build(st["keys"], case["v"], ids=st["ids"])
        return _signed(offsets=t.offsets, keys=t.keys, ids=t.ids, counts=hg.probe(t, st["queries"]))
    if kind == "lookup":
        return _signed(counts=hg.probe(st["table"], st["queries"]))
    if kind == "learned":
        t = hg.build(st["keys"], case["v"], model=st["model"])
        return _signed(offsets=t.offsets, keys=t.keys, ids=t.ids, counts=hg.probe(t, st["queries"]))
    if kind == "join_count":
        total, per_bucket = hg.join_count(st["a"], st["b"])
        return {"total": total, "per_bucket": per_bucket}
    if kind == "join_pairs":
        hg.join_count_into(st["a"], st["b"], st["total"], st["per_bucket"], st["ws"])
        hg.join_materialize_into(st["a"], st["b"], st["out_a"], st["out_b"], st["total"], st["ws"], after_count=True)
        return {"total": st["total"], "per_bucket": st["per_bucket"], "a": st["out_a"], "b": st["out_b"]}
    if kind == "batched":
        b = st["bufs"]
        st["plan"].run(b)
        return _signed(offsets=b["offsets"], keys=b["csr_keys"], ids=b["csr_ids"], counts=b["counts"])
    t = st["table"]
    hg.build_probe_host(st["cfg"], st["h_keys"], st["h_queries"], st["h_counts"], st["d_keys"], st["d_queries"],
                        st["d_counts"], t, st["ws"], st["probe_ws"])
    return _signed(offsets=t.offsets, keys=t.keys, ids=t.ids, counts=st["h_counts"])


def work(case):
    """Every input read once and every output written once.  The path has no floating-point work."""
    kind = case["kind"]
    if kind == "batched":
        n = case["total"]
        return {"bytes": 4 * n + 4 * n + (4 + 4 + 4) * n + 4 * n, "flops": 0}
    kb = 8 if case["key"] == "u64" else 4
    n, v, q = case["n"], case["v"], case["q"]
    if kind == "lookup":  # each query reads its two offsets and its keys, at most the whole table
        return {"bytes": kb * q + 4 * q + min(q * (8 + kb), 4 * v + kb * n), "flops": 0}
    if kind == "join_count":
        return {"bytes": 2 * 4 * v + kb * (n + q) + 8 * v, "flops": 0}
    if kind == "join_pairs":
        pairs = n * q // case["ranks"]
        return {"bytes": 2 * 4 * v + (kb + 4) * (n + q) + 8 * v + 16 * pairs, "flops": 0}
    ids = 4 * n if case.get("ids") else 0
    return {"bytes": kb * n + ids + (kb + 4) * n + 4 * v + kb * q + 4 * q, "flops": 0}


# ------------------------------------------------------------ exact values
def _rotl(x, r):
    return ((x << r) | (x >> (32 - r))) & M32


def _murmur3(keys):
    """MurmurHash3_x86_32 (seed 0) of a signed key tensor, as int64 values below 2^32."""
    words = [keys.to(torch.int64) & M32]
    if keys.dtype == torch.int64:
        words.append(_lsr(keys, 32))
    h = torch.zeros_like(words[0])
    for k in words:
        k = _rotl((k * 0xCC9E2D51) & M32, 15)
        h = _rotl(h ^ ((k * 0x1B873593) & M32), 13)
        h = (h * 5 + 0xE6546B64) & M32
    h = h ^ (4 * len(words))
    h = ((h ^ (h >> 16)) * 0x85EBCA6B) & M32
    h = ((h ^ (h >> 13)) * 0xC2B2AE35) & M32
    return h ^ (h >> 16)


def _buckets(keys, v):
    out = torch.empty(keys.numel(), dtype=torch.int32, device="cuda")  # v < 2^31 here
    for a in range(0, keys.numel(), _CHUNK):
        out[a:a + _CHUNK] = (_murmur3(keys[a:a + _CHUNK]) % v).to(torch.int32)
    return out


def _table(keys, bucket, v):
    """Offsets and the stable order of the keys by bucket."""
    sorted_b, order = torch.sort(bucket, stable=True)
    ends = torch.arange(v + 1, dtype=torch.int32, device="cuda")
    offsets = torch.searchsorted(sorted_b, ends).to(torch.int32)
    return offsets, order


def _multiplicity(keys, queries):
    s = torch.sort(keys)[0]
    out = torch.empty(queries.numel(), dtype=torch.int32, device="cuda")
    for a in range(0, queries.numel(), _CHUNK):
        x = queries[a:a + _CHUNK]
        out[a:a + _CHUNK] = (torch.searchsorted(s, x, right=True) - torch.searchsorted(s, x)).to(torch.int32)
    return out


def _exact_batched(case, seed):
    st = prepare(case, seed)
    plan, b = st["plan"], st["bufs"]
    T = plan.T

    def side(begin, sizes, values):  # table of every position, and whether the position only pads
        begin = torch.from_numpy(begin.astype(np.int64)).cuda()
        t = torch.repeat_interleave(torch.arange(T, device="cuda"), begin[1:] - begin[:-1])
        local = torch.arange(values.numel(), device="cuda") - begin[t]
        return t, local, local >= torch.from_numpy(sizes.astype(np.int64)).cuda()[t]

    keys, queries = b["keys"].view(torch.int32), b["queries"].view(torch.int32)
    t, local, pad = side(plan.key_begin, plan.sizes, keys)
    ob = torch.from_numpy(plan.offset_begin.astype(np.int64)).cuda()
    vt = (ob[1:] - ob[:-1] - 1)[t]
    bucket = ob[t] + torch.where(pad, vt, _murmur3(keys) % vt)
    order = torch.sort(bucket, stable=True)[1]
    counts = torch.bincount(bucket, minlength=plan.total_offsets)
    offsets = torch.cumsum(counts, 0) - counts
    tq, _, padq = side(plan.query_begin, plan.qsizes, queries)
    word = lambda x, tab, p: ((tab + torch.where(p, T, 0)) << 32) | (x.to(torch.int64) & M32)  # noqa: E731
    return {"offsets": offsets.to(torch.int32), "keys": keys[order], "ids": local[order].to(torch.int32),
            "counts": _multiplicity(word(keys, t, pad), word(queries, tq, padq))}


def exact(case, seed):
    """run()'s answer from plain torch integer arithmetic."""
    kind = case["kind"]
    if kind == "batched":
        return _exact_batched(case, seed)
    k, q = _inputs(case, seed)
    if kind == "lookup":
        return {"counts": _multiplicity(k, q)}
    if kind == "learned":  # the order of the table is the model's
        return {"offsets": None, "keys": None, "ids": None, "counts": _multiplicity(k, q)}
    v = case["v"]
    if kind in ("join_count", "join_pairs"):
        bucket = _buckets(k, v)
        m = _multiplicity(q, k).to(torch.int64)
        out = {"total": m.sum().reshape(1),
               "per_bucket": torch.zeros(v, dtype=torch.int64, device="cuda").index_add_(0, bucket.to(torch.int64), m)}
        if kind == "join_count":
            return out
        order = _table(k, bucket, v)[1]  # A's edges in canonical order
        k, m = k[order], m[order]
        del bucket
        sq, pos = torch.sort(q, stable=True)
        # an edge's r-th match is the r-th of its key in B's input order
        lead = torch.searchsorted(sq, k) - (torch.cumsum(m, 0) - m)
        a = torch.repeat_interleave(order, m)
        b = pos[torch.repeat_interleave(lead, m) + torch.arange(a.numel(), device="cuda")]
        cap = _capacity(case)
        for name, x in (("a", a[:cap]), ("b", b[:cap])):  # the room beyond the pairs is left as it was
            out[name] = torch.cat([x, torch.zeros(cap - x.numel(), dtype=torch.int64, device="cuda")])
        return out
    offsets, order = _table(k, _buckets(k, v), v)
    ids = _row_ids(case["n"], seed)[order] if case.get("ids") else order.to(torch.int32)
    return {"offsets": offsets, "keys": k[order], "ids": ids, "counts": _multiplicity(k, q)}
