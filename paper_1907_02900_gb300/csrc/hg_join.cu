// HashGraph-Probe-New (Alg. 3): intersect the adjacency arrays of two tables
// bucket by bucket.  Both tables are built with the same V and bucket map,
// so equal keys always meet in the same bucket index.
//
// Both CSRs hold their edges in bucket order, so the kernels walk them side
// by side in tiles (bucket-major, merge-style) and take every edge's bucket
// from A's offsets instead of evaluating the bucket map:
//   k_join_merge   per edge a of table A: m(a) = number of edges of B's bucket
//                  with key(a); per bucket and per tile: sums of m; join total
//   scan of the tile sums -> output position of every tile
//   k_join_write   every tile writes its (A id, B id) pairs, in canonical
//                  order (bucket, A's CSR position, B's CSR position)
#include "hg_build.cuh"
#include "hg_trace.h"
#include "hg_scan.cuh"

namespace hg {

// Which tables a workspace's per-edge match counts belong to: written by the
// count, checked by the materialisation that reuses them.
struct JoinStamp {
  uint64_t w[8];
};
constexpr uint64_t kJoinStampMagic = 0x544E434E494F4A48ull;  // "HJOINCNT"

static JoinStamp join_stamp(const hg_table* A, const hg_table* B, uint64_t V) {
  JoinStamp s{};
  s.w[0] = kJoinStampMagic;
  s.w[1] = A->n;
  s.w[2] = B->n;
  s.w[3] = V;
  s.w[4] = (uint64_t)(uintptr_t)A->d_offsets;
  s.w[5] = (uint64_t)(uintptr_t)A->d_keys;
  s.w[6] = (uint64_t)(uintptr_t)B->d_offsets;
  s.w[7] = (uint64_t)(uintptr_t)B->d_keys;
  return s;
}

constexpr int kJoinThreads = 256;
// A tile is kJoinTile consecutive items of the merged sequence "bucket v,
// then its A edges" (bucket v at item offA[v] + v, A edge j of bucket v at
// item j + v + 1): at most kJoinTile A edges and kJoinTile + 1 buckets, so
// its slices of both offset arrays always fit shared memory, however sparse
// or skewed the table.
constexpr uint32_t kJoinTile = 2048;
constexpr uint32_t kJoinPer = kJoinTile / kJoinThreads;
constexpr uint32_t kJoinOffCap = kJoinTile + 2;  // offsets staged per table
constexpr uint32_t kJoinKeyBytes = kJoinTile * 8;  // B keys staged

// Merge-path split of every tile boundary w = t * kJoinTile: the bucket v
// holding item w (the last v with offA[v] + v <= w) and the first A edge at
// or after item w.  tv[tiles] closes the last tile.  Only these buckets can
// have edges in several tiles, which add their sums: their counts start at 0
// (bucket_counts may be null).
__global__ void k_join_tiles(const uint32_t* __restrict__ offA, uint64_t V, uint64_t nA, uint64_t tiles,
                             uint2* __restrict__ tv, unsigned long long* __restrict__ bucket_counts) {
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= tiles;
       t += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t w = t * kJoinTile;
    uint64_t v, j;
    if (w >= nA + V) {
      v = V - 1;
      j = nA;
    } else {
      uint64_t lo = 0, hi = V;  // item(lo) <= w < item(hi), item(V) = nA + V
      while (hi - lo > 1) {
        const uint64_t mid = lo + ((hi - lo) >> 1);
        if ((uint64_t)__ldg(offA + mid) + mid <= w) lo = mid;
        else hi = mid;
      }
      v = lo;
      const uint64_t o = __ldg(offA + v);
      j = w - v > o ? w - v - 1 : o;
    }
    tv[t] = make_uint2((uint32_t)v, (uint32_t)j);
    if (bucket_counts) bucket_counts[v] = 0;
  }
}

// One tile of the two tables: A edges [j0, j1) in buckets v0 .. v1, and the
// offsets of those buckets (and of v1 + 1) staged from both tables.  Ends
// with a barrier.
struct JoinTile {
  uint32_t v0, nv;  // buckets v0 .. v0 + nv - 1
  uint32_t j0, ne;  // A edges j0 .. j0 + ne - 1
};

__device__ __forceinline__ JoinTile join_tile(const uint2* __restrict__ tv, uint64_t t) {
  const uint2 c = tv[t], d = tv[t + 1];
  return JoinTile{c.x, d.x - c.x + 1, c.y, d.y - c.y};  // nv <= kJoinTile + 1, ne <= kJoinTile
}
// The tile's offsets of both tables to shared memory (no barrier).  NT: the
// block's threads.
template <int NT>
__device__ __forceinline__ void join_offsets(const JoinTile& T, const uint32_t* __restrict__ offA,
                                             const uint32_t* __restrict__ offB, uint32_t* oa, uint32_t* ob) {
  for (uint32_t k = threadIdx.x; k <= T.nv; k += NT) {
    oa[k] = __ldg(offA + T.v0 + k);
    ob[k] = __ldg(offB + T.v0 + k);
  }
}

// Local bucket of every A edge of the tile, edges PER * tid .. in bk[]: every
// bucket with edges in the tile marks its first one, and a running maximum
// carries the marks on.  mark: u16[kJoinTile] shared scratch (16-byte
// aligned), wmax: u32[32].  Starts and ends with a barrier (the offsets must
// have been written before).
template <int NT, int PER>
__device__ __forceinline__ void join_buckets(const JoinTile& T, const uint32_t* oa, uint16_t* mark, uint32_t* wmax,
                                             uint32_t (&bk)[PER]) {
  static_assert(NT * PER == (int)kJoinTile && PER % 4 == 0, "a thread's marks are whole 8-byte pieces");
  const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  uint2* const mine = reinterpret_cast<uint2*>(mark) + tid * (PER / 4);
#pragma unroll
  for (int i = 0; i < PER / 4; ++i) mine[i] = make_uint2(0, 0);
  __syncthreads();
  for (uint32_t k = tid; k < T.nv; k += NT) {
    const uint32_t lo = max(oa[k], T.j0), hi = min(oa[k + 1], T.j0 + T.ne);
    if (lo < hi) mark[lo - T.j0] = (uint16_t)k;
  }
  __syncthreads();
  uint32_t run = 0;
#pragma unroll
  for (int i = 0; i < PER / 4; ++i) {
    const uint2 x = mine[i];
    bk[4 * i] = run = max(run, x.x & 0xffffu);
    bk[4 * i + 1] = run = max(run, x.x >> 16);
    bk[4 * i + 2] = run = max(run, x.y & 0xffffu);
    bk[4 * i + 3] = run = max(run, x.y >> 16);
  }
  uint32_t incl = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, incl, o);
    if (lane >= (uint32_t)o) incl = max(incl, y);
  }
  uint32_t before = __shfl_up_sync(kFull, incl, 1);
  if (lane == 0) before = 0;
  if (lane == 31) wmax[warp] = incl;
  __syncthreads();
  before = max(before, __reduce_max_sync(kFull, lane < warp ? wmax[lane] : 0u));
#pragma unroll
  for (int i = 0; i < PER; ++i) bk[i] = max(bk[i], before);
}

// Matches of key among B's edges [s, e) (read from global memory).
template <typename K>
__device__ __forceinline__ uint32_t bucket_matches(const K* __restrict__ keysB, uint32_t s, uint32_t e, K key) {
  uint32_t m = 0, k = s;
  for (; k + 4 <= e; k += 4) {
    const K b0 = __ldg(keysB + k), b1 = __ldg(keysB + k + 1), b2 = __ldg(keysB + k + 2), b3 = __ldg(keysB + k + 3);
    m += (b0 == key) + (b1 == key) + (b2 == key) + (b3 == key);
  }
  for (; k < e; ++k) m += __ldg(keysB + k) == key;
  return m;
}

// Count (merge-style, bucket-major): both tables hold their edges in bucket
// order, so a tile of A's edges meets one contiguous run of B's edges; the
// kernel streams the two CSR arrays side by side, stages the run of B's keys
// when it fits, and never evaluates the bucket map.  Per A edge: m = matches
// in B's bucket (kept for the materialisation, as a bit mask of the bucket's
// edges where it has at most 32); per tile: its sum (kept), and
// added to the join total; per bucket: the sum of m, stored by the tile that
// holds the bucket and all of its A edges or added by every tile that holds
// some (zeroed by k_join_tiles).  bucket_counts, total null: not wanted.
//
// Bound by instruction issue (67% active; passes over the tile in shared
// memory).  3 * 10^7 against 2 * 10^7 uint32 keys, V = 2^25: 0.49 -> 0.37 ms
// with running maxima instead of a binary search per edge, 4-byte instead of
// 8-byte counts and no zeroing pass over the bucket counts.
template <typename K>
__global__ void __launch_bounds__(kJoinThreads) k_join_merge(const uint32_t* __restrict__ offA,
                                                             const K* __restrict__ keysA,
                                                             const uint32_t* __restrict__ offB,
                                                             const K* __restrict__ keysB,
                                                             const uint2* __restrict__ tv, uint64_t tiles,
                                                             uint32_t* __restrict__ m_out,
                                                             uint64_t* __restrict__ tile_sums,
                                                             unsigned long long* __restrict__ bucket_counts,
                                                             unsigned long long* __restrict__ total,
                                                             JoinStamp stamp, uint64_t* __restrict__ stamp_out) {
  __shared__ uint32_t oa[kJoinOffCap], ob[kJoinOffCap];
  __shared__ __align__(16) uint8_t region[kJoinKeyBytes + 32];  // B keys, and room to read 3 past them
  __shared__ __align__(16) uint16_t mark[kJoinTile];
  __shared__ uint32_t msm[kJoinTile];
  __shared__ uint32_t wmax[32];
  __shared__ unsigned long long wsum64[kJoinThreads / 32];
  if (stamp_out && blockIdx.x == 0 && threadIdx.x < 8) stamp_out[threadIdx.x] = stamp.w[threadIdx.x];
  const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  K* const kbs = (K*)region;
  constexpr uint32_t cap_b = kJoinKeyBytes / sizeof(K);
  unsigned long long acc = 0;
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const JoinTile T = join_tile(tv, t);
    // the tile's A keys to registers: in flight during the next steps
    K ka[kJoinPer];
#pragma unroll
    for (int r = 0; r < (int)kJoinPer; ++r) {
      const uint32_t i = tid + r * kJoinThreads;
      ka[r] = i < T.ne ? __ldcs(keysA + T.j0 + i) : K(0);
    }
    join_offsets<kJoinThreads>(T, offA, offB, oa, ob);
    uint32_t bk[kJoinPer];
    join_buckets<kJoinThreads, (int)kJoinPer>(T, oa, mark, wmax, bk);
    const uint32_t bb0 = ob[0], nbt = ob[T.nv] - bb0;
    const bool staged = nbt <= cap_b;
    if (staged)
      for (uint32_t k = tid; k < nbt; k += kJoinThreads) kbs[k] = __ldg(keysB + bb0 + k);
    reinterpret_cast<uint4*>(mark)[tid] = make_uint4(bk[0] | bk[1] << 16, bk[2] | bk[3] << 16, bk[4] | bk[5] << 16,
                                                     bk[6] | bk[7] << 16);  // (every thread has read its marks)
    __syncthreads();
    unsigned long long mine = 0;
#pragma unroll
    for (int r = 0; r < (int)kJoinPer; ++r) {
      const uint32_t i = tid + r * kJoinThreads;
      if (i < T.ne) {
        const uint32_t b = mark[i], s = ob[b], e = ob[b + 1];
        uint32_t m = 0, kept;
        const uint32_t len = e - s;
        if (len <= 32) {
          kept = 0;
          if (staged) {  // most buckets have at most four edges: no loop
            const K* const kb = kbs + (s - bb0);
            const uint32_t four = (uint32_t)(kb[0] == ka[r]) | (uint32_t)(kb[1] == ka[r]) << 1 |
                                  (uint32_t)(kb[2] == ka[r]) << 2 | (uint32_t)(kb[3] == ka[r]) << 3;
            kept = len >= 4 ? four : four & ((1u << len) - 1u);
            for (uint32_t x = 4; x < len; ++x) kept |= (uint32_t)(kb[x] == ka[r]) << x;
          } else {
            for (uint32_t x = 0; x < len; ++x) kept |= (uint32_t)(__ldg(keysB + s + x) == ka[r]) << x;
          }
          m = __popc(kept);
        } else {
          if (staged)
            for (uint32_t k = s - bb0; k < e - bb0; ++k) m += kbs[k] == ka[r];
          else
            m = bucket_matches(keysB, s, e, ka[r]);
          kept = m;
        }
        __stcs(m_out + T.j0 + i, kept);
        msm[i] = m;
        mine += m;
      }
    }
    mine = warp_sum(mine);
    if (lane == 0) wsum64[warp] = mine;
    __syncthreads();
    if (tid == 0) {
      unsigned long long sum = 0;
#pragma unroll
      for (int w = 0; w < kJoinThreads / 32; ++w) sum += wsum64[w];
      tile_sums[t] = sum;
      acc += sum;
    }
    if (bucket_counts) {
      // one thread per bucket: the sum over its edges of this tile.  The
      // first bucket's own item may lie in an earlier tile, the last one's
      // in the next; such a bucket is added to, or left to that tile.
      const uint64_t w0 = t * kJoinTile, w1 = w0 + kJoinTile;
      for (uint32_t k0 = warp * 32u; k0 < T.nv; k0 += kJoinThreads) {
        const uint32_t k = k0 + lane;
        uint32_t lo = 0, hi = 0;
        bool whole = false, here = false;
        if (k < T.nv) {
          const uint32_t bs = oa[k], be = oa[k + 1];
          const uint64_t item = (uint64_t)T.v0 + k + bs;  // of the bucket itself
          here = item >= w0 && item < w1;
          whole = here && be <= T.j0 + T.ne;
          lo = max(bs, T.j0) - T.j0;
          hi = min(be, T.j0 + T.ne) - T.j0;
          if (lo > hi) hi = lo;
        }
        unsigned long long c = 0;
        const bool many = hi - lo > 32;
        if (!many)
          for (uint32_t i = lo; i < hi; ++i) c += msm[i];
        for (uint32_t mm = __ballot_sync(kFull, many); mm; mm &= mm - 1) {  // long ones by the whole warp
          const int src = __ffs(mm) - 1;
          const uint32_t l = __shfl_sync(kFull, lo, src), h = __shfl_sync(kFull, hi, src);
          unsigned long long x = 0;
          for (uint32_t i = l + lane; i < h; i += 32) x += msm[i];
          x = warp_sum(x);
          if ((int)lane == src) c = x;
        }
        if (whole) bucket_counts[T.v0 + k] = c;
        else if (c) atomicAdd(bucket_counts + T.v0 + k, c);
      }
    }
    __syncthreads();
  }
  if (total && tid == 0 && acc) atomicAdd(total, acc);
}

// Pairs.  Per tile: the edges with matches are listed with their first output
// position (relative to the tile's); then every warp takes an equal range of
// the tile's outputs, 32 at a time.  The listed positions that fall into the
// 32 outputs, one bit each, give every lane its edge by a population count,
// so the pairs of an edge with many matches are written by many lanes and all
// stores are whole lines.  Matches that do not fill their bucket are found
// through the bit mask the count kept (buckets of more than 32 edges of B are
// walked).
//
// Bound by issue (66% active, 111 instructions per 32 pairs) and the stores
// (16 bytes a pair, 48% of DRAM peak).  2^29 pairs of a Zipf and a uniform
// side of 2^26 keys: 2.77 -> 2.36 ms against one lane per edge with windows
// staged in shared memory, and the scan over all edges (0.52 ms) is gone.
constexpr int kJoinWriteThreads = 512;
constexpr uint32_t kJoinIds = kJoinTile;  // B ids staged
template <typename K>
__global__ void __launch_bounds__(kJoinWriteThreads, 3)
    k_join_write(const uint32_t* __restrict__ offA, const K* __restrict__ keysA, const uint32_t* __restrict__ idsA,
                 const uint32_t* __restrict__ offB, const K* __restrict__ keysB, const uint32_t* __restrict__ idsB,
                 const uint2* __restrict__ tv, uint64_t tiles, const uint32_t* __restrict__ m_in,
                 const uint64_t* __restrict__ tile_base, int64_t* __restrict__ outA, int64_t* __restrict__ outB,
                 uint64_t cap, const uint32_t* __restrict__ abort) {
  constexpr int NT = kJoinWriteThreads, NW = NT / 32, PER = kJoinTile / NT;
  extern __shared__ __align__(16) uint8_t jsm[];
  uint8_t* sp = jsm;
  uint16_t* const mark = (uint16_t*)sp; sp += kJoinTile * 2;
  uint32_t* const cstart = (uint32_t*)sp; sp += kJoinTile * 4;  // listed edges: first output (relative)
  // listed edges: start of B's bucket from the tile's first B edge; A id;
  // matches in the bucket (0: all of it, ~0: to be walked); edge | bucket << 16
  uint4* const cinfo = (uint4*)sp; sp += kJoinTile * 16;
  uint32_t* const bid = (uint32_t*)sp; sp += kJoinIds * 4;      // the tile's B ids
  uint32_t* const oa = (uint32_t*)sp; sp += kJoinOffCap * 4;
  uint32_t* const ob = (uint32_t*)sp; sp += kJoinOffCap * 4;
  uint32_t* const wmax = (uint32_t*)sp; sp += 32 * 4;
  uint32_t* const wcnt = (uint32_t*)sp; sp += 32 * 4;
  unsigned long long* const wsum = (unsigned long long*)sp;
  if (*(volatile const uint32_t*)abort) return;
  const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint64_t base = tile_base[t];
    uint64_t n64 = tile_base[t + 1] - base;  // pairs of the tile
    if (n64 == 0) continue;                  // block-uniform
    if (base >= cap) return;                 // and so are all later tiles
    const JoinTile T = join_tile(tv, t);
    join_offsets<NT>(T, offA, offB, oa, ob);
    uint32_t kept[PER], bk[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const uint32_t i = tid * PER + r;
      kept[r] = i < T.ne ? __ldg(m_in + T.j0 + i) : 0u;
    }
    join_buckets<NT, PER>(T, oa, mark, wmax, bk);
    auto matches = [&](int r) { return ob[bk[r] + 1] - ob[bk[r]] <= 32 ? (uint32_t)__popc(kept[r]) : kept[r]; };
    const uint32_t bb0 = ob[0], nbt = ob[T.nv] - bb0;
    const bool staged = nbt <= kJoinIds;
    if (staged)
      for (uint32_t k = tid; k < nbt; k += NT) bid[k] = __ldg(idsB + bb0 + k);
    // first output and list place of every edge with matches
    unsigned long long sum = 0;
    uint32_t cnt = 0;
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      sum += matches(r);
      cnt += kept[r] != 0;
    }
    const unsigned long long isum = warp_incl_scan(sum);
    const uint32_t icnt = warp_incl_scan(cnt);
    if (lane == 31) {
      wsum[warp] = isum;
      wcnt[warp] = icnt;
    }
    __syncthreads();
    unsigned long long at = isum - sum;
    uint32_t c = icnt - cnt, listed = 0;
#pragma unroll
    for (uint32_t w = 0; w < NW; ++w) {
      if (w < warp) {
        at += wsum[w];
        c += wcnt[w];
      }
      listed += wcnt[w];
    }
    // a tile of 2^31 pairs or more keeps every edge's m in place of its start
    const bool huge = n64 >= 1ull << 31;
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      if (kept[r] == 0) continue;
      const uint32_t i = tid * PER + r, b = bk[r], s = ob[b], len = ob[b + 1] - s, m = matches(r);
      const uint32_t mask = m == len ? 0u : len <= 32 ? kept[r] : 0xffffffffu;  // (a full mask is never ~0: m == len)
      cstart[c] = huge ? m : (uint32_t)at;
      cinfo[c] = make_uint4(s - bb0, __ldg(idsA + T.j0 + i), mask, i | b << 16);
      at += m;
      ++c;
    }
    __syncthreads();
    if (n64 > cap - base) n64 = cap - base;
    // match r of a listed edge, counted from the tile's first B edge
    auto match = [&](const uint4& y, uint32_t r) {
      uint32_t k = y.x, mask = y.z;
      if (mask == 0) return k + r;
      if (mask == 0xffffffffu) {  // (k stays inside the bucket)
        const K key = __ldg(keysA + T.j0 + (y.w & 0xffffu));
        const uint32_t e = ob[(y.w >> 16) + 1] - bb0;
        for (; k + 1 < e; ++k)
          if (__ldg(keysB + bb0 + k) == key && r-- == 0) break;
        return k;
      }
#pragma unroll
      for (uint32_t h = 16; h > 0; h >>= 1) {  // set bit r of the mask, by halves
        const uint32_t low = __popc(mask & ((1u << h) - 1u));
        if (r >= low) {
          r -= low;
          mask >>= h;
          k += h;
        }
      }
      return k;
    };
    long long* const oA = (long long*)outA + base;
    long long* const oB = (long long*)outB + base;
    if (huge) {  // edges of a million matches on average: one after another, the whole block on each
      uint64_t done = 0;
      for (uint32_t q = 0; q < listed; ++q) {
        const uint32_t mq = cstart[q];
        for (uint64_t r = tid; r < mq && done + r < n64; r += NT) {
          __stcs(oA + done + r, (long long)cinfo[q].y);
          __stcs(oB + done + r, (long long)__ldg(idsB + bb0 + match(cinfo[q], (uint32_t)r)));
        }
        done += mq;
      }
      __syncthreads();
      continue;
    }
    // outputs [x0, x1) of this warp
    const uint32_t n = (uint32_t)n64;
    const uint32_t per = ((n + NW - 1) / NW + 31) / 32 * 32;
    const uint32_t x0 = min(warp * per, n), x1 = min(x0 + per, n);
    uint32_t e0;  // the last listed edge that starts at or before xb
    {
      uint32_t lo = 0, hi = listed;
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (cstart[mid] <= x0) lo = mid;
        else hi = mid;
      }
      e0 = lo;
    }
    const uint32_t upto = 0xffffffffu >> (31u - lane);
    for (uint32_t xb = x0; xb < x1; xb += 32) {
      const uint32_t idx = e0 + 1 + lane;
      const uint32_t rel = idx < listed ? cstart[idx] - xb : 32u;  // (later starts are at or beyond xb)
      const uint32_t starts = __reduce_or_sync(kFull, rel < 32 ? 1u << rel : 0u);
      const uint32_t q = e0 + __popc(starts & upto), x = xb + lane;
      if (x < x1) {
        const uint4 y = cinfo[q];
        const uint32_t k = match(y, x - cstart[q]);
        __stcs(oA + x, (long long)y.y);
        __stcs(oB + x, (long long)(staged ? bid[k] : __ldg(idsB + bb0 + k)));
      }
      e0 += __popc(starts);
    }
    __syncthreads();
  }
}
constexpr size_t kJoinWriteSmem =
    kJoinTile * 2 + kJoinTile * 4 + kJoinTile * 16 + kJoinIds * 4 + 2 * kJoinOffCap * 4 + 2 * 32 * 4 + 32 * 8;

__global__ void k_join_finish(const uint64_t* __restrict__ pairs, uint64_t cap, int64_t* __restrict__ d_total,
                              uint32_t* status, const uint32_t* abort, uint64_t* stamp) {
  stamp[0] = 0;  // the tile sums are now output positions: no later call may reuse them
  if (*abort) {
    *d_total = 0;
    return;
  }
  const uint64_t t = pairs ? *pairs : 0;
  *d_total = (int64_t)t;
  if (t > cap) set_status(status, HG_ERR_OVERFLOW);
}

// The materialisation after a count: the workspace must hold the per-edge
// match counts of exactly these tables (stamp).  On a mismatch nothing is
// written and the status reads HG_ERR_INVALID_ARG.
__global__ void k_join_check(JoinStamp want, const uint64_t* __restrict__ stamp, uint32_t* abort,
                             uint32_t* status) {
  bool ok = true;
  for (int i = 0; i < 8; ++i) ok &= stamp[i] == want.w[i];
  *abort = ok ? 0u : 1u;
  if (!ok) set_status(status, HG_ERR_INVALID_ARG);
}

struct JoinWs {
  uint32_t* m;          // matches of every A edge
  uint64_t* tile_sums;  // tiles + 1: pairs of every tile, then their output positions
  uint64_t* part;
  uint2* tv;            // tile splits (tiles + 1)
  uint64_t tiles;
  size_t total;
};

static JoinWs join_layout(uint8_t* ws, uint64_t nA, uint64_t V) {
  JoinWs w{};
  size_t o = sizeof(WsHeader);
  w.tiles = (nA + V + kJoinTile - 1) / kJoinTile;
  w.m = (uint32_t*)(ws + o);          o = align_up(o + (nA + 1) * 4);
  w.tile_sums = (uint64_t*)(ws + o);  o = align_up(o + (w.tiles + 1) * 8);
  w.part = (uint64_t*)(ws + o);       o = align_up(o + scan_workspace_bytes<uint64_t>(w.tiles + 1));
  w.tv = (uint2*)(ws + o);            o = align_up(o + (w.tiles + 1) * 8);
  w.total = o;
  return w;
}

size_t join_workspace_bytes(uint64_t nA, uint64_t V) { return join_layout(nullptr, nA, V).total; }

// Grid of a bucket-major kernel: one wave of resident CTAs (a second,
// partial wave would leave most SMs idle while it runs), at most one per tile.
template <typename F>
static unsigned join_grid(F* kern, uint64_t tiles, int threads, size_t smem) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm <= 0)
    per_sm = 1;
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(tiles, (uint64_t)dev_info().sms * per_sm));
}

static hg_status join_tiles(const hg_table* A, uint64_t V, const JoinWs& w, unsigned long long* bc,
                            cudaStream_t st) {
  HG_TRACE("k_join_tiles", st);
  const uint64_t g = std::min<uint64_t>((w.tiles + 1 + 255) / 256, (uint64_t)dev_info().sms * 8);
  k_join_tiles<<<(unsigned)g, 256, 0, st>>>(A->d_offsets, V, A->n, w.tiles, w.tv, bc);
  return last_launch_status();
}

template <typename K>
static hg_status join_merge(const hg_table* A, const hg_table* B, const JoinWs& w, unsigned long long* bc,
                            unsigned long long* total, const JoinStamp& stamp, uint64_t* stamp_out, cudaStream_t st) {
  HG_TRACE("k_join_merge", st);
  k_join_merge<K><<<join_grid(k_join_merge<K>, w.tiles, kJoinThreads, 0), kJoinThreads, 0, st>>>(
      A->d_offsets, (const K*)A->d_keys, B->d_offsets, (const K*)B->d_keys, w.tv, w.tiles, w.m, w.tile_sums, bc, total,
      stamp, stamp_out);
  return last_launch_status();
}

// The bucket map is not evaluated: the tables' CSR order gives every edge's
// bucket.  (Map stays in the signature: the tables must come from it.)
template <typename K, typename Map>
hg_status join_count_impl(const hg_config* cfg, const hg_table* A, const hg_table* B, int64_t* d_total,
                          int64_t* d_bucket_counts, uint8_t* ws, cudaStream_t st, Map) {
  const uint64_t V = cfg->num_buckets, nA = A->n;
  JoinWs w = join_layout(ws, nA, V);
  unsigned long long* bc = (unsigned long long*)d_bucket_counts;
  if (cudaMemsetAsync(d_total, 0, 8, st) != cudaSuccess) return HG_ERR_CUDA;
  hg_status rc = join_tiles(A, V, w, bc, st);
  if (rc != HG_OK) return rc;
  return join_merge<K>(A, B, w, bc, (unsigned long long*)d_total, join_stamp(A, B, V), ((WsHeader*)ws)->join_stamp, st);
}

// after_count: the tile splits, per-edge match counts and tile sums come from
// the hg_join_count call that last used this workspace on the same tables
// (checked on the device) instead of a second intersection pass.
template <typename K, typename Map>
hg_status join_materialize_impl(const hg_config* cfg, const hg_table* A, const hg_table* B, int64_t* outA,
                                int64_t* outB, uint64_t cap, int64_t* d_total, uint8_t* ws, cudaStream_t st,
                                Map, bool after_count) {
  const uint64_t V = cfg->num_buckets, nA = A->n;
  JoinWs w = join_layout(ws, nA, V);
  WsHeader* hdr = (WsHeader*)ws;
  if (after_count) {
    HG_TRACE("k_join_check", st);
    k_join_check<<<1, 1, 0, st>>>(join_stamp(A, B, V), hdr->join_stamp, &hdr->join_abort, &hdr->status);
  }
  if (nA > 0) {
    if (!after_count) {
      hg_status rc = join_tiles(A, V, w, nullptr, st);
      if (rc == HG_OK) rc = join_merge<K>(A, B, w, nullptr, nullptr, JoinStamp{}, nullptr, st);
      if (rc != HG_OK) return rc;
    }
    // (the closing element's input value does not matter)
    hg_status rc = device_excl_scan<uint64_t>(w.tile_sums, w.tiles + 1, w.part, st);
    if (rc != HG_OK) return rc;
    {
      HG_TRACE("k_join_write", st);
      auto kern = k_join_write<K>;
      // (set on every call: it holds again after a device reset)
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kJoinWriteSmem);
      kern<<<join_grid(kern, w.tiles, kJoinWriteThreads, kJoinWriteSmem), kJoinWriteThreads, kJoinWriteSmem, st>>>(
          A->d_offsets, (const K*)A->d_keys, A->d_ids, B->d_offsets, (const K*)B->d_keys, B->d_ids, w.tv, w.tiles,
          w.m, w.tile_sums, outA, outB, cap, &hdr->join_abort);
    }
  }
  {
    HG_TRACE("k_join_finish", st);
    k_join_finish<<<1, 1, 0, st>>>(nA > 0 ? w.tile_sums + w.tiles : nullptr, cap, d_total, &hdr->status,
                                   &hdr->join_abort, hdr->join_stamp);
  }
  return last_launch_status();
}

#define HG_INST(K, M)                                                                                          \
  template hg_status join_count_impl<K, M>(const hg_config*, const hg_table*, const hg_table*, int64_t*,       \
                                           int64_t*, uint8_t*, cudaStream_t, M);                              \
  template hg_status join_materialize_impl<K, M>(const hg_config*, const hg_table*, const hg_table*, int64_t*, \
                                                 int64_t*, uint64_t, int64_t*, uint8_t*, cudaStream_t, M, bool);
HG_INST(uint32_t, MurmurMap<true>)
HG_INST(uint64_t, MurmurMap<true>)
HG_INST(uint32_t, MurmurMap<false>)
HG_INST(uint64_t, MurmurMap<false>)
HG_INST(uint32_t, LearnedMap)
HG_INST(uint64_t, LearnedMap)
#undef HG_INST

}  // namespace hg
