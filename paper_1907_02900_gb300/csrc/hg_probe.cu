// HashGraph-Probe-Standard (Section 3.4): map the query to its bucket, read
// the bucket's two offsets, scan the bucket's edges and count every key equal
// to the query (all instances, Section 5.2).
#include "hg_build.cuh"
#include "hg_trace.h"
#include "hg_probe.cuh"

namespace hg {

// A bucket's two offsets and its matches.  Two forms, chosen per map:
// Sectors (plain hash maps): every random access takes a whole aligned
// 32-byte sector.  The sector of the bucket's offset holds its end too for 7
// buckets of 8, and the bucket's keys seldom reach a second one.  Equal keys
// share a bucket, so whatever equals the query in a sector belongs to its
// bucket and nothing is masked.
// Pieces (the learned map, whose queries crowd into few buckets and hit L1,
// so instructions bound it; batched tables, where the next table's bucket may
// hold the same key): 16-byte offset quads; 4-byte keys in masked 16-byte
// pieces, 8-byte keys one by one.  With sectors: learned 0.71 ms for 0.64
// (2^26 queries), batched 3.62 for 3.32 (2500 tables).
template <bool SECTORS>
struct TableReader;

struct Sector {
  uint32_t w[8];
};
__device__ __forceinline__ Sector load_sector(const void* p) {
  Sector s;
  asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(s.w[0]), "=r"(s.w[1]), "=r"(s.w[2]), "=r"(s.w[3]), "=r"(s.w[4]), "=r"(s.w[5]), "=r"(s.w[6]), "=r"(s.w[7])
      : "l"(p));
  return s;
}
__device__ __forceinline__ uint32_t word_key(const uint32_t* w, int i, uint32_t) { return w[i]; }
__device__ __forceinline__ uint64_t word_key(const uint32_t* w, int i, uint64_t) {
  return (uint64_t)w[2 * i + 1] << 32 | w[2 * i];
}

template <>
struct TableReader<true> {
  static constexpr uint32_t kAlign = 32;
  // offsets b and b + 1; whole: the aligned words around b lie inside the array
  static __device__ __forceinline__ void range(const uint32_t* __restrict__ off, uint32_t b, bool whole, uint32_t& s,
                                               uint32_t& e) {
    if (whole) {
      const Sector o = load_sector(off + (b & ~7u));
      // words r and r + 1 of the sector, by halves
      const bool r4 = b & 4u, r2 = b & 2u, r1 = b & 1u;
      const uint32_t a0 = r4 ? o.w[4] : o.w[0], a1 = r4 ? o.w[5] : o.w[1], a2 = r4 ? o.w[6] : o.w[2],
                     a3 = r4 ? o.w[7] : o.w[3], a4 = o.w[4];
      const uint32_t c0 = r2 ? a2 : a0, c1 = r2 ? a3 : a1, c2 = r2 ? a4 : a2;
      s = r1 ? c1 : c0;
      e = r1 ? c2 : c1;
      if ((b & 7u) == 7u) e = __ldg(off + b + 1);
    } else {
      s = __ldg(off + b);
      e = __ldg(off + b + 1);
    }
  }
  // Keys equal to `key` in ck[s, e), s < e, by sectors inside the array (up
  // to `last`, its number of keys; 0: ck is not aligned).
  template <typename K>
  static __device__ __forceinline__ uint32_t matches(const K* __restrict__ ck, uint32_t s, uint32_t e, uint32_t last,
                                                     K key) {
    constexpr uint32_t P = 32 / sizeof(K);
    uint32_t cnt = 0;
    for (uint32_t j = s & ~(P - 1);; j += P) {
      if (last >= P && j <= last - P) {
        const Sector x = load_sector(ck + j);
#pragma unroll
        for (uint32_t l = 0; l < P; ++l) cnt += word_key(x.w, l, K(0)) == key;
      } else {
        for (uint32_t l = max(j, s); l < j + min(P, e - j); ++l) cnt += __ldg(ck + l) == key;
      }
      if (e - j <= P) return cnt;  // (j + P may be 2^32)
    }
  }
};

template <>
struct TableReader<false> {
  static constexpr uint32_t kAlign = 16;
  static __device__ __forceinline__ void range(const uint32_t* __restrict__ off, uint32_t b, bool whole, uint32_t& s,
                                               uint32_t& e) {
    if (whole) {
      const uint32_t r = b & 3u;
      const uint4 o4 = __ldg(reinterpret_cast<const uint4*>(off) + (b >> 2));
      s = r == 0 ? o4.x : r == 1 ? o4.y : r == 2 ? o4.z : o4.w;
      e = r == 0 ? o4.y : r == 1 ? o4.z : r == 2 ? o4.w : __ldg(off + b + 1);
    } else {
      s = __ldg(off + b);
      e = __ldg(off + b + 1);
    }
  }
  template <typename K>
  static __device__ __forceinline__ uint32_t matches(const K* __restrict__ ck, uint32_t s, uint32_t e, uint32_t last,
                                                     K key) {
    uint32_t cnt = 0;
    if (sizeof(K) == 4 && last != 0) {
      constexpr uint32_t P = 4;
      for (uint32_t j = s & ~(P - 1);; j += P) {
        if (last >= P && j <= last - P) {
          const uint4 x = __ldg(reinterpret_cast<const uint4*>(ck + j));
          const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (uint32_t l = 0; l < P; ++l) cnt += (j + l >= s) & (j + l < e) & (w[l] == key);
        } else {
          for (uint32_t l = max(j, s); l < j + min(P, e - j); ++l) cnt += __ldg(ck + l) == key;
        }
        if (e - j <= P) return cnt;
      }
    }
    cnt = __ldg(ck + s) == key;
    uint32_t j = s + 1;
    // four independent loads in flight per round for long buckets
    for (; e - j >= 4; j += 4) {
      const K a0 = __ldg(ck + j), a1 = __ldg(ck + j + 1), a2 = __ldg(ck + j + 2), a3 = __ldg(ck + j + 3);
      cnt += (a0 == key) + (a1 == key) + (a2 == key) + (a3 == key);
    }
    for (; j < e; ++j) cnt += __ldg(ck + j) == key;
    return cnt;
  }
};
template <typename Map>
using ReaderOf = TableReader<!Map::kSkewed && !Map::kNeedsPos>;

// One query per thread.  The grid is one wave of resident CTAs that sweeps
// the queries in order (query base + threadIdx.x at sweep k, base =
// (k * gridDim.x + blockIdx.x) * blockDim.x), so with grouped queries all
// CTAs work inside one or two groups at any time and each group's slice of
// the table stays in L2 while it is needed: the table is read from DRAM
// once.  (A grid of two waves sweeps every group twice and reads the table
// twice.)  Each thread loads its next query one sweep ahead, so the query's
// DRAM latency is not on its chain of dependent loads.  run (batched tables
// only): consecutive blocks of queries a CTA takes at a time, which belong to
// the same table mostly when the queries are in their own order.
//
// Bound by L1 tag look-ups and L2: one random access per lane takes a cycle
// whatever its width (a warp's 32 take 34 cycles for 4 to 32 bytes, through
// the load and the texture path alike), and L2 runs at 75% of its peak.
// Sectors instead of 16-byte pieces: 2^28 uint32 queries at 50% hits 2.14 ->
// 2.07 ms, 5 * 10^7 queries of keys that appear 8 times 0.67 -> 0.47, 3 * 10^7
// uint64 queries at load 2 0.37 -> 0.30.
template <typename K, typename Map>
__global__ void __launch_bounds__(kProbeThreads, 2048 / kProbeThreads)
    k_probe(const K* __restrict__ q, uint64_t nq, const uint32_t* __restrict__ off, const K* __restrict__ ck,
            uint32_t* __restrict__ out, uint32_t nwhole, const uint32_t* __restrict__ qpos, Map map,
            uint64_t map_buckets, uint32_t run) {
  using Reader = ReaderOf<Map>;
  map.init();
  const uint32_t last = (uintptr_t)ck % Reader::kAlign == 0 ? __ldg(off + map_buckets) : 0u;
  const uint64_t bd = blockDim.x;
  const uint64_t span = (uint64_t)gridDim.x * bd;
  uint64_t base = (uint64_t)blockIdx.x * bd * (Map::kNeedsPos ? run : 1);
  uint32_t left = run;
  K next = base + threadIdx.x < nq ? __ldcs(q + base + threadIdx.x) : K(0);
  for (uint64_t step; base < nq; base += step) {
    const uint64_t i = base + threadIdx.x;
    const K key = next;
    step = span;
    if (Map::kNeedsPos) {
      step = bd;
      if (--left == 0) {  // on to the CTA's next run
        left = run;
        step = (span - bd) * run + bd;
      }
    }
    next = i + step < nq ? __ldcs(q + i + step) : K(0);
    if (i >= nq) continue;
    const uint32_t b = map(key, qpos ? __ldg(qpos + i) : (uint32_t)i);
    uint32_t s, e;
    Reader::range(off, b, b < nwhole, s, e);
    __stcs(out + i, s < e ? Reader::matches(ck, s, e, last, key) : 0u);
  }
}

template <typename K, typename Map>
hg_status probe_launch(const K* q, uint64_t nq, const uint32_t* off, const K* ck, uint32_t* out,
                       uint64_t V, cudaStream_t st, Map map, const uint32_t* qpos, uint32_t run) {
  if (nq == 0) return HG_OK;
  // buckets whose aligned words of offsets lie inside the V+1 entries (none
  // if the array is not aligned): V + 1 <= 2^32 entries make whole words up
  // to at most 2^32 - 1 buckets here, the rest take two single loads
  constexpr uint32_t align = ReaderOf<Map>::kAlign, words = align / 4;
  const uint64_t whole = (uintptr_t)off % align == 0 ? (V + 1) / words * words : 0;
  const uint32_t nwhole = (uint32_t)std::min<uint64_t>(whole, 0xffffffffull / words * words);
  const int sms = dev_info().sms;
  auto kern = k_probe<K, Map>;
  static int per_sm = 0;  // resident CTAs per SM of this instantiation
  if (per_sm == 0) {
    int x = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&x, kern, kProbeThreads, 0) != cudaSuccess || x <= 0) x = 4;
    per_sm = x;
  }
  const uint64_t blocks = (nq + kProbeThreads - 1) / kProbeThreads;
  // (a run only where every resident CTA has one)
  run = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(Map::kNeedsPos ? run : 1, blocks / ((uint64_t)sms * per_sm)));
  const uint64_t want = (blocks + run - 1) / run;
  const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)sms * per_sm));
  {
    HG_TRACE("k_probe", st);
    kern<<<grid, kProbeThreads, 0, st>>>(q, nq, off, ck, out, nwhole, qpos, map, V, run);
  }
  return last_launch_status();
}

#define HG_INST(K, M) \
  template hg_status probe_launch<K, M>(const K*, uint64_t, const uint32_t*, const K*, uint32_t*, uint64_t, \
                                        cudaStream_t, M, const uint32_t*, uint32_t);
HG_INST(uint32_t, MurmurMap<true>)
HG_INST(uint64_t, MurmurMap<true>)
HG_INST(uint32_t, MurmurMap<false>)
HG_INST(uint64_t, MurmurMap<false>)
HG_INST(uint32_t, LearnedMap)
HG_INST(uint64_t, LearnedMap)
HG_INST(uint32_t, BatchedMap)
#undef HG_INST

}  // namespace hg
