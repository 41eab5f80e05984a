// HashGraph build: V2 (Alg. 2, two-level, shared-memory bins) and V1 (Alg. 1).
//
// V2 on GB300 is organised as three streaming passes plus an on-chip finish:
//   k_hist       per input chunk g: histogram of bins (bin = bucket >> s),
//                bins held in shared memory (Alg. 2 Phase 1, "Bin Counting")
//   k_colscan    per bin: exclusive prefix over chunks; bin totals
//   k_scan_bins  exclusive scan of bin totals -> bin starts (Phase 2 prefix
//                sum); the order mode (see below)
//   k_partition  pass A: chunk -> super-bins (256-way partition);
//                pass B: (super-bin, chunk) -> bins (<=256-way partition)
//                (Phase 2, "Bin Placement and Data Reorganization")
//   k_binbuild   per bin, in shared memory: local bucket index, counting
//                sort, CSR offsets and edges (Phase 3, "HashGraph Creation")
//                bins larger than shared memory are streamed by one CTA each
// The table comes out in the canonical order (bucket, then input position)
// without atomics deciding any position: either both partitions are stable
// and the bin build ranks each bucket by bin position, or (implicit ids and
// every bin in shared memory: order mode 0) the partitions rank tiles in any
// order and the bin build ranks each bucket by id, which is the position.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <mutex>
#include <unordered_map>

#include "hg_build.cuh"
#include "hg_trace.h"
#include "hg_partition.cuh"
#include "hg_scan.cuh"
#include "hg_probe.cuh"

namespace hg {

// ===========================================================================
// Plan
// ===========================================================================
static int ceil_log2_u64(uint64_t x) {
  int l = 0;
  while ((1ull << l) < x) ++l;
  return l;
}

// stream_runs' shared memory after the cursors: tile keys and ids, four u16
// tile arrays, the ranking counters and a scan scratch (last 128 bytes)
__host__ __device__ inline size_t big_rest_bytes(int kb) {
  return align_up((size_t)kBigTile * (kb + 4) + 4 * (size_t)kBigTile * 2, 16) + (size_t)rank_words<kBinNW>() * 4 +
         32 * 4;
}

size_t big_smem_bytes(int kb, uint32_t nb) { return align_up((size_t)nb * 4, 16) + big_rest_bytes(kb) + 64; }

size_t part_smem_bytes(int kb, bool ids_in, int ipt, bool item_list, int nw) {
  const size_t tile = (size_t)nw * 32 * ipt;
  const size_t tb = tile + 16;
  const size_t rw = (size_t)256 * (nw + 1 + (nw & 1));  // rank_words<nw>()
  size_t b = 2 * tb * kb + (ids_in ? 2 * tb * 4 : 0) + tile * (kb + 4 + 1) + rw * 4 +
             2 * 256 * 4;
  return align_up(b, 16) + (item_list ? 2 * kMaxItemsPerCta * 4 : 0) + 32 * 4 + 2 * 8 + 64;
}

bool make_plan_v2(const hg_config* cfg, uint64_t n, Plan* p) {
  const DevInfo& di = dev_info();
  p->kb = cfg->key_type == HG_KEY_U64 ? 8 : 4;
  p->n = n;
  p->V = cfg->num_buckets;
  p->emax = p->kb == 4 ? kBinEmaxU32 : kBinEmaxU64;
  p->tpb = cfg->threads_per_bin;  // 0 (automatic), 512 or 1024
  const uint64_t V = p->V;
  int s;
  if (cfg->bin_shift) {
    s = (int)cfg->bin_shift;
  } else {
    const double target = 0.75 * p->emax;
    const double bpb = n ? target * (double)V / (double)n : (double)V;
    s = bpb <= 1.0 ? 0 : (int)std::floor(std::log2(bpb));
  }
  if (!cfg->bin_shift) {
    s = std::min(s, (int)kMaxBinShift);
    // small builds: 128 bins all the same, about one per SM, rather than a
    // few large ones
    s = std::min(s, std::max(0, ceil_log2_u64(V) - 7));
  }
  s = std::max(s, ceil_log2_u64(V) - (int)kMaxBinsLog2);
  s = std::max(s, 0);
  if (s > (int)kMaxBinShift) return false;
  p->s = (uint32_t)s;
  const uint64_t nbins = ((V - 1) >> s) + 1;
  if (nbins > (1ull << kMaxBinsLog2)) return false;
  p->nbins = (uint32_t)nbins;
  const int lb = ceil_log2_u64(nbins);
  p->sshift = lb > 8 ? (uint32_t)(lb - 8) : 0u;
  p->nsb = (uint32_t)(((nbins - 1) >> p->sshift) + 1);
  const int sms = std::max(di.sms, 1);
  uint64_t chunk = std::max<uint64_t>(kPartTile, (n + 2 * sms - 1) / (2 * sms));
  chunk = (chunk + 15) / 16 * 16;
  p->chunk = chunk;
  p->G = (uint32_t)std::max<uint64_t>(1, (n + chunk - 1) / chunk);
  size_t o = sizeof(WsHeader);
  p->o_H = o;   o = align_up(o + (size_t)p->G * p->nbins * 4);
  p->o_C = o;   o = align_up(o + (size_t)p->G * p->nsb * 4);
  p->o_CT = o;  o = align_up(o + (size_t)p->nsb * 4);
  p->o_T = o;   o = align_up(o + (size_t)p->nbins * 4);
  p->o_BS = o;  o = align_up(o + ((size_t)p->nbins + 1) * 4);
  p->o_ovf = o; o = align_up(o + (size_t)p->nbins * 4);
  // a huge bin holds more than kHugeSeg edges, so there are at most n / kHugeSeg
  // of them and their segments number at most 2 n / kHugeSeg
  p->max_rows = (uint32_t)(2 * (n / kHugeSeg) + 2);
  p->o_hlist = o;   o = align_up(o + (size_t)(n / kHugeSeg + 1) * 3 * 4);
  p->o_rowdesc = o; o = align_up(o + (size_t)p->max_rows * 2 * 4);
  p->o_rowcnt = o;  o = align_up(o + (size_t)p->max_rows * ((size_t)1 << p->s) * 4);
  p->o_bk = o;  o = align_up(o + ((size_t)n + 16) * p->kb);
  p->o_bi = o;  o = align_up(o + ((size_t)n + 16) * 4);
  p->total = o;
  return true;
}

// ===========================================================================
// Kernels
// ===========================================================================
template <typename K>
__device__ __forceinline__ void unpack16(const uint4& x, K (&k)[16 / sizeof(K)]);
template <>
__device__ __forceinline__ void unpack16<uint32_t>(const uint4& x, uint32_t (&k)[4]) {
  k[0] = x.x; k[1] = x.y; k[2] = x.z; k[3] = x.w;
}
template <>
__device__ __forceinline__ void unpack16<uint64_t>(const uint4& x, uint64_t (&k)[2]) {
  k[0] = ((uint64_t)x.y << 32) | x.x;
  k[1] = ((uint64_t)x.w << 32) | x.z;
}

// Shared memory of k_hist: the histogram (at least 1 KB), then the bucket
// map's staged tables (Map::kStageBytes).
__host__ __device__ inline size_t hist_stage_offset(uint32_t nbins) {
  return align_up((size_t)(nbins < 256u ? 256u : nbins) * 4, 16);
}

// Phase 1: per-chunk bin histogram in shared memory; per super-bin sums.
// header (may be null): the workspace header, cleared here for the kernels
// that follow.
template <typename K, typename Map>
__global__ void __launch_bounds__(kHistThreads) k_hist(const K* __restrict__ keys, uint64_t n,
                                                       uint64_t chunk, uint32_t s, uint32_t nbins,
                                                       uint32_t sshift, uint32_t nsb,
                                                       uint32_t* __restrict__ H,
                                                       uint32_t* __restrict__ C, Map map,
                                                       uint32_t stage_bytes, WsHeader* header) {
  extern __shared__ __align__(16) uint32_t hist[];
  if (header != nullptr && blockIdx.x == 0 && threadIdx.x < sizeof(WsHeader) / 4)
    reinterpret_cast<uint32_t*>(header)[threadIdx.x] = 0;
  map.init();
  map.stage((uint8_t*)hist + hist_stage_offset(nbins), stage_bytes);
  for (uint32_t i = threadIdx.x; i < nbins; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  constexpr int per = 16 / sizeof(K);
  const uint64_t c0 = (uint64_t)blockIdx.x * chunk;
  const uint64_t c1 = min(c0 + chunk, n);
  // 16-byte vector loads between the first and the last 16-byte address
  // boundary of the chunk (keys may start anywhere: a slab of a larger
  // build), single loads before and after
  const uint64_t off = ((uintptr_t)keys / sizeof(K)) % per;
  const uint64_t y0 = (c0 + off + per - 1) / per * per, y1 = (c1 + off) / per * per;
  const uint64_t b0 = y1 > y0 ? y0 - off : c1, b1 = y1 > y0 ? y1 - off : c1;
  const uint4* kv = reinterpret_cast<const uint4*>(keys + b0);
  const uint64_t nv = (b1 - b0) / per;
  const uint32_t bd = blockDim.x;
  uint64_t v = threadIdx.x;
  for (; v + 3 * (uint64_t)bd < nv; v += 4 * (uint64_t)bd) {
    uint4 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = __ldcs(kv + v + u * bd);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      K k[per];
      unpack16<K>(x[u], k);
      const uint32_t p0 = (uint32_t)(b0 + (v + u * bd) * per);
#pragma unroll
      for (int e = 0; e < per; ++e) atomicAdd(&hist[map(k[e], p0 + e) >> s], 1u);
    }
  }
  for (; v < nv; v += bd) {
    K k[per];
    unpack16<K>(__ldcs(kv + v), k);
    const uint32_t p0 = (uint32_t)(b0 + v * per);
#pragma unroll
    for (int e = 0; e < per; ++e) atomicAdd(&hist[map(k[e], p0 + e) >> s], 1u);
  }
  for (uint64_t i = c0 + threadIdx.x; i < b0; i += bd) atomicAdd(&hist[map(keys[i], (uint32_t)i) >> s], 1u);
  for (uint64_t i = b1 + threadIdx.x; i < c1; i += bd) atomicAdd(&hist[map(keys[i], (uint32_t)i) >> s], 1u);
  __syncthreads();
  uint32_t* row = H + (uint64_t)blockIdx.x * nbins;
  for (uint32_t i = threadIdx.x; i < nbins; i += bd) row[i] = hist[i];
  const uint32_t lane = lane_id(), w = threadIdx.x >> 5, nw = bd >> 5;
  const uint32_t bps = 1u << sshift;
  for (uint32_t sb = w; sb < nsb; sb += nw) {
    uint32_t sum = 0;
    for (uint32_t j = lane; j < bps; j += 32) {
      const uint32_t b = (sb << sshift) + j;
      if (b < nbins) sum += hist[b];
    }
    sum = warp_sum(sum);
    if (lane == 0) C[(uint64_t)blockIdx.x * nsb + sb] = sum;
  }
}

// Exclusive prefix down every column of a rows x cols table, in place;
// column totals to coltot (may be null).  A CTA takes 32 consecutive columns
// (lane = column) and splits the rows into 32 segments (warp = segment), so
// every row access of a warp is one coalesced 128-byte line: segment sums,
// a scan of each column's 32 segment sums, then the segment rewritten with
// its prefix.  Launch with colscan_launch().
constexpr int kColScanThreads = 1024;
__global__ void __launch_bounds__(kColScanThreads) k_colscan(uint32_t* __restrict__ tab, uint32_t rows,
                                                             uint32_t cols, uint32_t* __restrict__ coltot) {
  __shared__ uint32_t seg[32][33];
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
  const uint32_t c = blockIdx.x * 32u + lane;
  const uint32_t R = (rows + 31u) / 32u;
  const uint32_t r0 = min(w * R, rows), r1 = min(r0 + R, rows);
  uint32_t* p = tab + c;
  uint32_t sum = 0;
  if (c < cols)
    for (uint32_t r = r0; r < r1; ++r) sum += p[(uint64_t)r * cols];
  seg[w][lane] = sum;
  __syncthreads();
  {  // warp w scans column w's 32 segment sums (lane = segment)
    const uint32_t v = seg[lane][w];
    const uint32_t incl = warp_incl_scan(v);
    seg[lane][w] = incl - v;
  }
  __syncthreads();
  if (c >= cols) return;
  uint32_t run = seg[w][lane];
  for (uint32_t r = r0; r < r1; ++r) {
    const uint32_t v = p[(uint64_t)r * cols];
    p[(uint64_t)r * cols] = run;
    run += v;
  }
  if (coltot && w == 31) coltot[c] = run;
}

static void colscan_launch(uint32_t* tab, uint32_t rows, uint32_t cols, uint32_t* coltot, cudaStream_t st) {
  k_colscan<<<(cols + 31) / 32, kColScanThreads, 0, st>>>(tab, rows, cols, coltot);
}

// Bins above kHugeSeg edges: list entries (bin, first row, rows) and one
// row (bin, segment) per kHugeSeg-edge segment.  Null list: no such split.
struct HugeArgs {
  uint32_t* list;
  uint32_t* count;
  uint32_t* rows;
  uint32_t* rowdesc;
  uint32_t max_rows;
  uint32_t* status;
};

// Exclusive scan of the bin totals (one CTA); list of bins too large for the
// shared-memory bin build (huge ones split into segments); closing CSR
// offset offsets[V] = n; the bins' write cursors of k_partition_any's pass B
// (cur_bin, may be null); with wide_count, the number of bins of more than
// wide_lo and at most emax edges (the bin build's second launch).
__global__ void __launch_bounds__(1024) k_scan_bins(const uint32_t* __restrict__ T, uint32_t nbins,
                                                    uint32_t* __restrict__ BS, uint32_t emax,
                                                    uint32_t* __restrict__ ovf_list,
                                                    uint32_t* __restrict__ ovf_count,
                                                    uint32_t* __restrict__ offsets, uint64_t V,
                                                    uint32_t n_end, HugeArgs h, uint32_t* order,
                                                    uint32_t wide_lo = 0, uint32_t* wide_count = nullptr,
                                                    uint32_t* __restrict__ cur_bin = nullptr) {
  // Each warp scans a contiguous range of whole 32-bin rows (lane = bin of
  // the row), so every access is coalesced: the range's sum, an exclusive
  // scan of the warp sums, then the range again from its base.
  __shared__ uint32_t wbase[32];
  __shared__ uint32_t wtotal;
  const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t rows = (nbins + 31u) / 32u, per = (rows + nw - 1) / nw;
  const uint32_t row0 = min(w * per, rows), row1 = min(row0 + per, rows);
  uint32_t part = 0;
  for (uint32_t r = row0; r < row1; ++r) {
    const uint32_t i = r * 32u + lane;
    part += i < nbins ? T[i] : 0u;
  }
  part = warp_sum(part);
  if (lane == 0) wbase[w] = part;
  __syncthreads();
  if (w == 0) {
    const uint32_t v = lane < nw ? wbase[lane] : 0u;
    const uint32_t incl = warp_incl_scan(v);
    if (lane < nw) wbase[lane] = incl - v;
    if (lane == 31) wtotal = incl;
  }
  __syncthreads();
  uint32_t base = wbase[w];
  for (uint32_t r = row0; r < row1; ++r) {
    const uint32_t i = r * 32u + lane;
    const uint32_t t = i < nbins ? T[i] : 0u;
    const uint32_t incl = warp_incl_scan(t);
    if (i < nbins) {
      const uint32_t start = base + incl - t;
      BS[i] = start;
      if (cur_bin) cur_bin[i] = start;
    }
    base += __shfl_sync(kFull, incl, 31);
    if (wide_count && i < nbins && t > wide_lo && t <= emax) atomicAdd(wide_count, 1u);
    if (i >= nbins || t <= emax) continue;
    if (order) *order = 1u;  // this bin is built outside shared memory: stable partitions needed
    if (h.list == nullptr || t <= kHugeSeg) {
      ovf_list[atomicAdd(ovf_count, 1u)] = i;
      continue;
    }
    const uint32_t nr = (t + kHugeSeg - 1) / kHugeSeg;
    const uint32_t q0 = atomicAdd(h.rows, nr);
    if (q0 + nr > h.max_rows) {  // cannot happen: the bound counts every huge bin
      set_status(h.status, HG_ERR_OVERFLOW);
      continue;
    }
    const uint32_t k = atomicAdd(h.count, 1u);
    h.list[3 * k] = i;
    h.list[3 * k + 1] = q0;
    h.list[3 * k + 2] = nr;
    for (uint32_t x = 0; x < nr; ++x) {
      h.rowdesc[2 * (q0 + x)] = i;
      h.rowdesc[2 * (q0 + x) + 1] = x;
    }
  }
  if (threadIdx.x == 0) {
    BS[nbins] = wtotal;
    offsets[V] = n_end;
  }
}

// k_colscan and k_scan_bins in one, for builds of one partition pass (at most
// 256 bins) and few chunks: thread = (bin, quarter of the chunks), every
// count read once.  2^16 keys: one launch of 4 us for three of 10 us.
constexpr uint32_t kScanSmallChunks = 64;
__global__ void __launch_bounds__(1024) k_scan_small(uint32_t* __restrict__ C, uint32_t G, uint32_t nbins,
                                                     uint32_t* __restrict__ CT, uint32_t* __restrict__ BS,
                                                     uint32_t emax, uint32_t* __restrict__ ovf_list,
                                                     uint32_t* __restrict__ ovf_count, uint32_t* __restrict__ offsets,
                                                     uint64_t V, uint32_t n_end, uint32_t* order, uint32_t wide_lo,
                                                     uint32_t* wide_count) {
  constexpr uint32_t R = kScanSmallChunks / 4;
  __shared__ uint32_t part[4][256];
  __shared__ uint32_t wsum[32];
  const uint32_t b = threadIdx.x & 255u, q = threadIdx.x >> 8;
  uint32_t c[R], sum = 0;
#pragma unroll
  for (uint32_t i = 0; i < R; ++i) {
    const uint32_t g = q * R + i;
    c[i] = b < nbins && g < G ? C[(uint64_t)g * nbins + b] : 0u;
  }
#pragma unroll
  for (uint32_t i = 0; i < R; ++i) sum += c[i];
  part[q][b] = sum;
  __syncthreads();
  uint32_t run = 0, t = 0;
#pragma unroll
  for (uint32_t i = 0; i < 4; ++i) {
    run += i < q ? part[i][b] : 0u;
    t += part[i][b];
  }
#pragma unroll
  for (uint32_t i = 0; i < R; ++i) {
    const uint32_t g = q * R + i;
    if (b < nbins && g < G) C[(uint64_t)g * nbins + b] = run;
    run += c[i];
  }
  uint32_t total;
  const uint32_t start = block_excl_scan<uint32_t>(q == 0 ? t : 0u, wsum, &total);  // the first 256 threads' totals
  if (q == 0 && b < nbins) {
    CT[b] = t;
    BS[b] = start;
    if (wide_count && t > wide_lo && t <= emax) atomicAdd(wide_count, 1u);
    if (t > emax) {
      if (order) *order = 1u;
      ovf_list[atomicAdd(ovf_count, 1u)] = b;
    }
  }
  if (threadIdx.x == 0) {
    BS[nbins] = total;
    offsets[V] = n_end;
  }
}

// Phase 2 (both passes).  Pass A: items are input chunks; digit = super-bin.
// Pass B: items are (super-bin, group of gg consecutive chunks) sub-ranges of
// pass A's output, contiguous in memory; digit = bin inside the super-bin.
// A group's elements are in input order, so one running cursor per bin,
// started at the bin start plus the earlier chunks' counts, keeps the pass
// stable when its tiles are.  Tiles stream through shared memory by TMA bulk
// copies, double-buffered; each tile is partitioned (stably, or in any order
// with ANY) and written out as contiguous runs.
template <typename K>
struct PartArgs {
  const K* in_k;
  const uint32_t* in_i;  // null: ids are input positions
  K* out_k;
  uint32_t* out_i;
  uint64_t n, chunk;
  uint32_t G, s, sshift, nbins, nsb;
  uint32_t gg, ngroups;  // pass B: chunks per item, items per super-bin
  uint32_t piece;        // k_partition_any, pass B: tiles a CTA takes at a time
  const uint32_t* H;   // per (chunk, bin) exclusive column prefix; row 0 (all zero) is not read: it
                       // holds k_partition_any's cursors
  const uint32_t* C;   // per (chunk, super-bin) exclusive column prefix
  const uint32_t* CT;  // per super-bin totals
  const uint32_t* BS;  // bin starts
  uint32_t* status;
  uint32_t stage_bytes;  // shared memory after the kernel's own, for the bucket map's tables
  uint32_t* cur_bin;   // k_partition_any, pass B: next free element of every bin
  // order mode word (null: always stable); see k_partition
  const uint32_t* order;
  // optional: per tile (tiles start at multiples of the kernel's tile size),
  // the tile's count of every digit, nbins 16-bit entries per tile
  uint16_t* tile_counts;
};

// The stable partition.  The unordered one (partition_any) runs only when
// every bin fits the shared-memory bin build, which then restores the
// canonical order by id; k_scan_bins writes which it is (order mode).
template <typename K, typename Map, bool PASS_B, int IPT, int NW>
__device__ __forceinline__ void partition_stable(const PartArgs<K>& a, Map& map) {
  constexpr uint32_t TILE = NW * 32 * IPT;
  constexpr uint32_t TB = TILE + 16;
  static_assert(TILE <= 65536, "tile indexes are packed into 16 bits");
  const bool has_ids = PASS_B || a.in_i != nullptr;
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sp = smem;
  // staging buffer b of keys at kin0 + b * TB, of ids at iin0 + b * TB
  K* const kin0 = (K*)sp; sp += 2 * TB * sizeof(K);
  uint32_t* const iin0 = has_ids ? (uint32_t*)sp : nullptr;
  if (has_ids) sp += 2 * TB * 4;
  K* sk = (K*)sp; sp += TILE * sizeof(K);
  uint32_t* sv = (uint32_t*)sp; sp += TILE * 4;
  uint32_t* wc = (uint32_t*)sp; sp += rank_words<NW>() * 4;
  uint32_t* dstart = (uint32_t*)sp; sp += 256 * 4;
  uint32_t* cursor = (uint32_t*)sp; sp += 256 * 4;
  uint8_t* sd = sp; sp += TILE;
  sp = (uint8_t*)(((uintptr_t)sp + 15) & ~(uintptr_t)15);
  uint32_t* ilo = (uint32_t*)sp; sp += PASS_B ? kMaxItemsPerCta * 4 : 0;
  uint32_t* ihi = (uint32_t*)sp; sp += PASS_B ? kMaxItemsPerCta * 4 : 0;
  uint32_t* wsum = (uint32_t*)sp; sp += 32 * 4;
  uint64_t* bar = (uint64_t*)sp; sp += 2 * 8;
  uint8_t* stage = sp;  // a.stage_bytes (16-byte aligned)

  map.init();
  map.stage(stage, a.stage_bytes);
  const uint32_t koff = align_first<sizeof(K)>(a.in_k), ioff = has_ids ? align_first<4>(a.in_i) : 0u;
  for (int i = threadIdx.x; i < rank_words<NW>(); i += blockDim.x) wc[i] = 0;
  const uint64_t nitems = PASS_B ? (uint64_t)a.nsb * a.ngroups : (uint64_t)a.G;
  if (PASS_B) {
    // input ranges of this CTA's items, gathered once (keeps global loads out
    // of the tile loop's control path)
    for (uint64_t j = threadIdx.x, item = blockIdx.x + j * gridDim.x; item < nitems;
         j += blockDim.x, item = blockIdx.x + j * gridDim.x) {
      const uint32_t sb = (uint32_t)(item / a.ngroups), grp = (uint32_t)(item % a.ngroups);
      const uint32_t g0 = grp * a.gg, g1 = min(g0 + a.gg, a.G);
      const uint32_t base = a.BS[sb << a.sshift];
      ilo[j] = base + a.C[(uint64_t)g0 * a.nsb + sb];
      ihi[j] = base + (g1 < a.G ? a.C[(uint64_t)g1 * a.nsb + sb] : a.CT[sb]);
    }
  }
  // This CTA's items are blockIdx.x + j * gridDim.x for j = 0, 1, ...; the
  // tile stream walks them by j (32-bit), tiles of TILE elements.
  const uint32_t nmine = blockIdx.x < nitems ? (uint32_t)((nitems - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0u;
  auto item_range = [&](uint32_t j, uint64_t& i0, uint64_t& i1) {
    if (!PASS_B) {
      i0 = ((uint64_t)blockIdx.x + (uint64_t)j * gridDim.x) * a.chunk;
      i1 = min(i0 + a.chunk, a.n);
    } else {
      i0 = ilo[j];
      i1 = ihi[j];
    }
  };
  struct Ref {
    uint32_t j;
    bool ok;
    uint64_t t0, t1;
  };
  auto first_from = [&](uint32_t j) -> Ref {
    for (; j < nmine; ++j) {
      uint64_t i0, i1;
      item_range(j, i0, i1);
      if (i1 > i0) return Ref{j, true, i0, min(i0 + TILE, i1)};
    }
    return Ref{0, false, 0, 0};
  };
  auto next_of = [&](const Ref& r) -> Ref {
    uint64_t i0, i1;
    item_range(r.j, i0, i1);
    if (r.t1 < i1) return Ref{r.j, true, r.t1, min(r.t1 + TILE, i1)};
    return first_from(r.j + 1);
  };
  auto issue = [&](const Ref& r, int buf) {
    if (threadIdx.x == 0) {
      const TileSpan<sizeof(K)> sk_ = tile_span<sizeof(K)>(koff, r.t0, r.t1);
      uint32_t bytes = sk_.bytes();
      TileSpan<4> si_{};
      if (has_ids) {
        si_ = tile_span<4>(ioff, r.t0, r.t1);
        bytes += si_.bytes();
      }
      mbar_arrive_expect_tx(&bar[buf], bytes);
      if (sk_.body) tma_load_1d(kin0 + buf * TB + sk_.dst(), a.in_k + sk_.b0, sk_.bytes(), &bar[buf]);
      if (has_ids && si_.body) tma_load_1d(iin0 + buf * TB + si_.dst(), a.in_i + si_.b0, si_.bytes(), &bar[buf]);
    }
  };

  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();

  Ref cur = first_from(0);
  if (!cur.ok) return;
  issue(cur, 0);
  uint32_t cur_j = ~0u, sb = 0;
  int ndig = 0;
  const uint32_t seg0 = (threadIdx.x >> 5) * (32u * IPT), lane = lane_id();
  for (uint32_t it = 0; cur.ok; ++it) {
    const int buf = it & 1;
    const Ref nxt = next_of(cur);
    if (nxt.ok) issue(nxt, buf ^ 1);
    if (!mbar_wait_block(&bar[buf], (it >> 1) & 1u, a.status)) return;
    const TileSpan<sizeof(K)> sk_ = tile_span<sizeof(K)>(koff, cur.t0, cur.t1);
    TileSpan<4> si_{};
    if (has_ids) si_ = tile_span<4>(ioff, cur.t0, cur.t1);
    // elements outside the 16-byte boundaries (only where a tile starts or
    // ends unaligned) come in by plain loads; the barrier is needed only then
    bool sync_needed = sk_.edges() || (has_ids && si_.edges());
    load_edges<sizeof(K)>(kin0 + buf * TB, a.in_k, sk_);
    if (has_ids) load_edges<4>(iin0 + buf * TB, a.in_i, si_);
    if (cur.j != cur_j) {  // cursors are first read after tile_partition_fast's first barrier
      cur_j = cur.j;
      const uint32_t item = blockIdx.x + cur.j * gridDim.x;
      if (!PASS_B) {
        ndig = (int)a.nsb;
        for (int d = threadIdx.x; d < ndig; d += blockDim.x)
          cursor[d] = a.BS[(uint32_t)d << a.sshift] + a.C[(uint64_t)item * a.nsb + d];
      } else {
        sb = item / a.ngroups;
        const uint32_t g = (item - sb * a.ngroups) * a.gg;
        const uint32_t b0 = sb << a.sshift;
        ndig = (int)min(1u << a.sshift, a.nbins - b0);
        for (int d = threadIdx.x; d < ndig; d += blockDim.x)
          cursor[d] = a.BS[b0 + d] + (g ? a.H[(uint64_t)g * a.nbins + b0 + d] : 0u);
      }
    }
    if (sync_needed) __syncthreads();  // block-uniform condition
    const uint32_t cnt = (uint32_t)(cur.t1 - cur.t0);
    const K* kk = kin0 + buf * TB + sk_.lead();
    const uint32_t* ii = has_ids ? iin0 + buf * TB + si_.lead() : nullptr;
    K key[IPT];
    uint32_t val[IPT], dig[IPT];
#pragma unroll
    for (int r = 0; r < IPT; ++r) {
      const uint32_t idx = seg0 + (uint32_t)r * 32u + lane;
      if (idx < cnt) {
        key[r] = kk[idx];
        val[r] = has_ids ? ii[idx] : idx;
        const uint32_t bucket = map(key[r], has_ids ? val[r] : (uint32_t)(cur.t0 + idx));
        dig[r] = PASS_B ? (bucket >> a.s) - (sb << a.sshift) : bucket >> (a.s + a.sshift);
      } else {
        key[r] = 0;
        val[r] = 0;
        dig[r] = 0;
      }
    }
    if (has_ids)
      tile_partition_fast<K, IPT, NW, false>(key, val, dig, cnt, ndig, sk, sv, sd, wc, dstart, cursor, wsum, a.out_k,
                                             a.out_i, 0u);
    else
      tile_partition_fast<K, IPT, NW, true>(key, val, dig, cnt, ndig, sk, sv, sd, wc, dstart, cursor, wsum, a.out_k,
                                            a.out_i, (uint32_t)cur.t0);
    cur = nxt;
  }
}

// The stable partition as a kernel of its own (explicit ids, pass B, slabs,
// the sample sort): returns at once when the order mode (if there is one)
// asks for the other.
template <typename K, typename Map, bool PASS_B, int IPT, int NW, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB) k_partition(PartArgs<K> a, Map map) {
  if (a.order != nullptr && *(volatile const uint32_t*)a.order == 0u) return;
  partition_stable<K, Map, PASS_B, IPT, NW>(a, map);
}

// Shared memory of k_partition_any (see there).
static size_t part_any_smem(int kb, bool ids, int tile, int digits) {
  return align_up((size_t)tile * (kb + 4 + (ids ? 1 : 0)), 16) + 4 * (size_t)digits * 4;
}

// The same passes with equal digits in any order: an element's rank in its
// digit is the old value of a shared-memory atomic, so a tile costs one
// atomic per element and one warp's scan of the DIG counters (256 or 512).
// Pass A (and the query partition): a CTA takes chunks, whose tiles follow
// one another within each digit from the chunk's own start in it.
// Pass B: the CTAs take equal pieces of pass A's output in turn, so all of
// them work in a window of a few super-bins, and every tile takes its room in
// a bin from the bin's one cursor (global atomics).  The pieces are equal
// whatever the order or skew of the input.
//   1. digit and rank of every element, packed in a register
//   2. one warp: scan of the digit counts, room taken, counters cleared
//   3. elements to their place in the digit-sorted tile in shared memory;
//      output base of every digit (delta)
//   4. the next tile's elements are loaded to registers, then the sorted tile
//      is written out as runs per digit
// IDS: the elements carry ids (else an id is the element's input position,
// staged as its index in the tile next to its digit).
//
// Bound by shared-memory wavefronts: about 27 per 32 elements with the loads
// and stores, of which the random accesses (atomic, digit start, placement)
// make 12.  Loads go straight to registers and shared memory holds one tile
// only, so tiles are as large as the registers allow (a run's length, TILE /
// digits, sets how well the stores coalesce), or two CTAs share the SM.
// 2^28 uint32 keys, against tiles staged by TMA through a double buffer:
// pass A 1.18 -> 0.96 ms, pass B 1.41 -> 1.08, queries 1.10 -> 0.92; 2^26
// uint64 keys under the learned map 0.63 -> 0.47, 0.78 -> 0.46, 0.49 -> 0.41.
template <typename K, typename Map, bool PASS_B, bool IDS, int DIG, int NT, int IPT>
__device__ __forceinline__ void partition_any(const PartArgs<K>& a, Map& map) {
  constexpr uint32_t TILE = NT * IPT;
  static_assert(TILE <= 65536 && TILE % 16 == 0, "tile indexes are packed into 16 bits");
  static_assert(DIG == 256 || (DIG == 512 && !IDS && NT >= 512), "digits fit their packings");
  constexpr int DBITS = DIG == 512 ? 9 : 8, PER = DIG / 32;
  constexpr bool kPair = sizeof(K) == 4;  // key and id (or index) staged as one 8-byte element
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sp = smem;
  uint2* const spair = (uint2*)sp;
  K* const sk = (K*)sp; sp += TILE * sizeof(K);
  uint32_t* const sv = (uint32_t*)sp; sp += TILE * 4;
  uint8_t* const sd = sp; sp += IDS ? TILE : 0;  // digits (with IDS); every size here is a multiple of 16
  uint32_t* const tcnt = (uint32_t*)sp; sp += DIG * 4;
  uint32_t* const dstart = (uint32_t*)sp; sp += DIG * 4;
  uint32_t* const delta = (uint32_t*)sp; sp += DIG * 4;
  uint32_t* const cursor = (uint32_t*)sp; sp += DIG * 4;  // pass A
  map.init();
  map.stage(sp, a.stage_bytes);
  const uint32_t tid = threadIdx.x, lane = tid & 31u;
  for (uint32_t d = tid; d < DIG; d += NT) tcnt[d] = 0;
  __syncthreads();
  // Tile stream: the tile starts at t0 and ends at most at `end`, the end of
  // its chunk (item) or of the part of its super-bin (item) in the CTA's
  // piece, which ends at lim.
  struct Ref {
    uint32_t item, t0, end, lim;
    bool ok;
  };
  const uint64_t span = PASS_B ? (uint64_t)a.piece * TILE : a.chunk;
  auto take = [&](uint64_t c) -> Ref {  // the c-th chunk or piece
    const uint64_t i0 = c * span;
    const uint32_t lo = (uint32_t)i0, lim = (uint32_t)min(i0 + span, a.n);
    if (i0 >= a.n) return Ref{0, 0, 0, 0, false};
    if (!PASS_B) return Ref{(uint32_t)c, lo, lim, lim, true};
    uint32_t x = 0, y = a.nsb;  // the last super-bin that starts at or before lo (of equal starts, the non-empty one)
    while (y - x > 1) {
      const uint32_t m = (x + y) >> 1;
      if (__ldg(a.BS + (m << a.sshift)) <= lo) x = m;
      else y = m;
    }
    return Ref{x, lo, min(__ldg(a.BS + min((x + 1) << a.sshift, a.nbins)), lim), lim, true};
  };
  uint64_t c_next = blockIdx.x;
  auto advance = [&](Ref& r) {
    r.t0 += min(r.end - r.t0, TILE);
    if (r.t0 < r.end) return;
    if (r.t0 < r.lim) {  // on to the piece's next super-bin that is not empty
      do r.end = min(__ldg(a.BS + min((++r.item + 1) << a.sshift, a.nbins)), r.lim);
      while (r.end <= r.t0);
      return;
    }
    r = take(c_next += gridDim.x);
  };
  K key[IPT];
  uint32_t id[IDS ? IPT : 1];
  auto load = [&](const Ref& r) {
    const K* const gk = a.in_k + r.t0 + tid;
    const uint32_t* const gi = IDS ? a.in_i + r.t0 + tid : nullptr;
    const uint32_t cnt = min(r.end - r.t0, TILE);
    if (cnt == TILE) {
#pragma unroll
      for (int c = 0; c < IPT; ++c) {
        key[c] = __ldcs(gk + c * NT);
        if (IDS) id[IDS ? c : 0] = __ldcs(gi + c * NT);
      }
    } else {
      const int left = (int)cnt - (int)tid;
#pragma unroll
      for (int c = 0; c < IPT; ++c) {
        key[c] = left > c * NT ? __ldcs(gk + c * NT) : K(0);
        if (IDS) id[IDS ? c : 0] = left > c * NT ? __ldcs(gi + c * NT) : 0u;
      }
    }
  };
  Ref cur = take(c_next);
  if (cur.ok) load(cur);
  const uint32_t shift = PASS_B ? a.s : a.s + a.sshift;
  const uint32_t dmask = PASS_B ? (1u << a.sshift) - 1u : 0xffffffffu;  // pass B: bin inside the super-bin
  uint32_t at = ~0u;  // chunk whose cursors are loaded
  while (cur.ok) {
    const uint32_t cnt = min(cur.end - cur.t0, TILE), t0 = cur.t0, item = cur.item;
    const int left = (int)cnt - (int)tid;
    if (!PASS_B && item != at) {  // first read by the scan, after a barrier
      at = item;
      if (tid < a.nsb) cursor[tid] = a.BS[tid << a.sshift] + a.C[(uint64_t)item * a.nsb + tid];
    }
    // every element through f(c): full tiles without a test per element
    auto each = [&](auto&& f) {
      if (cnt == TILE) {
#pragma unroll
        for (int c = 0; c < IPT; ++c) f(c);
      } else {
#pragma unroll
        for (int c = 0; c < IPT; ++c)
          if (left > c * NT) f(c);
      }
    };
    // 1. digits and ranks
    uint32_t dr[IPT];  // digit | rank << DBITS
    each([&](int c) {
      const uint32_t d = (map(key[c], IDS ? id[IDS ? c : 0] : t0 + tid + c * NT) >> shift) & dmask;
      dr[c] = d | (atomicAdd(&tcnt[d], 1u) << DBITS);
    });
    __syncthreads();
    // 2. scan of the counts (lane: PER consecutive digits)
    uint32_t room[PASS_B ? PER : 1];
    if (tid < 32) {
      uint32_t c[PER];
      uint32_t sum = 0;
#pragma unroll
      for (int i = 0; i < PER; i += 4) {
        uint4* const q = reinterpret_cast<uint4*>(tcnt + lane * PER + i);
        const uint4 x = *q;
        *q = make_uint4(0, 0, 0, 0);
        c[i] = x.x;
        c[i + 1] = x.y;
        c[i + 2] = x.z;
        c[i + 3] = x.w;
        sum += x.x + x.y + x.z + x.w;
      }
      uint32_t run = warp_incl_scan(sum) - sum;
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        const uint32_t d = lane * PER + i;
        if (PASS_B) {  // (back by the time step 3 is done)
          room[PASS_B ? i : 0] = c[i] ? atomicAdd(a.cur_bin + (item << a.sshift) + d, c[i]) : 0u;
        } else {
          const uint32_t at_d = cursor[d];
          delta[d] = at_d - run;
          cursor[d] = at_d + c[i];
          if (!IDS && a.tile_counts != nullptr && d < a.nbins)
            a.tile_counts[(uint64_t)(t0 / TILE) * a.nbins + d] = (uint16_t)c[i];
        }
        dstart[d] = run;
        run += c[i];
      }
    }
    __syncthreads();
    // 3. the digit-sorted tile
    each([&](int c) {
      const uint32_t d = dr[c] & (DIG - 1u), dest = dstart[d] + (dr[c] >> DBITS);
      const uint32_t v = IDS ? id[IDS ? c : 0] : (tid + c * NT) | (d << 16);
      if (kPair) {
        spair[dest] = make_uint2((uint32_t)key[c], v);
      } else {
        sk[dest] = key[c];
        sv[dest] = v;
      }
      if (IDS) sd[dest] = (uint8_t)d;
    });
    if (PASS_B && tid < 32) {
#pragma unroll
      for (int i = 0; i < PER; ++i) delta[lane * PER + i] = room[PASS_B ? i : 0] - dstart[lane * PER + i];
    }
    // 4. next tile's loads, this tile's stores
    advance(cur);
    if (cur.ok) load(cur);
    __syncthreads();
    auto out = [&](uint32_t j) {
      K k;
      uint32_t v;
      if (kPair) {
        const uint2 x = spair[j];
        k = (K)x.x;
        v = x.y;
      } else {
        k = sk[j];
        v = sv[j];
      }
      const uint32_t g = delta[IDS ? (uint32_t)sd[j] : v >> 16] + j;
      a.out_k[g] = k;
      a.out_i[g] = IDS ? v : t0 + (v & 0xffffu);
    };
    if (cnt == TILE) {
#pragma unroll 4
      for (int c = 0; c < IPT; ++c) out(tid + c * NT);
    } else {
      for (uint32_t j = tid; j < cnt; j += NT) out(j);
    }
    __syncthreads();
  }
}

// ... as a kernel of its own; returns at once when the order mode (if there is
// one) asks for the stable partition.
template <typename K, typename Map, bool PASS_B, bool IDS, int DIG, int NT, int IPT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_partition_any(PartArgs<K> a, Map map) {
  if (a.order != nullptr && *(volatile const uint32_t*)a.order != 0u) return;
  partition_any<K, Map, PASS_B, IDS, DIG, NT, IPT>(a, map);
}

// Pass A of small builds with implicit ids: whichever the order mode asks
// for, in one launch (a second one that returns at once costs 3 us).  Large
// builds launch the two forms apart: together their code is slower (2^28
// uint32 keys 1.01 against 0.96 ms).
template <typename K, typename Map>
__global__ void __launch_bounds__(PartA<K>::NT, PartA<K>::MINB) k_partition_a(PartArgs<K> a, Map map) {
  static_assert(PartA<K>::NT == kPartNW * 32, "both forms have the same threads");
  if (*(volatile const uint32_t*)a.order == 0u)
    partition_any<K, Map, false, false, 256, PartA<K>::NT, PartA<K>::IPT>(a, map);
  else
    partition_stable<K, Map, false, part_ipt_keys<K>(), kPartNW>(a, map);
}

// Bin totals after pass A, for builds of more bins than one shared-memory
// histogram of the whole input holds: the CTAs take equal pieces of pass A's
// output in turn and count a piece's bins super-bin by super-bin (up to 256
// bins each), then add the counts to T (zeroed before).
constexpr uint32_t kLatePiece = 32768;
template <typename K, typename Map>
__global__ void __launch_bounds__(512) k_hist_late(PartArgs<K> a, uint32_t* __restrict__ T, Map map) {
  __shared__ uint32_t hist[256];
  map.init();
  const uint32_t dmask = (1u << a.sshift) - 1u;
  for (uint64_t i0 = (uint64_t)blockIdx.x * kLatePiece; i0 < a.n; i0 += (uint64_t)gridDim.x * kLatePiece) {
    const uint32_t lim = (uint32_t)min(i0 + kLatePiece, a.n);
    uint32_t x = 0, y = a.nsb;  // the last super-bin that starts at or before i0
    while (y - x > 1) {
      const uint32_t m = (x + y) >> 1;
      if (__ldg(a.BS + m) <= (uint32_t)i0) x = m;
      else y = m;
    }
    for (uint32_t t0 = (uint32_t)i0; t0 < lim; ++x) {
      const uint32_t end = min(__ldg(a.BS + x + 1), lim);
      if (end <= t0) continue;  // (block-uniform) an empty super-bin
      if (threadIdx.x < 256) hist[threadIdx.x] = 0;
      __syncthreads();
      const K* const in = a.in_k + t0;
      const uint32_t len = end - t0;
      uint32_t j = threadIdx.x;
      for (; j + 7 * 512 < len; j += 8 * 512) {  // eight loads in flight
        K k[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) k[u] = __ldcs(in + j + u * 512);
#pragma unroll
        for (int u = 0; u < 8; ++u) atomicAdd(&hist[(map(k[u]) >> a.s) & dmask], 1u);
      }
      for (; j < len; j += 512) atomicAdd(&hist[(map(__ldcs(in + j)) >> a.s) & dmask], 1u);
      __syncthreads();
      if (threadIdx.x <= dmask && hist[threadIdx.x] != 0) atomicAdd(T + ((uint64_t)x << a.sshift) + threadIdx.x, hist[threadIdx.x]);
      __syncthreads();
      t0 = end;
    }
  }
}

// Phase 3: build every bin in shared memory.  Persistent CTAs take bins
// round-robin; bins above emax are skipped here.
template <typename K>
struct BinArgs {
  const K* in_k;
  const uint32_t* in_i;
  K* csr_k;
  uint32_t* csr_i;
  uint32_t* offsets;
  const uint32_t* T;
  const uint32_t* BS;
  uint64_t V;
  uint32_t nbins, s, emax;
  uint32_t list;      // bins one CTA may take (room in its bin list)
  uint32_t emin;      // bins of at most emin edges are another launch's; 0: no lower bound (empty
                      // bins are built too: their buckets' offsets must be written)
  uint32_t pos_base;  // added to every offset written (position of element 0 in the CSR arrays)
  bool has_pos;           // room for bin positions: the launch can rank by position
  const uint32_t* order;  // order mode word (null: partitions were stable); see k_partition
  const uint32_t* gate;   // null, or a count written by k_scan_bins: no bin for the launch when it is 0
  const uint32_t* ovf_list;   // launch of 1024-thread CTAs: bins for build_big_bins, and their number
  const uint32_t* ovf_count;  // (null: none)
};

// Streams edges [start, start + len) of a bin in tiles of kBigTile, sorts
// every tile stably by local bucket and appends each run at its bucket's
// cursor (cur: absolute CSR positions of the bin's nb buckets, advanced).
// Tiles follow input order and each is sorted stably, so every bucket keeps
// ascending input position.
template <typename K, typename Map, int NW>
__device__ __forceinline__ void stream_runs(const BinArgs<K>& a, const Map& map, uint32_t start, uint32_t len,
                                            uint64_t bucket0, uint32_t nb, uint32_t* cur, uint8_t* sp) {
  constexpr int IPT = kBigTile / (NW * 32);
  K* tk = (K*)sp; sp += (size_t)kBigTile * sizeof(K);
  uint32_t* ti = (uint32_t*)sp; sp += (size_t)kBigTile * 4;
  uint16_t* lb = (uint16_t*)sp; sp += kBigTile * 2;
  uint16_t* tmp = (uint16_t*)sp; sp += kBigTile * 2;
  uint16_t* perm = (uint16_t*)sp; sp += kBigTile * 2;
  uint16_t* slb = (uint16_t*)sp; sp += kBigTile * 2;
  sp = (uint8_t*)(((uintptr_t)sp + 15) & ~(uintptr_t)15);
  uint32_t* wc = (uint32_t*)sp; sp += rank_words<NW>() * 4;
  uint32_t* wsum = (uint32_t*)sp;
  for (uint32_t t0 = 0; t0 < len; t0 += kBigTile) {
    const uint32_t cnt = min((uint32_t)kBigTile, len - t0);
    for (uint32_t e = threadIdx.x; e < cnt; e += blockDim.x) {
      const K key = a.in_k[start + t0 + e];
      const uint32_t id = a.in_i[start + t0 + e];
      tk[e] = key;
      ti[e] = id;
      lb[e] = (uint16_t)(map(key, id) - (uint32_t)bucket0);
    }
    __syncthreads();
    const uint16_t* sorted = sort_positions_by_bucket<IPT, NW>(lb, cnt, nb, tmp, perm, wc, wsum);
    for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x) slb[j] = lb[sorted[j]];
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x) {
      const uint16_t l = slb[j];
      uint32_t lo = 0, hi = j;  // first index with slb == l
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (slb[mid] < l) lo = mid + 1; else hi = mid;
      }
      const uint32_t g = cur[l] + (j - lo);
      const uint32_t p = sorted[j];
      a.csr_k[g] = tk[p];
      a.csr_i[g] = map.out_id(ti[p]);
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x) {
      const uint16_t l = slb[j];
      if (j + 1 == cnt || slb[j + 1] != l) {
        uint32_t lo = 0, hi = j;
        while (lo < hi) {
          const uint32_t mid = (lo + hi) >> 1;
          if (slb[mid] < l) lo = mid + 1; else hi = mid;
        }
        cur[l] += j - lo + 1;
      }
    }
    __syncthreads();
  }
}

// Local-bucket counts of edges [start, start + len) of a bin into cur[]
// (zeroed first).  Equal buckets of a warp are merged by __match_any_sync,
// so a bucket holding most of the bin (duplicates) costs one shared-memory
// atomic per warp instead of one per edge.
template <typename K, typename Map>
__device__ __forceinline__ void count_local(const BinArgs<K>& a, const Map& map, uint32_t start, uint32_t len,
                                            uint64_t bucket0, uint32_t nb, uint32_t* cur) {
  for (uint32_t v = threadIdx.x; v < nb; v += blockDim.x) cur[v] = 0;
  __syncthreads();
  const uint32_t lane = lane_id();
  for (uint32_t base = threadIdx.x & ~31u; base < len; base += blockDim.x) {
    const uint32_t e = base + lane;
    const bool valid = e < len;
    const uint32_t l = valid ? map(a.in_k[start + e], a.in_i[start + e]) - (uint32_t)bucket0 : 0xffffffffu;
    const uint32_t peers = __match_any_sync(kFull, l);
    if (valid && lane == (uint32_t)(__ffs(peers) - 1)) atomicAdd(&cur[l], (uint32_t)__popc(peers));
  }
  __syncthreads();
}

// Bins too large for shared memory (duplicates, skew, tiny V) with at most
// kHugeSeg edges: one CTA per bin counts its local buckets, writes the bin's
// offsets and streams the bin (stream_runs).  Called by the bin build's launch
// of 1024-thread CTAs after its own bins.
template <typename K, typename Map>
__device__ __noinline__ void build_big_bins(BinArgs<K> a, uint32_t novf, Map map, uint8_t* smem) {
  const uint32_t nbmax = 1u << a.s;
  uint32_t* cur = (uint32_t*)smem;
  uint8_t* rest = smem + align_up((size_t)nbmax * 4, 16);
  uint32_t* wsum = (uint32_t*)(rest + big_rest_bytes(sizeof(K)) - 32 * 4);
  for (uint32_t k = blockIdx.x; k < novf; k += gridDim.x) {
    const uint32_t b = a.ovf_list[k];
    const uint32_t E = a.T[b], start = a.BS[b];
    const uint64_t bucket0 = (uint64_t)b << a.s;
    const uint32_t nb = (uint32_t)min((uint64_t)nbmax, a.V - bucket0);
    count_local(a, map, start, E, bucket0, nb, cur);
    block_excl_scan_smem(cur, (int)nb, wsum);
    for (uint32_t v = threadIdx.x; v < nb; v += blockDim.x) {
      a.offsets[bucket0 + v] = a.pos_base + start + cur[v];
      cur[v] += start;
    }
    __syncthreads();
    stream_runs<K, Map, kBinNW>(a, map, start, E, bucket0, nb, cur, rest);
  }
}

// Edges per thread of the bin build: a CTA of NT threads builds bins of up to
// NT * bin_ipt<K>() edges (9216 uint32 or 7168 uint64 edges with 512 threads).
template <typename K>
__host__ __device__ constexpr int bin_ipt() {
  return sizeof(K) == 8 ? 14 : 18;
}
constexpr uint32_t kBinInfo = 255;   // longest bucket whose length and arrival ranks fit one slot's 16 bits
constexpr uint32_t kBinBitmaps = 4;  // warps (and bitmaps) ranking longer buckets of stable partitions
constexpr int kBinUnroll = 6;        // comparisons of a bucket made without a loop

// Shared memory of k_binbuild: the bin's keys and ids in bucket order (and up
// to 3 entries before them), packed u16 bucket counters, the CTA's list of
// `list` bins, and two bytes per edge for the bucket list or the slot words;
// with pos also the bin positions, and the list and bitmaps of long buckets.
__host__ __device__ inline uint32_t bin_cnt_words(uint32_t s) {  // one more counter than buckets, whole 16-byte pieces
  return (uint32_t)((((size_t)1 << s) + 2) / 2 + 3) & ~3u;
}
__host__ __device__ inline uint32_t bin_map_words(uint32_t emax) { return (emax + 31) / 32; }
static size_t bin_smem_bytes(int kb, uint32_t emax, uint32_t s, uint32_t list, bool pos) {
  size_t b = (size_t)(emax + 4) * (kb + 4) + (size_t)emax * 2 + (size_t)bin_cnt_words(s) * 4 + 32 * 4 + 16 +
             2 * (size_t)list * 4;
  if (pos) b += (size_t)emax * 2 + kBinBitmaps * (size_t)bin_map_words(emax) * 6 + (emax / (kBinInfo + 1) + 1) * 2;
  return align_up(b, 16);
}

__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {  // whole 16-byte pieces inside [p, p + bytes)
  const uintptr_t a = ((uintptr_t)p + 15) & ~(uintptr_t)15, e = ((uintptr_t)p + bytes) & ~(uintptr_t)15;
  if (e > a)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((uint32_t)(e - a)) : "memory");
}

// Copies n elements from shared to global memory in 16-byte pieces: src is
// 16-byte aligned, element i lies at src[shift + i], and dst - shift is
// 16-byte aligned.
template <int NT, typename T>
__device__ __forceinline__ void copy_out(T* __restrict__ dst, const T* src, uint32_t shift, uint32_t n) {
  constexpr uint32_t P = 16 / sizeof(T);
  const uint32_t pieces = (shift + n + P - 1) / P;
  for (uint32_t v = threadIdx.x; v < pieces; v += NT) {
    const uint32_t i = v * P;
    if (i >= shift && i + P <= shift + n) {
      *reinterpret_cast<uint4*>(dst + (i - shift)) = *reinterpret_cast<const uint4*>(src + i);
    } else {
      for (uint32_t k = i; k < i + P; ++k)
        if (k >= shift && k < shift + n) dst[k - shift] = src[k];
    }
  }
}

// Per bin (E <= emax edges, nb local buckets):
//   1. local bucket of every edge; a shared-memory atomic on the bucket's
//      counter (two 16-bit counters per word) counts it and gives the edge
//      its arrival rank in the bucket; (bucket, rank) stays in a register
//   2. exclusive scan of the counts -> bucket starts, packed the same way,
//      and a list of the buckets of two or more edges
//   3. every edge goes to slot (bucket start + arrival rank) in shared
//      memory; the bin's offsets are written, coalesced
//   4. the buckets are put in canonical order, ascending id (order mode 0:
//      the ids are input positions, distinct) or bin position (stable
//      partitions: bin positions follow the input), and written out
// Step 4, where the order is by id and few buckets are long (the usual case
// at load 1): one thread sorts a bucket of up to 4 edges in registers, one
// warp a bucket of up to 32 edges, in place in shared memory; then keys and
// ids leave as straight 16-byte copies.  Else ("dense"): every slot gets a
// 16-bit word of its bucket's length and its own arrival rank in step 3, and
// the edge of each slot goes straight to its place, the number of its
// bucket's edges with a smaller id or position; neighbouring slots hold
// neighbouring buckets, so these reads and the stores are coalesced.
// Buckets above kBinInfo edges find their range through the map again; with
// stable partitions they get their places from a bitmap of their positions
// (a prefix count) instead of comparisons.
// A bin takes this kernel when E <= emax and, for emin > 0, E > emin: one
// launch (emin = 0) covers every bin of the expected size, empty ones
// included, a second one with the largest CTAs the larger ones up to its own
// emax, and every bin when the order mode asks for positions the first
// launch has no room for.
//
// Bound by instruction issue and shared-memory accesses, not HBM: keys are
// loaded twice and ids once, in whole warps, straight to registers, from L2
// (the next bin is prefetched there).  Several CTAs per SM (1024 threads in
// all) overlap one bin's loads and barriers with another's work.  Measured
// with uint32 keys at load 1, against one 1024-thread CTA per SM that staged
// bins by TMA, claimed slots in a second round of atomics and gathered every
// edge through a slot list: 1.61 against 2.38 ms at 2^28 keys (bins of 8192),
// 0.76 against 1.51 ms at 2^27 (bins of 4096).  ncu at 2^26: 126 instructions
// per 32 edges (issue active 53%) and shared-memory wavefronts 69% of peak.
template <typename K, typename Map, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_binbuild(BinArgs<K> a, Map map) {
  constexpr int IPT = bin_ipt<K>();
  constexpr int G = sizeof(K) == 8 ? 7 : 6;  // edges per thread taken together
  static_assert(IPT % G == 0, "whole groups");
  const bool pos = a.order == nullptr || *(volatile const uint32_t*)a.order != 0u;
  if (pos && !a.has_pos) return;
  uint32_t emin = a.emin;
  bool idle = false;  // no bin for this launch
  if (emin != 0) {  // second launch
    if (pos && a.order != nullptr) emin = 0;  // the first launch took no bin
    else idle = *(volatile const uint32_t*)a.gate == 0u;
  }
  const uint32_t novf = NT == kBinNW * 32 && a.ovf_count != nullptr ? *(volatile const uint32_t*)a.ovf_count : 0u;
  if (idle && novf == 0) return;
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sp = smem;
  K* const ks0 = (K*)sp; sp += (size_t)(a.emax + 4) * sizeof(K);
  uint32_t* const is0 = (uint32_t*)sp; sp += (size_t)(a.emax + 4) * 4;
  uint32_t* const cnt = (uint32_t*)sp; sp += (size_t)bin_cnt_words(a.s) * 4;
  const uint16_t* const cnt16 = (const uint16_t*)cnt;
  uint32_t* const wsum = (uint32_t*)sp; sp += 32 * 4;
  uint32_t* const nlong = (uint32_t*)sp; sp += 16;  // [0] buckets of 5 .. 32 edges + 2^16 * longer; [1] buckets above kBinInfo
  uint32_t* const bl_start = (uint32_t*)sp; sp += (size_t)a.list * 4;  // this CTA's bins: start, size
  uint32_t* const bl_size = (uint32_t*)sp; sp += (size_t)a.list * 4;
  uint32_t* const multi = (uint32_t*)sp;  // buckets of 2 or more edges: start | length << 16 (at most emax / 2)
  uint16_t* const info = (uint16_t*)sp; sp += (size_t)a.emax * 2;  // dense: length | arrival rank << 8; 0: longer
  // used only with pos (sizes: whole words)
  uint16_t* const ps = (uint16_t*)sp; sp += (size_t)a.emax * 2;
  const uint32_t map_words = bin_map_words(a.emax);
  uint32_t* const hbits = (uint32_t*)sp; sp += kBinBitmaps * (size_t)map_words * 4;
  uint16_t* const hpre = (uint16_t*)sp; sp += kBinBitmaps * (size_t)map_words * 2;
  uint16_t* const heavy = (uint16_t*)sp;

  map.init();
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  // Bins blockIdx.x, +gridDim.x, ...: starts and sizes gathered once, so the
  // loop below needs no global loads to find its next bin.
  const uint32_t nmine =
      !idle && blockIdx.x < a.nbins ? (a.nbins - blockIdx.x + gridDim.x - 1) / gridDim.x : 0u;
  for (uint32_t j = tid; j < nmine; j += NT) {
    const uint32_t bb = blockIdx.x + j * gridDim.x;
    bl_start[j] = a.BS[bb];
    bl_size[j] = a.T[bb];
  }
  const uint32_t cnt_words = bin_cnt_words(a.s);
  for (uint32_t w = tid; w < cnt_words; w += NT) cnt[w] = 0;
  if (tid < 2) nlong[tid] = 0;
  __syncthreads();
  auto skip = [&](uint32_t j) {  // the CTA's first bin from its j-th on that this launch takes
    while (j < nmine && (bl_size[j] > a.emax || (emin != 0 && bl_size[j] <= emin))) ++j;
    return j;
  };
  uint32_t jb = skip(0);
  while (jb < nmine) {
    const uint32_t E = bl_size[jb], start = bl_start[jb];
    const uint64_t bucket0 = (uint64_t)(blockIdx.x + jb * gridDim.x) << a.s;
    const uint32_t nb = (uint32_t)min((uint64_t)1 << a.s, a.V - bucket0);
    jb = skip(jb + 1);
    if (tid == 0 && jb < nmine) {
      prefetch_l2(a.in_k + bl_start[jb], bl_size[jb] * (uint32_t)sizeof(K));
      prefetch_l2(a.in_i + bl_start[jb], bl_size[jb] * 4u);
    }
    // edge tid + c * NT of the bin is this thread's when left > c * NT
    const int left = (int)E - (int)tid;
    const K* const gk = a.in_k + start + tid;
    const uint32_t* const gi = a.in_i + start + tid;
    K key[G];
    uint32_t id[G];
    auto load_keys = [&](int g) {  // of the edges g .. g + G - 1
#pragma unroll
      for (int u = 0; u < G; ++u) key[u] = left > (g + u) * NT ? __ldg(gk + (g + u) * NT) : K(0);
    };
    auto load_ids = [&](int g) {
#pragma unroll
      for (int u = 0; u < G; ++u) id[u] = left > (g + u) * NT ? __ldg(gi + (g + u) * NT) : 0u;
    };
    // a group of edges through f(c, u): whole groups without a test per edge
    auto group = [&](int g, auto&& f) {
      if ((uint32_t)(g + G) * NT <= E) {  // block-uniform
#pragma unroll
        for (int u = 0; u < G; ++u) f(g + u, u);
      } else {
#pragma unroll
        for (int u = 0; u < G; ++u)
          if (left > (g + u) * NT) f(g + u, u);
      }
    };
    // 1. local buckets, counts, arrival ranks
    uint32_t br[IPT];  // bucket | rank << 16
#pragma unroll
    for (int g = 0; g < IPT; g += G) {
      if ((uint32_t)g * NT >= E) break;  // block-uniform
      load_keys(g);
      if (Map::kNeedsPos) load_ids(g);
      group(g, [&](int c, int u) {
        const uint32_t l = map(key[u], Map::kNeedsPos ? id[u] : 0u) - (uint32_t)bucket0;
        const uint32_t odd = l & 1u;
        const uint32_t old = atomicAdd(&cnt[l >> 1], 1u + odd * 0xffffu);
        br[c] = __byte_perm(l, old, 0x5410u + odd * 0x2200u);  // the bucket's half of old above l
      });
    }
    load_keys(0);  // for step 3: these arrive during the scan
    load_ids(0);
    __syncthreads();
    // 2. exclusive scan of the counts (a thread's counts sum to at most E < 2^15)
    uint32_t nmulti;
    {
      const uint32_t words = (nb + 2) >> 1;  // the counter after the last bucket's receives E
      const uint32_t per = ((words + NT - 1) / NT + 3u) & ~3u;  // words per thread, whole 16-byte pieces
      const uint32_t w0 = min(tid * per, cnt_words), w1 = min(w0 + per, cnt_words);
      // of the two counters of a word: flags of those of at least m edges
      auto at_least = [](uint32_t x, uint32_t m) { return (x + (0x8000u - m) * 0x10001u) & 0x80008000u; };
      uint32_t sum = 0, two = 0, five = 0, big = 0;
      for (uint32_t w = w0; w < w1; w += 4) {
        const uint4 x = *reinterpret_cast<const uint4*>(cnt + w);
        sum += x.x + x.y + x.z + x.w;  // both halves at once
        two += __popc(at_least(x.x, 2) | (at_least(x.y, 2) >> 1) | (at_least(x.z, 2) >> 2) | (at_least(x.w, 2) >> 3));
        five += __popc(at_least(x.x, 5) | (at_least(x.y, 5) >> 1) | (at_least(x.z, 5) >> 2) | (at_least(x.w, 5) >> 3));
        big |= at_least(x.x, 33) | at_least(x.y, 33) | at_least(x.z, 33) | at_least(x.w, 33);
      }
      if (five) atomicAdd(nlong, big ? 0x10000u : five);
      const uint32_t v = ((sum & 0xffffu) + (sum >> 16)) | (two << 16);
      uint32_t base = block_excl_scan_nt<uint32_t>(v, wsum), at = base >> 16;
      nmulti = wsum[NT / 32 - 1] >> 16;
      base &= 0xffffu;
      for (uint32_t w = w0; w < w1; w += 4) {
        uint4 x = *reinterpret_cast<const uint4*>(cnt + w);
        auto word = [&](uint32_t c) {
          const uint32_t lo = c & 0xffffu, hi = c >> 16, mid = base + lo;
          const uint32_t out = __byte_perm(base, mid, 0x5410u);
          if (lo > 1) multi[at++] = base | (lo << 16);
          if (hi > 1) multi[at++] = mid | (c & 0xffff0000u);
          base = mid + hi;
          return out;
        };
        x.x = word(x.x);
        x.y = word(x.y);
        x.z = word(x.z);
        x.w = word(x.w);
        *reinterpret_cast<uint4*>(cnt + w) = x;
      }
    }
    __syncthreads();
    // block-uniform: too many or too long buckets for sorting them one by one
    const bool dense = pos || *nlong > E / 64;
    K* const ok = a.csr_k + start;
    uint32_t* const oi = a.csr_i + start;
    const uint32_t shk = dense ? 0u : (uint32_t)((uintptr_t)ok & 15u) / (uint32_t)sizeof(K);
    const uint32_t shi = dense ? 0u : (uint32_t)((uintptr_t)oi & 15u) / 4u;
    K* const ks = ks0 + shk;
    uint32_t* const is = is0 + shi;
    // 3. edges to their slots; offsets
#pragma unroll
    for (int g = 0; g < IPT; g += G) {
      if ((uint32_t)g * NT >= E) break;
      if (g > 0) {
        load_keys(g);
        load_ids(g);
      }
      if (!dense) {
        group(g, [&](int c, int u) {
          const uint32_t slot = cnt16[br[c] & 0xffffu] + (br[c] >> 16);
          ks[slot] = key[u];
          is[slot] = map.out_id(id[u]);
        });
      } else {
        group(g, [&](int c, int u) {
          const uint32_t l = br[c] & 0xffffu, r = br[c] >> 16;
          const uint32_t beg = cnt16[l], n = cnt16[l + 1] - beg;
          const uint32_t slot = beg + r;
          ks[slot] = key[u];
          is[slot] = id[u];
          info[slot] = (uint16_t)(n <= kBinInfo ? n | (r << 8) : 0u);
          if (pos) {
            ps[slot] = (uint16_t)(tid + c * NT);
            if (r == kBinInfo) heavy[atomicAdd(nlong + 1, 1u)] = (uint16_t)l;  // one edge of every longer bucket
          }
        });
      }
    }
    {
      uint32_t* const off = a.offsets + bucket0;
      const uint32_t o = a.pos_base + start;
      if (((uintptr_t)off & 7) == 0) {  // two buckets per store
        for (uint32_t w = tid; w < nb >> 1; w += NT) {
          const uint32_t x = cnt[w];
          *reinterpret_cast<uint2*>(off + 2 * w) = make_uint2(o + (x & 0xffffu), o + (x >> 16));
        }
        if ((nb & 1u) && tid == 0) off[nb - 1] = o + cnt16[nb - 1];
      } else {
        for (uint32_t v = tid; v < nb; v += NT) off[v] = o + cnt16[v];
      }
    }
    __syncthreads();
    auto clear = [&]() {
      for (uint32_t w = tid * 4; w < cnt_words; w += NT * 4)
        *reinterpret_cast<uint4*>(cnt + w) = make_uint4(0, 0, 0, 0);
      if (tid < 2) nlong[tid] = 0;
    };
    if (!dense) {
      // 4. buckets of 2 .. 4 edges by one thread each: (id, slot) pairs
      //    through a sorting network, then the keys by slot; longer ones by
      //    the warp, which ranks every lane's id against the others'
      clear();
      for (uint32_t t0 = warp * 32u; t0 < nmulti; t0 += NT) {
        const uint32_t x = t0 + lane < nmulti ? multi[t0 + lane] : 0u;
        const uint32_t beg = x & 0xffffu, n = x >> 16;
        if (n >= 2 && n <= 4) {
          uint32_t d[4], p[4];
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i) {
            d[i] = i < n ? is[beg + i] : 0xffffffffu;  // no edge has this id
            p[i] = i;
          }
          auto order = [&](int i, int j) {
            const bool sw = d[i] > d[j];
            const uint32_t di = d[i], pi = p[i];
            d[i] = sw ? d[j] : di;
            p[i] = sw ? p[j] : pi;
            d[j] = sw ? di : d[j];
            p[j] = sw ? pi : p[j];
          };
          order(0, 1);
          if (n > 2) {
            order(2, 3);
            order(0, 2);
            order(1, 3);
            order(1, 2);
          }
          K k[4];
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i)
            if (i < n) k[i] = ks[beg + p[i]];
#pragma unroll
          for (uint32_t i = 0; i < 4; ++i)
            if (i < n) {
              is[beg + i] = d[i];
              ks[beg + i] = k[i];
            }
        }
        for (uint32_t m = __ballot_sync(kFull, n > 4); m; m &= m - 1) {
          const uint32_t y = __shfl_sync(kFull, x, __ffs(m) - 1);
          const uint32_t b = y & 0xffffu, len = y >> 16;  // len <= 32
          const bool in = lane < len;
          const uint32_t cid = in ? is[b + lane] : 0u;
          const K k = in ? ks[b + lane] : K(0);
          uint32_t r = 0;
          for (uint32_t i = 0; i < len; ++i) r += __shfl_sync(kFull, cid, i) < cid;
          __syncwarp();
          if (in) {
            is[b + r] = cid;
            ks[b + r] = k;
          }
        }
      }
      __syncthreads();
      copy_out<NT>(ok, ks0, shk, E);
      copy_out<NT>(oi, is0, shi, E);
      __syncthreads();
      continue;
    }
    const uint32_t nh = nlong[1];
    // long buckets of stable partitions: the edge's place in its bucket
    // replaces its bin position
    if (nh > 0) {  // block-uniform
      const uint32_t words = (E + 31) >> 5;
      if (warp < kBinBitmaps) {
        uint32_t* const bm = hbits + warp * map_words;
        uint16_t* const pre = hpre + warp * map_words;
        for (uint32_t h = warp; h < nh; h += kBinBitmaps) {
          const uint32_t beg = cnt16[heavy[h]], end = cnt16[heavy[h] + 1];
          for (uint32_t k = lane; k < words; k += 32) bm[k] = 0;
          __syncwarp();
          for (uint32_t i = beg + lane; i < end; i += 32) atomicOr(&bm[ps[i] >> 5], 1u << (ps[i] & 31u));
          __syncwarp();
          uint32_t run = 0;
          for (uint32_t k0 = 0; k0 < words; k0 += 32) {
            const uint32_t c = k0 + lane < words ? __popc(bm[k0 + lane]) : 0u;
            const uint32_t incl = warp_incl_scan(c);
            if (k0 + lane < words) pre[k0 + lane] = (uint16_t)(run + incl - c);
            run += __shfl_sync(kFull, incl, 31);
          }
          __syncwarp();
          for (uint32_t i = beg + lane; i < end; i += 32) {
            const uint32_t p = ps[i];
            ps[i] = (uint16_t)(pre[p >> 5] + __popc(bm[p >> 5] & ((1u << (p & 31u)) - 1u)));
          }
          __syncwarp();
        }
      }
      __syncthreads();
    }
    // 4. dense: every slot's edge straight to its place
    for (uint32_t j = tid; j < E; j += NT) {
      const K k = ks[j];
      const uint32_t cid = is[j], x = info[j];
      uint32_t dst;
      if (x != 0) {  // bucket of 1 .. kBinInfo edges
        const uint32_t n = x & 0xffu;
        dst = j - (x >> 8);
        if (!pos) {
          const uint32_t* const q = is + dst;
#pragma unroll
          for (int i = 0; i < kBinUnroll; ++i)
            if ((uint32_t)i < n && q[i] < cid) ++dst;
          if (n > kBinUnroll)
            for (uint32_t i = kBinUnroll; i < n; ++i) dst += q[i] < cid;
        } else {
          const uint32_t p = ps[j];
          const uint16_t* const q = ps + dst;
#pragma unroll
          for (int i = 0; i < kBinUnroll; ++i)
            if ((uint32_t)i < n && q[i] < p) ++dst;
          if (n > kBinUnroll)
            for (uint32_t i = kBinUnroll; i < n; ++i) dst += q[i] < p;
        }
      } else {
        const uint32_t l = map(k, cid) - (uint32_t)bucket0;
        const uint32_t end = cnt16[l + 1];
        uint32_t i = cnt16[l];
        dst = i;
        if (pos) {
          dst += ps[j];
        } else {  // four ids per load
          for (; i & 3u; ++i) dst += is[i] < cid;
          for (; i + 4 <= end; i += 4) {
            const uint4 y = *reinterpret_cast<const uint4*>(is + i);
            dst += (y.x < cid) + (y.y < cid) + (y.z < cid) + (y.w < cid);
          }
          for (; i < end; ++i) dst += is[i] < cid;
        }
      }
      ok[dst] = k;
      oi[dst] = map.out_id(cid);
    }
    __syncthreads();
    clear();
    __syncthreads();
  }
  if (NT == kBinNW * 32 && novf != 0) {
    __syncthreads();
    build_big_bins<K, Map>(a, novf, map, smem);
  }
}

// Bin-build launch configuration.
struct BinCfg {
  uint32_t nt, grid, list, emax;
  bool pos;
  size_t smem;
};
// The launch with CTAs of nt threads, as many to an SM as make 1024 threads:
// the largest bin they can hold, at most nt * ipt edges.
template <typename K>
static BinCfg bin_config_for(const Plan& p, uint32_t nt, bool pos) {
  const DevInfo& di = dev_info();
  BinCfg c{};
  c.nt = nt;
  c.pos = pos;
  const uint32_t per_sm = 1024 / nt;
  c.grid = std::max<uint32_t>(std::min<uint32_t>(p.nbins, (uint32_t)di.sms * per_sm),
                              (p.nbins + kMaxBinsPerCta - 1) / kMaxBinsPerCta);
  c.list = (p.nbins + c.grid - 1) / c.grid;
  const size_t cap =
      per_sm == 1 ? (size_t)di.max_smem_optin : (size_t)di.smem_per_sm / per_sm - (size_t)di.smem_reserved;
  uint32_t e = nt * bin_ipt<K>();
  while (e > 32 && bin_smem_bytes(p.kb, e, p.s, c.list, pos) > cap) e -= 32;
  c.emax = e;
  c.smem = bin_smem_bytes(p.kb, e, p.s, c.list, pos);
  return c;
}
// CTAs of 256, 512 or 1024 threads, by the size bins are expected to have
// (Poisson: mean and five standard deviations): the smaller the CTA, the
// better its barriers are hidden by the other CTAs of the SM (uint32 keys at
// load 1, 256 / 512 / 1024 threads: 0.202 / 0.244 / 0.312 ms at 2^25 keys,
// 512 / 1024: 1.61 / 2.03 ms at 2^28).  Builds of at most two bins per SM
// take the largest, which finish a bin soonest (256 bins at 2^20 keys: 18.9
// us against 22.1 with 256 threads; 512 bins at 2^21: 30.4 against 27.5).  A
// size asked for by the caller stands.
template <typename K>
static BinCfg bin_config(const Plan& p, bool by_id) {
  if (p.tpb == 1024) return bin_config_for<K>(p, 1024, true);
  if (p.tpb == 512) return bin_config_for<K>(p, 512, !by_id);
  const double mean = (double)p.n * (double)(1ull << p.s) / (double)p.V;
  const double need = mean + 5.0 * std::sqrt(mean) + 16.0;
  if (p.nbins > 2 * (uint32_t)dev_info().sms) {
    for (uint32_t nt : {256u, 512u}) {
      const BinCfg c = bin_config_for<K>(p, nt, !by_id);
      if ((double)c.emax >= need) return c;
    }
  }
  return bin_config_for<K>(p, 1024, true);
}

// The two launches: bins up to first->emax, and larger ones up to
// second->emax (no such launch where both have 1024 threads).
template <typename K>
static void bin_configs(const Plan& p, bool by_id, BinCfg* first, BinCfg* second) {
  *first = bin_config<K>(p, by_id);
  *second = bin_config_for<K>(p, 1024, true);
  first->emax = std::min(first->emax, second->emax);
}

// Bins above kHugeSeg edges, split into segments of kHugeSeg edges (rows).
// 1. every row's local-bucket counts, one CTA per row
template <typename K, typename Map>
__global__ void __launch_bounds__(kBinNW * 32, 1) k_huge_count(BinArgs<K> a, const uint32_t* __restrict__ rows,
                                                             const uint32_t* __restrict__ rowdesc,
                                                             uint32_t* __restrict__ rowcnt, Map map) {
  extern __shared__ __align__(16) uint32_t hcur[];
  map.init();
  const uint32_t nbmax = 1u << a.s;
  const uint32_t R = *rows;
  for (uint32_t r = blockIdx.x; r < R; r += gridDim.x) {
    const uint32_t b = rowdesc[2 * r], sg = rowdesc[2 * r + 1];
    const uint32_t off = sg * kHugeSeg;
    const uint32_t len = min(kHugeSeg, a.T[b] - off);
    const uint64_t bucket0 = (uint64_t)b << a.s;
    const uint32_t nb = (uint32_t)min((uint64_t)nbmax, a.V - bucket0);
    count_local(a, map, a.BS[b] + off, len, bucket0, nb, hcur);
    for (uint32_t v = threadIdx.x; v < nb; v += blockDim.x) rowcnt[(uint64_t)r * nbmax + v] = hcur[v];
    __syncthreads();
  }
}

// 2. per huge bin: bucket totals over its rows, exclusive scan -> the bin's
//    offsets; every row's counts become its absolute CSR cursors
template <typename K>
__global__ void __launch_bounds__(1024) k_huge_scan(BinArgs<K> a, const uint32_t* __restrict__ hcount,
                                                    const uint32_t* __restrict__ hlist, uint32_t* __restrict__ rowcnt) {
  extern __shared__ __align__(16) uint32_t tot[];
  __shared__ uint32_t wsum[32];
  const uint32_t nbmax = 1u << a.s;
  const uint32_t H = *hcount;
  for (uint32_t k = blockIdx.x; k < H; k += gridDim.x) {
    const uint32_t b = hlist[3 * k], r0 = hlist[3 * k + 1], nr = hlist[3 * k + 2];
    const uint64_t bucket0 = (uint64_t)b << a.s;
    const uint32_t nb = (uint32_t)min((uint64_t)nbmax, a.V - bucket0);
    const uint32_t start = a.BS[b];
    for (uint32_t v = threadIdx.x; v < nb; v += blockDim.x) {
      uint32_t run = 0;
      for (uint32_t r = 0; r < nr; ++r) {
        uint32_t* p = rowcnt + (uint64_t)(r0 + r) * nbmax + v;
        const uint32_t c = *p;
        *p = run;
        run += c;
      }
      tot[v] = run;
    }
    __syncthreads();
    block_excl_scan_smem(tot, (int)nb, wsum);
    for (uint32_t v = threadIdx.x; v < nb; v += blockDim.x) {
      const uint32_t first = start + tot[v];
      a.offsets[bucket0 + v] = a.pos_base + first;
      for (uint32_t r = 0; r < nr; ++r) rowcnt[(uint64_t)(r0 + r) * nbmax + v] += first;
    }
    __syncthreads();
  }
}

// 3. every row streams its segment to its cursors, one CTA per row
template <typename K, typename Map>
__global__ void __launch_bounds__(kBinNW * 32, 1) k_huge_scatter(BinArgs<K> a, const uint32_t* __restrict__ rows,
                                                               const uint32_t* __restrict__ rowdesc,
                                                               const uint32_t* __restrict__ rowcnt, Map map) {
  extern __shared__ __align__(16) uint8_t smem[];
  map.init();
  const uint32_t nbmax = 1u << a.s;
  uint32_t* cur = (uint32_t*)smem;
  uint8_t* rest = smem + align_up((size_t)nbmax * 4, 16);
  const uint32_t R = *rows;
  for (uint32_t r = blockIdx.x; r < R; r += gridDim.x) {
    const uint32_t b = rowdesc[2 * r], sg = rowdesc[2 * r + 1];
    const uint32_t off = sg * kHugeSeg;
    const uint32_t len = min(kHugeSeg, a.T[b] - off);
    const uint64_t bucket0 = (uint64_t)b << a.s;
    const uint32_t nb = (uint32_t)min((uint64_t)nbmax, a.V - bucket0);
    for (uint32_t v = threadIdx.x; v < nb; v += blockDim.x) cur[v] = rowcnt[(uint64_t)r * nbmax + v];
    __syncthreads();
    stream_runs<K, Map, kBinNW>(a, map, a.BS[b] + off, len, bucket0, nb, cur, rest);
  }
}

// ===========================================================================
// V1 (Alg. 1): global histogram with atomics, prefix sum, atomic scatter.
// Atomics leave the order inside a bucket arbitrary; a fix-up then sorts
// every bucket by input position (the ids hold positions until the end).
// ===========================================================================
template <typename K, typename Map>
__global__ void k_v1_count(const K* __restrict__ keys, uint64_t n, uint32_t* __restrict__ counts, Map map) {
  map.init();
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    atomicAdd(&counts[map(keys[i])], 1u);
}

template <typename K, typename Map>
__global__ void k_v1_scatter(const K* __restrict__ keys, uint64_t n, const uint32_t* __restrict__ offsets,
                             uint32_t* __restrict__ cursor, K* __restrict__ csr_k,
                             uint32_t* __restrict__ csr_i, Map map) {
  map.init();
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const K key = keys[i];
    const uint32_t b = map(key);
    const uint32_t pos = offsets[b] + atomicAdd(&cursor[b], 1u);
    csr_k[pos] = key;
    csr_i[pos] = (uint32_t)i;
  }
}

// Buckets of up to kV1Small edges: insertion sort by position, one thread per
// bucket.  Longer buckets go to a list for k_v1_fix_heavy.
template <typename K>
__global__ void k_v1_fix_small(const uint32_t* __restrict__ offsets, uint64_t V, K* csr_k, uint32_t* csr_i,
                               uint32_t* heavy_list, uint32_t* heavy_count) {
  for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t s = offsets[v], e = offsets[v + 1];
    const uint32_t c = e - s;
    if (c <= 1) continue;
    if (c > kV1Small) {
      heavy_list[atomicAdd(heavy_count, 1u)] = (uint32_t)v;
      continue;
    }
    for (uint32_t i = s + 1; i < e; ++i) {
      const uint32_t p = csr_i[i];
      const K k = csr_k[i];
      uint32_t j = i;
      while (j > s && csr_i[j - 1] > p) {
        csr_i[j] = csr_i[j - 1];
        csr_k[j] = csr_k[j - 1];
        --j;
      }
      csr_i[j] = p;
      csr_k[j] = k;
    }
  }
}

// Heavy buckets: one CTA per bucket, least-significant-digit radix sort of
// the (position, key) pairs by position, 8 bits per pass.  Segments that fit
// shared memory are sorted in place there; longer ones stream through a
// global temporary, one stable tile partition at a time.
template <typename K>
__global__ void __launch_bounds__(kV1HeavyNW * 32) k_v1_fix_heavy(const uint32_t* __restrict__ offsets,
                                                                 const uint32_t* heavy_list,
                                                                 const uint32_t* heavy_count, K* csr_k,
                                                                 uint32_t* csr_i, K* tmp_k, uint32_t* tmp_i,
                                                                 uint32_t nbits) {
  constexpr int NW = kV1HeavyNW, IPT = kV1HeavyIPT;
  constexpr uint32_t TILE = NW * 32 * IPT;
  extern __shared__ __align__(16) uint8_t smem[];
  uint8_t* sp = smem;
  K* sk = (K*)sp; sp += TILE * sizeof(K);
  uint32_t* sv = (uint32_t*)sp; sp += TILE * 4;
  uint32_t* wc = (uint32_t*)sp; sp += rank_words<NW>() * 4;
  uint32_t* dstart = (uint32_t*)sp; sp += 256 * 4;
  uint32_t* cursor = (uint32_t*)sp; sp += 256 * 4;
  uint8_t* sd = sp; sp += TILE;
  sp = (uint8_t*)(((uintptr_t)sp + 15) & ~(uintptr_t)15);
  uint32_t* wsum = (uint32_t*)sp;
  const uint32_t seg0 = (threadIdx.x >> 5) * (32u * IPT), lane = lane_id();
  const uint32_t nh = *heavy_count;
  for (uint32_t h = blockIdx.x; h < nh; h += gridDim.x) {
    const uint32_t v = heavy_list[h];
    const uint32_t s = offsets[v], c = offsets[v + 1] - s;
    K* src_k = csr_k + s;
    uint32_t* src_i = csr_i + s;
    K* dst_k = tmp_k + s;
    uint32_t* dst_i = tmp_i + s;
    for (uint32_t shift = 0; shift < nbits; shift += 8) {
      // count digits of this pass
      for (int d = threadIdx.x; d < 256; d += blockDim.x) cursor[d] = 0;
      __syncthreads();
      for (uint32_t e = threadIdx.x; e < c; e += blockDim.x) atomicAdd(&cursor[(src_i[e] >> shift) & 255u], 1u);
      __syncthreads();
      block_excl_scan_smem(cursor, 256, wsum);
      for (uint32_t t0 = 0; t0 < c; t0 += TILE) {
        const uint32_t cnt = min(TILE, c - t0);
        K key[IPT];
        uint32_t val[IPT], dig[IPT];
#pragma unroll
        for (int r = 0; r < IPT; ++r) {
          const uint32_t idx = seg0 + (uint32_t)r * 32u + lane;
          if (idx < cnt) {
            key[r] = src_k[t0 + idx];
            val[r] = src_i[t0 + idx];
            dig[r] = (val[r] >> shift) & 255u;
          } else {
            key[r] = 0; val[r] = 0; dig[r] = 0;
          }
        }
        tile_partition_out<K, IPT, NW>(key, val, dig, cnt, 256, sk, sv, sd, wc, dstart, cursor, wsum,
                                       dst_k, dst_i);
      }
      K* tk = src_k; src_k = dst_k; dst_k = tk;
      uint32_t* tv = src_i; src_i = dst_i; dst_i = tv;
    }
    if (src_k != csr_k + s) {  // odd number of passes: copy back
      for (uint32_t e = threadIdx.x; e < c; e += blockDim.x) {
        csr_k[s + e] = src_k[e];
        csr_i[s + e] = src_i[e];
      }
    }
    __syncthreads();
  }
}

__global__ void k_v1_ids(uint32_t* __restrict__ csr_i, const uint32_t* __restrict__ ids, uint64_t n) {
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x)
    csr_i[j] = ids[csr_i[j]];
}

// ===========================================================================
// Host drivers
// ===========================================================================
// The largest dynamic shared memory each kernel was asked for, per device.
static std::mutex g_smem_mu;
static std::unordered_map<const void*, size_t> g_smem_max[64];

template <typename F>
static void set_smem_once(F* kernel, size_t bytes) {
  // The attribute belongs to the kernel, process-wide, and a launch needs it
  // at least as large as its own request.  It is raised to the largest
  // request so far and never lowered, so a call on another host thread that
  // asked for more is not cut short; it is set on every call (cheap), so it
  // holds again after a device reset.
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  std::lock_guard<std::mutex> lk(g_smem_mu);
  size_t& top = g_smem_max[dev][(const void*)kernel];
  if (bytes > top) top = bytes;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)top);
}

// Launches k_partition_any with the tile of geometry T; the map's tables are
// staged only where T::MINB CTAs still fit an SM.
template <typename K, typename Map, bool PASS_B, bool IDS, typename T, int DIG = 256>
static void partition_any_launch(PartArgs<K> a, Map map, unsigned grid, cudaStream_t st) {
  const DevInfo& di = dev_info();
  const size_t own = part_any_smem(sizeof(K), IDS, T::NT * T::IPT, DIG);
  a.stage_bytes = own + Map::kStageBytes + di.smem_reserved <= (size_t)di.smem_per_sm / T::MINB ? (uint32_t)Map::kStageBytes : 0u;
  auto kern = k_partition_any<K, Map, PASS_B, IDS, DIG, T::NT, T::IPT, T::MINB>;
  set_smem_once(kern, own + a.stage_bytes);
  kern<<<grid, T::NT, own + a.stage_bytes, st>>>(a, map);
}

// Pass B in any order: four pieces or more per resident CTA, of at most
// kPartPiece tiles.
template <typename K, typename Map>
static void partition_b_any(PartArgs<K> a, Map map, cudaStream_t st) {
  constexpr uint64_t tile = (uint64_t)PartB<K>::NT * PartB<K>::IPT;
  const uint64_t resident = (uint64_t)PartB<K>::MINB * dev_info().sms, tiles = (a.n + tile - 1) / tile;
  a.piece = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(kPartPiece, tiles / (4 * resident)));
  const uint64_t pieces = (tiles + a.piece - 1) / a.piece;
  partition_any_launch<K, Map, true, true, PartB<K>>(a, map, (unsigned)std::min(pieces, resident), st);
}

// One bin-build launch (k_binbuild): bins of more than emin edges (0: all) up
// to the configuration's largest.
template <typename K, typename Map>
static void binbuild_launch(BinArgs<K> a, Map map, const BinCfg& c, uint32_t emin, const uint32_t* gate,
                            cudaStream_t st) {
  a.emax = c.emax;
  a.list = c.list;
  a.has_pos = c.pos;
  a.emin = emin;
  a.gate = gate;
  auto go = [&](auto kern) {
    set_smem_once(kern, c.smem);
    kern<<<c.grid, c.nt, c.smem, st>>>(a, map);
  };
  if (c.nt == 256) go(k_binbuild<K, Map, 256>);
  else if (c.nt == 512) go(k_binbuild<K, Map, 512>);
  else go(k_binbuild<K, Map, 1024>);
}

template <typename K, typename Map>
hg_status build_v2(const Plan& p, const K* keys, const uint32_t* ids, uint32_t* offsets, K* csr_k,
                   uint32_t* csr_i, uint8_t* ws, cudaStream_t st, Map map, uint32_t pos_base,
                   bool positional_ids) {
  WsHeader* hdr = (WsHeader*)ws;
  uint32_t* status = &hdr->status;
  uint32_t* H = (uint32_t*)(ws + p.o_H);
  uint32_t* C = (uint32_t*)(ws + p.o_C);
  uint32_t* CT = (uint32_t*)(ws + p.o_CT);
  uint32_t* BS = (uint32_t*)(ws + p.o_BS);
  uint32_t* ovf = (uint32_t*)(ws + p.o_ovf);
  K* bk = (K*)(ws + p.o_bk);
  uint32_t* bi = (uint32_t*)(ws + p.o_bi);
  const DevInfo& di = dev_info();

  {
    const size_t sm = hist_stage_offset(p.nbins) + Map::kStageBytes;
    auto kern = k_hist<K, Map>;
    set_smem_once(kern, sm);
    {
      HG_TRACE("k_hist", st);
      kern<<<p.G, kHistThreads, sm, st>>>(keys, p.n, p.chunk, p.s, p.nbins, p.sshift, p.nsb, H, C, map,
                                          (uint32_t)Map::kStageBytes, hdr);
    }
  }
  // With one pass a super-bin is a bin: C, CT serve for H, T.
  const bool two = p.sshift > 0;
  uint32_t* const T = two ? (uint32_t*)(ws + p.o_T) : CT;
  const bool small = !two && p.G <= kScanSmallChunks && p.nbins <= 256;
  if (two) {
    HG_TRACE("k_colscan", st);
    colscan_launch(H, p.G, p.nbins, T, st);
  }
  if (!small) {
    HG_TRACE("k_colscan", st);
    colscan_launch(C, p.G, p.nsb, CT, st);
  }
  // Implicit ids are input positions, so the bin build can restore the
  // canonical order (ascending position in every bucket) from the ids
  // alone; then, unless k_scan_bins finds a bin too large for the
  // shared-memory bin build, the partitions may rank tiles in any order.
  // Both variants of each such kernel are launched; the one that does not
  // match the order mode returns at once.
  const bool any_order = ids == nullptr || positional_ids;
  BinCfg bc, bw;
  bin_configs<K>(p, any_order, &bc, &bw);
  const uint32_t emax_all = bw.emax;
  const bool may_overflow = p.n > emax_all;  // else no bin can be too large for shared memory
  // bins for the bin build's second launch, counted by k_scan_bins
  uint32_t* const wide_count = (uint32_t*)&hdr->counters[7];
  if (small) {
    HG_TRACE("k_scan_bins", st);
    k_scan_small<<<1, 1024, 0, st>>>(C, p.G, p.nbins, CT, BS, emax_all, ovf, &hdr->ovf_count, offsets, p.V,
                                     pos_base + (uint32_t)p.n, any_order ? &hdr->order_mode : nullptr, bc.emax,
                                     bc.nt != bw.nt ? wide_count : nullptr);
  } else {
    HG_TRACE("k_scan_bins", st);
    HugeArgs h{};
    // below kHugeMinN keys every oversized bin goes to the one-CTA path (at
    // most a few million edges), which spares small builds three launches
    if (p.n >= kHugeMinN) h.list = (uint32_t*)(ws + p.o_hlist);
    h.count = (uint32_t*)&hdr->counters[0];
    h.rows = (uint32_t*)&hdr->counters[0] + 1;
    h.rowdesc = (uint32_t*)(ws + p.o_rowdesc);
    h.max_rows = p.max_rows;
    h.status = status;
    // bins above the largest the shared-memory bin build takes (the second
    // launch included) go to the oversized-bin kernels
    k_scan_bins<<<1, 1024, 0, st>>>(T, p.nbins, BS, emax_all, ovf, &hdr->ovf_count, offsets, p.V,
                                    pos_base + (uint32_t)p.n, h, any_order ? &hdr->order_mode : nullptr, bc.emax,
                                    bc.nt != bw.nt ? wide_count : nullptr, any_order && two ? H : nullptr);
  }

  PartArgs<K> pa{};
  pa.in_k = keys;
  pa.in_i = ids;
  // With two partition passes, pass A's output lives in the caller's CSR
  // arrays until pass B has read it; with one pass it goes straight to the
  // workspace, so that no bin build reads and writes the same region.
  pa.out_k = two ? csr_k : bk;
  pa.out_i = two ? csr_i : bi;
  pa.n = p.n;
  pa.chunk = p.chunk;
  pa.G = p.G;
  pa.s = p.s;
  pa.sshift = p.sshift;
  pa.nbins = p.nbins;
  pa.nsb = p.nsb;
  pa.H = H;
  pa.C = C;
  pa.CT = CT;
  pa.BS = BS;
  pa.cur_bin = H;  // chunk 0's row
  pa.status = status;
  {
    pa.order = any_order ? &hdr->order_mode : nullptr;
    HG_TRACE("k_partition_A", st);
    // the map's tables are staged only where they fit next to the tile
    constexpr int ipt = part_ipt_keys<K>();
    PartArgs<K> x = pa;
    const size_t own = part_smem_bytes(sizeof(K), ids != nullptr, ipt, false, kPartNW);
    if (ids == nullptr && p.n < kHugeMinN) {
      const size_t need = std::max(own, part_any_smem(sizeof(K), false, PartA<K>::NT * PartA<K>::IPT, 256));
      const size_t cap = std::min((size_t)di.max_smem_optin,
                                  (size_t)di.smem_per_sm / PartA<K>::MINB - (size_t)di.smem_reserved);
      x.stage_bytes = need + Map::kStageBytes <= cap ? (uint32_t)Map::kStageBytes : 0u;
      auto kern = k_partition_a<K, Map>;
      set_smem_once(kern, need + x.stage_bytes);
      kern<<<p.G, kPartNW * 32, need + x.stage_bytes, st>>>(x, map);
    } else {
      if (ids == nullptr) partition_any_launch<K, Map, false, false, PartA<K>>(pa, map, p.G, st);
      else if (any_order) partition_any_launch<K, Map, false, true, PartB<K>>(pa, map, p.G, st);
      auto kern = k_partition<K, Map, false, ipt, kPartNW, part_minb_keys<K>()>;
      x.stage_bytes = own + Map::kStageBytes <= (size_t)di.max_smem_optin ? (uint32_t)Map::kStageBytes : 0u;
      set_smem_once(kern, own + x.stage_bytes);
      kern<<<p.G, kPartNW * 32, own + x.stage_bytes, st>>>(x, map);
    }
  }
  if (two) {
    PartArgs<K> pb = pa;
    pb.in_k = csr_k;
    pb.in_i = csr_i;
    pb.out_k = bk;
    pb.out_i = bi;
    pb.stage_bytes = 0;  // (staging would cost pass B a resident CTA per SM)
    // ~32K edges per item: enough to amortise the per-item set-up
    const uint64_t per_chunk_sb = std::max<uint64_t>(1, p.n / ((uint64_t)p.G * p.nsb));
    pb.gg = (uint32_t)std::min<uint64_t>(p.G, std::max<uint64_t>(1, 32768 / per_chunk_sb));
    pb.ngroups = (p.G + pb.gg - 1) / pb.gg;
    const uint64_t items = (uint64_t)p.nsb * pb.ngroups;
    HG_TRACE("k_partition_B", st);
    if (any_order) partition_b_any<K, Map>(pb, map, st);
    if (!any_order || may_overflow) {
      auto kern = k_partition<K, Map, true, kPartIPTB, kPartNWB, kPartMinBlocksB>;
      const size_t sm = part_smem_bytes(sizeof(K), true, kPartIPTB, true, kPartNWB);
      set_smem_once(kern, sm);
      int per_sm = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPartNWB * 32, sm);
      unsigned grid = (unsigned)std::min<uint64_t>(items, (uint64_t)std::max(1, per_sm) * di.sms);
      grid = (unsigned)std::max<uint64_t>(grid, (items + kMaxItemsPerCta - 1) / kMaxItemsPerCta);
      kern<<<grid, kPartNWB * 32, sm, st>>>(pb, map);
    }
  }
  // A partition that could not be launched (say, a tile geometry built in at
  // compile time that needs more shared memory than a CTA may have) left the
  // bins unwritten: stop before the bin build reads them.
  if (cudaPeekAtLastError() != cudaSuccess) return last_launch_status();
  BinArgs<K> ba{};
  ba.in_k = bk;
  ba.in_i = bi;
  ba.csr_k = csr_k;
  ba.csr_i = csr_i;
  ba.offsets = offsets;
  ba.T = T;
  ba.BS = BS;
  ba.V = p.V;
  ba.nbins = p.nbins;
  ba.s = p.s;
  ba.pos_base = pos_base;
  ba.order = any_order ? &hdr->order_mode : nullptr;
  if (may_overflow) {  // (with room for them in the launch of 1024-thread CTAs)
    ba.ovf_list = ovf;
    ba.ovf_count = &hdr->ovf_count;
    const size_t big = big_smem_bytes(sizeof(K), 1u << p.s);
    bw.smem = std::max(bw.smem, big);
    if (bc.nt == bw.nt) bc.smem = std::max(bc.smem, big);
  }
  {
    HG_TRACE("k_binbuild", st);
    binbuild_launch<K, Map>(ba, map, bc, 0, nullptr, st);
    if (bc.nt != bw.nt) binbuild_launch<K, Map>(ba, map, bw, bc.emax, wide_count, st);
  }
  if (p.n >= kHugeMinN) {
    // bins above kHugeSeg edges (duplicates): several CTAs per bin
    const uint32_t nbmax = 1u << p.s;
    uint32_t* hcount = (uint32_t*)&hdr->counters[0];
    uint32_t* hrows = hcount + 1;
    const uint32_t* hlist = (const uint32_t*)(ws + p.o_hlist);
    const uint32_t* rowdesc = (const uint32_t*)(ws + p.o_rowdesc);
    uint32_t* rowcnt = (uint32_t*)(ws + p.o_rowcnt);
    const unsigned grid = (unsigned)std::min<uint64_t>(p.max_rows, (uint64_t)di.sms);
    const unsigned hgrid = (unsigned)std::min<uint64_t>(p.n / kHugeSeg + 1, (uint64_t)di.sms);
    HG_TRACE("k_binbuild_huge", st);
    auto kc = k_huge_count<K, Map>;
    set_smem_once(kc, (size_t)nbmax * 4);
    kc<<<grid, kBinNW * 32, (size_t)nbmax * 4, st>>>(ba, hrows, rowdesc, rowcnt, map);
    auto ks = k_huge_scan<K>;
    set_smem_once(ks, (size_t)nbmax * 4);
    ks<<<hgrid, 1024, (size_t)nbmax * 4, st>>>(ba, hcount, hlist, rowcnt);
    const size_t sm = big_smem_bytes(sizeof(K), nbmax);
    auto kx = k_huge_scatter<K, Map>;
    set_smem_once(kx, sm);
    kx<<<grid, kBinNW * 32, sm, st>>>(ba, hrows, rowdesc, rowcnt, map);
  }
  return last_launch_status();
}

bool v2_plan_fits(const Plan& p) {
  if (p.n == 0) return true;
  const double mean = (double)p.n * (double)(1ull << p.s) / (double)p.V;
  return mean + 5.0 * std::sqrt(mean) + 16.0 <= (double)p.emax;
}

bool make_slab_plan(const hg_config* cfg, uint64_t n, SlabPlan* p) {
  if (cfg->bin_shift != 0 || n == 0) return false;  // an explicit bin size asks for one two-level plan
  const DevInfo& di = dev_info();
  p->kb = cfg->key_type == HG_KEY_U64 ? 8 : 4;
  p->n = n;
  p->V = cfg->num_buckets;
  const double emax = p->kb == 4 ? kBinEmaxU32 : kBinEmaxU64;
  const double alpha = (double)n / (double)p->V;
  // largest bins (2^s buckets) that still fit shared memory at this load
  int s_fit = -1;
  for (int s = 0; s <= (int)kMaxBinShift; ++s) {
    const double mean = alpha * (double)(1ull << s);
    if (mean + 5.0 * std::sqrt(mean) + 16.0 <= emax) s_fit = s;
  }
  if (s_fit < 0) return false;  // a bin of one bucket would overflow: no relabeling helps
  p->Ls = (uint32_t)s_fit + kMaxBinsLog2;
  const uint64_t S = (p->V + (1ull << p->Ls) - 1) >> p->Ls;
  if (S < 2 || S > 256) return false;
  p->S = (uint32_t)S;
  const int sms = std::max(di.sms, 1);
  uint64_t chunk = std::max<uint64_t>(kPartTile, (n + 2 * sms - 1) / (2 * sms));
  chunk = (chunk + 15) / 16 * 16;
  p->chunk = chunk;
  p->G = (uint32_t)std::max<uint64_t>(1, (n + chunk - 1) / chunk);
  hg_config cs = *cfg;
  cs.num_buckets = std::min<uint64_t>(1ull << p->Ls, p->V);
  cs.bin_shift = 0;
  if (!make_plan_v2(&cs, n, &p->sub)) return false;
  size_t o = sizeof(WsHeader);
  p->o_H = o;   o = align_up(o + (size_t)p->G * p->S * 4);
  p->o_C = o;   o = align_up(o + (size_t)p->G * p->S * 4);
  p->o_CT = o;  o = align_up(o + (size_t)p->S * 4);
  p->o_T = o;   o = align_up(o + (size_t)p->S * 4);
  p->o_BS = o;  o = align_up(o + ((size_t)p->S + 1) * 4);
  p->o_ovf = o; o = align_up(o + (size_t)p->S * 4 + 16);
  p->o_k = o;   o = align_up(o + ((size_t)n + 16) * p->kb);
  p->o_i = o;   o = align_up(o + ((size_t)n + 16) * 4);
  p->o_sub = o; o = align_up(o + p->sub.total);
  p->total = o;
  // the same table as one two-level build (build_wide): bins of the slabs'
  // size, up to 256 in each of up to 512 super-bins
  Plan& w = p->wide;
  w = Plan{};
  const uint64_t nbins = ((p->V - 1) >> s_fit) + 1;
  if (nbins > (1ull << 17)) return true;
  w.kb = p->kb;
  w.n = n;
  w.V = p->V;
  w.s = (uint32_t)s_fit;
  w.sshift = 8;
  w.nbins = (uint32_t)nbins;
  w.nsb = (uint32_t)(((nbins - 1) >> w.sshift) + 1);
  w.G = p->G;
  w.chunk = p->chunk;
  w.emax = p->sub.emax;
  w.tpb = cfg->threads_per_bin;
  o = sizeof(WsHeader);
  w.o_H = o;      o = align_up(o + (size_t)w.G * w.nsb * 4);
  w.o_C = o;      o = align_up(o + (size_t)w.G * w.nsb * 4);
  w.o_CT = o;     o = align_up(o + (size_t)w.nsb * 4);
  w.o_T = o;      o = align_up(o + (size_t)w.nbins * 4);
  w.o_BS = o;     o = align_up(o + ((size_t)w.nbins + 1) * 4);
  p->o_wcur = o;  o = align_up(o + (size_t)w.nbins * 4);
  p->o_wsbs = o;  o = align_up(o + ((size_t)w.nsb + 1) * 4);
  w.o_ovf = o;    o = align_up(o + (size_t)w.nbins * 4 + 16);
  w.o_bk = o;     o = align_up(o + ((size_t)n + 16) * w.kb);
  w.o_bi = o;     o = align_up(o + ((size_t)n + 16) * 4);
  w.total = o;
  p->total = std::max(p->total, o);
  return true;
}

__global__ void k_fill_u32(uint32_t* __restrict__ a, uint64_t n, uint32_t v) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    a[i] = v;
}

// A slab build records its device errors in its own workspace header; they
// are carried over to the caller's.
__global__ void k_carry_status(const uint32_t* __restrict__ from, uint32_t* to) {
  if (*from) set_status(to, *from);
}

// Tables of more bins than one shared-memory histogram holds, implicit ids:
// one two-level build all the same, with up to 512 super-bins in pass A and
// the bin totals counted from pass A's output (k_hist_late).  The host reads
// whether every bin fits the shared-memory bin build (one stream
// synchronisation); if not, nothing is built (*done = false) and the slabs
// take over.  Spares the slabs' stable partition of the whole input: build of
// 2^30 uint32 keys 18.6 ms, of the same keys through the slabs 36.6 (explicit ids).
template <typename K, typename Map>
static hg_status build_wide(const SlabPlan& sp, const K* keys, uint32_t* offsets, K* csr_k, uint32_t* csr_i,
                            uint8_t* ws, cudaStream_t st, Map map, bool* done) {
  *done = false;
  const Plan& p = sp.wide;
  WsHeader* hdr = (WsHeader*)ws;
  uint32_t* H = (uint32_t*)(ws + p.o_H);
  uint32_t* C = (uint32_t*)(ws + p.o_C);
  uint32_t* CT = (uint32_t*)(ws + p.o_CT);
  uint32_t* T = (uint32_t*)(ws + p.o_T);
  uint32_t* BS = (uint32_t*)(ws + p.o_BS);
  uint32_t* cur = (uint32_t*)(ws + sp.o_wcur);
  uint32_t* sbs = (uint32_t*)(ws + sp.o_wsbs);
  uint32_t* ovf = (uint32_t*)(ws + p.o_ovf);
  K* bk = (K*)(ws + p.o_bk);
  uint32_t* bi = (uint32_t*)(ws + p.o_bi);
  const DevInfo& di = dev_info();
  const uint32_t sb_log2 = p.s + p.sshift;  // buckets per super-bin
  {
    const size_t sm = hist_stage_offset(p.nsb) + Map::kStageBytes;
    auto kern = k_hist<K, Map>;
    set_smem_once(kern, sm);
    HG_TRACE("k_hist", st);
    kern<<<p.G, kHistThreads, sm, st>>>(keys, p.n, p.chunk, sb_log2, p.nsb, 0, p.nsb, H, C, map,
                                        (uint32_t)Map::kStageBytes, nullptr);
    colscan_launch(C, p.G, p.nsb, CT, st);
    k_scan_bins<<<1, 1024, 0, st>>>(CT, p.nsb, sbs, 0xffffffffu, ovf, &hdr->ovf_count, ovf + p.nsb, 0, (uint32_t)p.n,
                                    HugeArgs{}, nullptr);
  }
  PartArgs<K> a{};
  a.in_k = keys;
  a.out_k = csr_k;
  a.out_i = csr_i;
  a.n = p.n;
  a.chunk = p.chunk;
  a.G = p.G;
  a.s = sb_log2;  // pass A and the late histogram know super-bins by their starts alone
  a.nbins = p.nsb;
  a.nsb = p.nsb;
  a.C = C;
  a.CT = CT;
  a.BS = sbs;
  a.status = &hdr->status;
  {
    HG_TRACE("k_partition_A", st);
    partition_any_launch<K, Map, false, false, PartA<K>, 512>(a, map, p.G, st);
  }
  a.in_k = csr_k;
  a.in_i = csr_i;
  a.out_k = bk;
  a.out_i = bi;
  a.s = p.s;
  a.sshift = p.sshift;
  a.nbins = p.nbins;
  if (cudaMemsetAsync(T, 0, (size_t)p.nbins * 4, st) != cudaSuccess) return HG_ERR_CUDA;
  {
    HG_TRACE("k_hist_late", st);
    const uint64_t pieces = (p.n + kLatePiece - 1) / kLatePiece;
    k_hist_late<K, Map><<<(unsigned)std::min<uint64_t>(pieces, 4ull * di.sms), 512, 0, st>>>(a, T, map);
  }
  BinCfg bc, bw;
  bin_configs<K>(p, true, &bc, &bw);
  uint32_t* const wide_count = (uint32_t*)&hdr->counters[7];
  {
    HG_TRACE("k_scan_bins", st);
    k_scan_bins<<<1, 1024, 0, st>>>(T, p.nbins, BS, bw.emax, ovf, &hdr->ovf_count, offsets, p.V, (uint32_t)p.n,
                                    HugeArgs{}, &hdr->order_mode, bc.emax, bc.nt != bw.nt ? wide_count : nullptr, cur);
  }
  if (cudaPeekAtLastError() != cudaSuccess) return last_launch_status();
  uint32_t order = 1;
  if (cudaMemcpyAsync(&order, &hdr->order_mode, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return HG_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return HG_ERR_CUDA;
  if (order != 0) return HG_OK;
  *done = true;
  a.BS = BS;
  a.cur_bin = cur;
  {
    HG_TRACE("k_partition_B", st);
    partition_b_any<K, Map>(a, map, st);
  }
  if (cudaPeekAtLastError() != cudaSuccess) return last_launch_status();
  BinArgs<K> ba{};
  ba.in_k = bk;
  ba.in_i = bi;
  ba.csr_k = csr_k;
  ba.csr_i = csr_i;
  ba.offsets = offsets;
  ba.T = T;
  ba.BS = BS;
  ba.V = p.V;
  ba.nbins = p.nbins;
  ba.s = p.s;
  ba.order = &hdr->order_mode;
  HG_TRACE("k_binbuild", st);
  binbuild_launch<K, Map>(ba, map, bc, 0, nullptr, st);
  if (bc.nt != bw.nt) binbuild_launch<K, Map>(ba, map, bw, bc.emax, wide_count, st);
  return last_launch_status();
}

template <typename K, typename Map>
hg_status build_slabs(const hg_config* cfg, const SlabPlan& p, const K* keys, const uint32_t* ids,
                      uint32_t* offsets, K* csr_k, uint32_t* csr_i, uint8_t* ws, cudaStream_t st, Map map) {
  WsHeader* hdr = (WsHeader*)ws;
  uint32_t* H = (uint32_t*)(ws + p.o_H);
  uint32_t* C = (uint32_t*)(ws + p.o_C);
  uint32_t* CT = (uint32_t*)(ws + p.o_CT);
  uint32_t* T = (uint32_t*)(ws + p.o_T);
  uint32_t* BS = (uint32_t*)(ws + p.o_BS);
  uint32_t* ovf = (uint32_t*)(ws + p.o_ovf);
  K* lk = (K*)(ws + p.o_k);
  uint32_t* li = (uint32_t*)(ws + p.o_i);
  uint8_t* sub = ws + p.o_sub;
  const DevInfo& di = dev_info();
  if (p.wide.total != 0 && ids == nullptr) {
    bool done;
    const hg_status rc = build_wide<K, Map>(p, keys, offsets, csr_k, csr_i, ws, st, map, &done);
    if (rc != HG_OK || done) return rc;
    if (cudaMemsetAsync(ws, 0, sizeof(WsHeader), st) != cudaSuccess) return HG_ERR_CUDA;
  }
  // 1. slab of every key (bucket >> Ls), counted per input chunk
  {
    const size_t sm = hist_stage_offset(p.S) + Map::kStageBytes;
    auto kern = k_hist<K, Map>;
    set_smem_once(kern, sm);
    HG_TRACE("k_hist_slab", st);
    kern<<<p.G, kHistThreads, sm, st>>>(keys, p.n, p.chunk, p.Ls, p.S, 0, p.S, H, C, map,
                                        (uint32_t)Map::kStageBytes, nullptr);
    colscan_launch(H, p.G, p.S, T, st);
    colscan_launch(C, p.G, p.S, CT, st);
    k_scan_bins<<<1, 1024, 0, st>>>(T, p.S, BS, 0xffffffffu, ovf, &hdr->ovf_count, ovf + p.S, 0, (uint32_t)p.n,
                                    HugeArgs{}, nullptr);
  }
  // 2. stable partition by slab: each slab keeps its keys in input order,
  //    with their ids (the input positions when none are given)
  {
    PartArgs<K> pa{};
    pa.in_k = keys;
    pa.in_i = ids;
    pa.out_k = lk;
    pa.out_i = li;
    pa.n = p.n;
    pa.chunk = p.chunk;
    pa.G = p.G;
    pa.s = p.Ls;
    pa.sshift = 0;
    pa.nbins = p.S;
    pa.nsb = p.S;
    pa.H = H;
    pa.C = C;
    pa.CT = CT;
    pa.BS = BS;
    pa.status = &hdr->status;
    pa.order = nullptr;
    constexpr int ipt = part_ipt_keys<K>();
    auto kern = k_partition<K, Map, false, ipt, kPartNW, part_minb_keys<K>()>;
    const size_t own = part_smem_bytes(sizeof(K), ids != nullptr, ipt, false, kPartNW);
    pa.stage_bytes = own + Map::kStageBytes <= (size_t)di.max_smem_optin ? (uint32_t)Map::kStageBytes : 0u;
    set_smem_once(kern, own + pa.stage_bytes);
    HG_TRACE("k_partition_slab", st);
    kern<<<p.G, kPartNW * 32, own + pa.stage_bytes, st>>>(pa, map);
  }
  if (cudaPeekAtLastError() != cudaSuccess) return last_launch_status();  // partition not launched
  // 3. slab sizes to the host, then one two-level build per slab
  uint32_t hT[256];
  if (cudaMemcpyAsync(hT, T, (size_t)p.S * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return HG_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return HG_ERR_CUDA;
  uint64_t start = 0;
  for (uint32_t sl = 0; sl < p.S; ++sl) {
    const uint64_t b0 = (uint64_t)sl << p.Ls;
    const uint64_t Vs = std::min<uint64_t>(1ull << p.Ls, p.V - b0);
    const uint64_t ns = hT[sl];
    if (ns == 0) {
      k_fill_u32<<<(unsigned)std::min<uint64_t>((Vs + 256) / 256, (uint64_t)di.sms * 8), 256, 0, st>>>(
          offsets + b0, Vs + 1, (uint32_t)start);
      continue;
    }
    hg_config cs = *cfg;
    cs.num_buckets = Vs;
    cs.bin_shift = 0;
    Plan ps{};
    if (!make_plan_v2(&cs, ns, &ps) || ps.total > p.sub.total) return HG_ERR_UNSUPPORTED;
    Map ms = map;
    ms.slab_base = (uint32_t)b0;
    if (cudaMemsetAsync(sub, 0, sizeof(WsHeader), st) != cudaSuccess) return HG_ERR_CUDA;
    hg_status rc = build_v2<K, Map>(ps, lk + start, li + start, offsets + b0, csr_k + start, csr_i + start, sub, st,
                                    ms, (uint32_t)start, ids == nullptr);
    if (rc != HG_OK) return rc;
    k_carry_status<<<1, 1, 0, st>>>(&((WsHeader*)sub)->status, &hdr->status);
    start += ns;
  }
  return last_launch_status();
}

size_t v1_workspace_bytes(int kb, uint64_t n, uint64_t V) {
  size_t o = sizeof(WsHeader);
  o = align_up(o + (size_t)V * 4);                  // cursors
  o = align_up(o + scan_workspace_bytes<uint32_t>(V + 1));    // scan partials
  o = align_up(o + (size_t)V * 4);                  // heavy list
  o = align_up(o + ((size_t)n + 16) * kb);          // temp keys
  o = align_up(o + ((size_t)n + 16) * 4);           // temp positions
  return o;
}

template <typename K, typename Map>
hg_status build_v1(uint64_t n, uint64_t V, const K* keys, const uint32_t* ids, uint32_t* offsets, K* csr_k,
                   uint32_t* csr_i, uint8_t* ws, cudaStream_t st, Map map) {
  WsHeader* hdr = (WsHeader*)ws;
  size_t o = sizeof(WsHeader);
  uint32_t* cursor = (uint32_t*)(ws + o); o = align_up(o + (size_t)V * 4);
  uint32_t* part = (uint32_t*)(ws + o);   o = align_up(o + scan_workspace_bytes<uint32_t>(V + 1));
  uint32_t* heavy = (uint32_t*)(ws + o);  o = align_up(o + (size_t)V * 4);
  K* tk = (K*)(ws + o);                   o = align_up(o + ((size_t)n + 16) * sizeof(K));
  uint32_t* ti = (uint32_t*)(ws + o);
  const int sms = dev_info().sms;
  const unsigned grid = (unsigned)std::max(1, sms * 8);
  cudaMemsetAsync(offsets, 0, (size_t)(V + 1) * 4, st);
  cudaMemsetAsync(cursor, 0, (size_t)V * 4, st);
  {
    HG_TRACE("k_v1_count", st);
    k_v1_count<K, Map><<<grid, 256, 0, st>>>(keys, n, offsets, map);
  }
  hg_status rc = device_excl_scan<uint32_t>(offsets, V + 1, part, st);
  if (rc != HG_OK) return rc;
  {
    HG_TRACE("k_v1_scatter", st);
    k_v1_scatter<K, Map><<<grid, 256, 0, st>>>(keys, n, offsets, cursor, csr_k, csr_i, map);
  }
  {
    HG_TRACE("k_v1_fix_small", st);
    k_v1_fix_small<K><<<grid, 256, 0, st>>>(offsets, V, csr_k, csr_i, heavy, &hdr->heavy_count);
  }
  uint32_t nbits = 8;
  while (nbits < 32 && (n - 1) >> nbits) nbits += 8;
  {
    const size_t sm = align_up((size_t)kV1HeavyNW * 32 * kV1HeavyIPT * (sizeof(K) + 5) +
                               (size_t)rank_words<kV1HeavyNW>() * 4 + 2 * 256 * 4, 16) + 32 * 4 + 64;
    auto kern = k_v1_fix_heavy<K>;
    set_smem_once(kern, sm);
    {
      HG_TRACE("k_v1_fix_heavy", st);
      kern<<<(unsigned)std::max(1, sms), kV1HeavyNW * 32, sm, st>>>(offsets, heavy, &hdr->heavy_count, csr_k,
                                                                    csr_i, tk, ti, nbits);
    }
  }
  if (ids) {
    HG_TRACE("k_v1_ids", st);
    k_v1_ids<<<grid, 256, 0, st>>>(csr_i, ids, n);
  }
  return last_launch_status();
}

// ===========================================================================
// Binned probe.  HashGraph-Probe-Standard answers each query with random
// reads into the table; on HBM every random 4-byte read costs a whole DRAM
// burst.  Here the queries are first partitioned by bucket range into ng
// groups (the build's histogram and partition kernels, applied to the
// queries), so that the group being probed touches one table slice small
// enough to stay in L2; the per-query counts are then put back in query
// order by a merge over the groups (inside a group the query positions
// ascend from one block of kQueryBlock positions to the next).
// ===========================================================================
// Counts back to query order when the positions inside every group come in
// long ascending runs (batched tables: a table's queries fall into one or two
// groups): a plain in-order scatter, coalesced along each run.
__global__ void k_scatter_counts(const uint32_t* __restrict__ Qi, const uint32_t* __restrict__ Qc, uint64_t Q,
                                 uint32_t* __restrict__ counts) {
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < Q; j += (uint64_t)gridDim.x * blockDim.x)
    counts[__ldcs(Qi + j)] = __ldcs(Qc + j);
}

#ifndef HG_UNPERMUTE_TILE
#define HG_UNPERMUTE_TILE 32768
#endif
constexpr int kUnpermuteThreads = 1024;
constexpr uint32_t kUnpermuteTile = HG_UNPERMUTE_TILE;  // outputs per merge tile (shared memory: 4 B each)

// Every warp merges the groups warp, warp + 32, ... (GPW of them); per round
// it loads UNR runs of 32 (position, count) pairs of each of its groups, so
// GPW * UNR pairs per lane are in flight (eight for any number of groups).
template <int GPW, int UNR>
__global__ void __launch_bounds__(kUnpermuteThreads) k_unpermute(const uint32_t* __restrict__ Qi,
                                                                 const uint32_t* __restrict__ Qc,
                                                                 const uint32_t* __restrict__ GS, uint32_t ng,
                                                                 uint64_t Q, uint64_t span,
                                                                 uint32_t* __restrict__ counts) {
  __shared__ uint32_t cur[256], gend[256];
  extern __shared__ uint32_t out_s[];  // kUnpermuteTile entries
  const uint64_t ob = (uint64_t)blockIdx.x * span;
  if (ob >= Q) return;
  const uint64_t oe = min(ob + span, Q);
  if (threadIdx.x < ng) {  // first query of each group at or after ob
    uint32_t lo = GS[threadIdx.x], hi = GS[threadIdx.x + 1];
    gend[threadIdx.x] = hi;
    while (lo < hi) {
      const uint32_t mid = lo + ((hi - lo) >> 1);
      if (Qi[mid] < ob) lo = mid + 1; else hi = mid;
    }
    cur[threadIdx.x] = lo;
  }
  __syncthreads();
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (uint64_t o0 = ob; o0 < oe; o0 += kUnpermuteTile) {
    const uint64_t o1 = min(o0 + (uint64_t)kUnpermuteTile, oe);
    uint32_t c[GPW], e[GPW];
    bool act[GPW];
#pragma unroll
    for (int k = 0; k < GPW; ++k) {
      const uint32_t g = warp + k * nw;
      act[k] = g < ng;
      c[k] = act[k] ? cur[g] : 0u;
      e[k] = act[k] ? gend[g] : 0u;
    }
    bool any = true;
    while (any) {
      uint32_t v[GPW][UNR], x[GPW][UNR];
#pragma unroll
      for (int k = 0; k < GPW; ++k) {
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
          v[k][u] = 0xffffffffu;
          x[k][u] = 0u;
          const uint32_t j = c[k] + 32u * u + lane;
          if (act[k] && j < e[k]) {
            v[k][u] = __ldcs(Qi + j);
            x[k][u] = __ldcs(Qc + j);
          }
        }
      }
      any = false;
#pragma unroll
      for (int k = 0; k < GPW; ++k) {
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
          if (!act[k]) break;  // warp-uniform
          const bool in = (uint64_t)v[k][u] < o1;
          if (in) out_s[v[k][u] - (uint32_t)o0] = x[k][u];
          const uint32_t n = __popc(__ballot_sync(kFull, in));
          c[k] += n;
          act[k] = n == 32;
        }
        any |= act[k];
      }
    }
#pragma unroll
    for (int k = 0; k < GPW; ++k) {
      const uint32_t g = warp + k * nw;
      if (g < ng && lane == 0) cur[g] = c[k];
    }
    __syncthreads();
    for (uint32_t t = threadIdx.x; t < (uint32_t)(o1 - o0); t += blockDim.x) __stcs(counts + o0 + t, out_s[t]);
    __syncthreads();
  }
}

// Counts back to query order, balanced over the warps whatever the group
// sizes (a skewed bucket map can put half of the queries into one group).
// For every output tile [o0, o1) the run of each group (its elements with
// positions in the tile, contiguous in its arrays) has the length the query
// partition recorded for the partition tiles that make up the output tile
// (TC: ng 16-bit counts per partition tile of ptile queries).  The runs,
// back to back, are split evenly over the warps; each lane keeps
// kUnpermuteUNR (position, count) pairs in flight and scatters them into the
// tile in shared memory, which is then written out coalesced.
constexpr int kUnpermuteUNR = 8;
__global__ void __launch_bounds__(kUnpermuteThreads) k_unpermute_bal(
    const uint32_t* __restrict__ Qi, const uint32_t* __restrict__ Qc, const uint32_t* __restrict__ GS, uint32_t ng,
    const uint16_t* __restrict__ TC, uint32_t ptile, uint64_t Q, uint64_t span, uint32_t* __restrict__ counts) {
  __shared__ uint32_t cur[256], run[256], rstart[257], wsum[32];
  extern __shared__ uint32_t out_s[];  // kUnpermuteTile entries
  const uint64_t ob = (uint64_t)blockIdx.x * span;
  if (ob >= Q) return;
  const uint64_t oe = min(ob + span, Q);
  if (threadIdx.x < ng) {  // first query of each group at or after ob
    uint32_t lo = GS[threadIdx.x], hi = GS[threadIdx.x + 1];
    while (lo < hi) {
      const uint32_t mid = lo + ((hi - lo) >> 1);
      if (Qi[mid] < ob) lo = mid + 1; else hi = mid;
    }
    cur[threadIdx.x] = lo;
  }
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (uint64_t o0 = ob; o0 < oe; o0 += kUnpermuteTile) {
    const uint64_t o1 = min(o0 + (uint64_t)kUnpermuteTile, oe);
    const uint32_t total = (uint32_t)(o1 - o0);
    // 1. every group's run in this tile, and where it starts among all runs
    uint32_t r = 0;
    if (threadIdx.x < ng)
      for (uint64_t t = o0 / ptile; t * ptile < o1; ++t) r += TC[t * ng + threadIdx.x];
    const uint32_t st = block_excl_scan<uint32_t>(r, wsum, (uint32_t*)nullptr);
    if (threadIdx.x < ng) {
      run[threadIdx.x] = r;
      rstart[threadIdx.x] = st;
    }
    if (threadIdx.x == 0) rstart[ng] = total;
    __syncthreads();
    // 2. the runs back to back, an equal slice per warp
    const uint32_t per = (total + nw - 1) / nw;
    const uint32_t x0 = min(warp * per, total), x1 = min(x0 + per, total);
    uint32_t g = 0;  // last group whose run starts at or before x0
    {
      uint32_t lo = 0, hi = ng;
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (rstart[mid] <= x0) lo = mid; else hi = mid;
      }
      g = lo;
    }
    for (uint32_t xb = x0; xb < x1; xb += 32u * kUnpermuteUNR) {
      uint32_t v[kUnpermuteUNR], c[kUnpermuteUNR];
#pragma unroll
      for (int u = 0; u < kUnpermuteUNR; ++u) {
        const uint32_t x = xb + 32u * u + lane;
        v[u] = 0xffffffffu;
        c[u] = 0u;
        if (x < x1) {
          while (rstart[g + 1] <= x) ++g;
          const uint32_t j = cur[g] + (x - rstart[g]);
          v[u] = __ldcs(Qi + j);
          c[u] = __ldcs(Qc + j);
        }
      }
#pragma unroll
      for (int u = 0; u < kUnpermuteUNR; ++u)
        if (v[u] != 0xffffffffu) out_s[v[u] - (uint32_t)o0] = c[u];
    }
    __syncthreads();
    if (threadIdx.x < ng) cur[threadIdx.x] += run[threadIdx.x];
    for (uint32_t t = threadIdx.x; t < total; t += blockDim.x) __stcs(counts + o0 + t, out_s[t]);
    __syncthreads();
  }
}

// Queries are grouped by a partition that ranks each tile in any order
// (whole tiles make up a block of kQueryBlock positions, but for the end of
// the queries).  A group's positions are therefore ascending from block to
// block, though not inside a block's run, and the merge works in output
// tiles made of whole blocks: within a group, every query of an earlier
// output tile precedes every query of a later one, which is all its
// cursors need.
constexpr uint64_t kQueryBlock = 8192;
static_assert(kQueryBlock % (PartQ<uint32_t>::NT * PartQ<uint32_t>::IPT) == 0 &&
                  kQueryBlock % (PartQ<uint64_t>::NT * PartQ<uint64_t>::IPT) == 0 && kUnpermuteTile % kQueryBlock == 0,
              "query blocks are whole partition tiles; merge tiles are whole blocks");

// Elements per tile of the query partition (whole tiles per query block).
static uint32_t query_tile(int kb) {
  return kb == 8 ? (uint32_t)(PartQ<uint64_t>::NT * PartQ<uint64_t>::IPT)
                 : (uint32_t)(PartQ<uint32_t>::NT * PartQ<uint32_t>::IPT);
}

bool make_probe_plan(const hg_config* cfg, uint64_t table_n, uint64_t q, ProbePlan* p) {
  const DevInfo& di = dev_info();
  const int kb = cfg->key_type == HG_KEY_U64 ? 8 : 4;
  const uint64_t V = cfg->num_buckets;
  // 128 groups (fewer only for V < 128): a group's slice of the table stays
  // well below L2 up to 2^28 buckets (16 MB slices at load 1), and with many
  // groups every output tile of the merge draws on many of them, which keeps
  // its warps evenly loaded.  256 groups above (32 MB slices at 2^30 buckets).
  (void)table_n;
  int sg = ceil_log2_u64(V) - (V <= (1ull << 28) ? 7 : 8);
  if (sg < 0) sg = 0;
  p->sg = (uint32_t)sg;
  p->ng = (uint32_t)(((V - 1) >> sg) + 1);
  if (p->ng > 256) return false;
  const int sms = std::max(di.sms, 1);
  // chunks are whole query blocks, so every partition tile lies in one
  // block (the merge below relies on it)
  uint64_t chunk = std::max<uint64_t>(kPartTile, (q + 2 * sms - 1) / (2 * sms));
  chunk = (chunk + kQueryBlock - 1) / kQueryBlock * kQueryBlock;
  p->chunk = chunk;
  p->G = (uint32_t)std::max<uint64_t>(1, (q + chunk - 1) / chunk);
  size_t o = sizeof(WsHeader);
  p->o_H = o;   o = align_up(o + (size_t)p->G * p->ng * 4);
  p->o_C = o;   o = align_up(o + (size_t)p->G * p->ng * 4);
  p->o_CT = o;  o = align_up(o + (size_t)p->ng * 4);
  p->o_GS = o;  o = align_up(o + ((size_t)p->ng + 1) * 4);
  p->o_ovf = o; o = align_up(o + (size_t)p->ng * 4 + 16);
  p->o_qk = o;  o = align_up(o + ((size_t)q + 16) * kb);
  p->o_qi = o;  o = align_up(o + ((size_t)q + 16) * 4);
  p->o_qc = o;  o = align_up(o + ((size_t)q + 16) * 4);
  p->ptile = query_tile(kb);
  p->o_tc = o;  o = align_up(o + ((size_t)(q + p->ptile - 1) / p->ptile) * p->ng * 2);
  p->total = o;
  return true;
}

template <typename K, typename Map>
hg_status probe_binned_impl(const ProbePlan& p, uint64_t V, const hg_table* t, const K* queries, uint64_t q,
                            uint32_t* counts, uint8_t* ws, cudaStream_t st, Map map) {
  WsHeader* hdr = (WsHeader*)ws;
  uint32_t* H = (uint32_t*)(ws + p.o_H);
  uint32_t* C = (uint32_t*)(ws + p.o_C);
  uint32_t* CT = (uint32_t*)(ws + p.o_CT);
  uint32_t* GS = (uint32_t*)(ws + p.o_GS);
  uint32_t* ovf = (uint32_t*)(ws + p.o_ovf);
  K* qk = (K*)(ws + p.o_qk);
  uint32_t* qi = (uint32_t*)(ws + p.o_qi);
  uint32_t* qc = (uint32_t*)(ws + p.o_qc);
  const DevInfo& di = dev_info();
  {
    const size_t sm = hist_stage_offset(p.ng) + Map::kStageBytes;
    auto kern = k_hist<K, Map>;
    set_smem_once(kern, sm);
    HG_TRACE("k_hist_Q", st);
    kern<<<p.G, kHistThreads, sm, st>>>(queries, q, p.chunk, p.sg, p.ng, 0, p.ng, H, C, map,
                                        (uint32_t)Map::kStageBytes, nullptr);
  }
  {
    HG_TRACE("k_colscan_Q", st);
    colscan_launch(C, p.G, p.ng, CT, st);
  }
  {
    HG_TRACE("k_scan_Q", st);
    // no bin is "oversized" here; the closing-offset store goes to scratch
    k_scan_bins<<<1, 1024, 0, st>>>(CT, p.ng, GS, 0xffffffffu, ovf, &hdr->ovf_count, ovf + p.ng, 0,
                                    (uint32_t)q, HugeArgs{}, nullptr);
  }
  PartArgs<K> pa{};
  pa.in_k = queries;
  pa.in_i = nullptr;  // ids = query positions
  pa.out_k = qk;
  pa.out_i = qi;
  pa.n = q;
  pa.chunk = p.chunk;
  pa.G = p.G;
  pa.s = p.sg;
  pa.sshift = 0;
  pa.nbins = p.ng;
  pa.nsb = p.ng;
  pa.H = H;
  pa.C = C;
  pa.CT = CT;
  pa.BS = GS;
  pa.status = &hdr->status;
  pa.tile_counts = Map::kSkewed ? (uint16_t*)(ws + p.o_tc) : nullptr;
  {
    HG_TRACE("k_partition_Q", st);
    partition_any_launch<K, Map, false, false, PartQ<K>>(pa, map, p.G, st);
  }
  // the probe and the merge index by the grouped positions: none may run on
  // a query partition that was not launched
  if (cudaPeekAtLastError() != cudaSuccess) return last_launch_status();
  // The CTAs of a launch drift apart as they sweep the groups, and with them
  // the table slices in use; where a few of these do not fit L2 together, a
  // launch takes only so many queries (k_probe in all, one launch / launches
  // of 2^26: uint32 keys 2^28 2.07 / 2.11 ms (slices of 16 MB), 2^30 30.5 /
  // 8.9 (32 MB); uint64 2^28 2.70 / 2.28 (24 MB); 2500 batched tables 3.29 /
  // 2.79 with launches of 2^25, 3.03 with 2^26).
  const uint64_t slice = (4 * V + t->n * sizeof(K)) / p.ng;
  const uint64_t step = Map::kNeedsPos ? 1ull << 25 : slice > (17ull << 20) ? 1ull << 26 : q;
  for (uint64_t i = 0; i < q; i += step) {
    hg_status rc = probe_launch<K, Map>(qk + i, std::min(q - i, step), t->d_offsets, (const K*)t->d_keys, qc + i, V,
                                        st, map, Map::kNeedsPos ? qi + i : nullptr);
    if (rc != HG_OK) return rc;
  }
  {
    // every CTA merges a span of at least one block of outputs (in tiles of up to
    // kUnpermuteTile), so small batches still spread over the SMs
    const uint64_t blocks = (q + kQueryBlock - 1) / kQueryBlock;
    const uint64_t grid = std::max<uint64_t>(1, std::min<uint64_t>(blocks, (uint64_t)2 * di.sms));
    const uint64_t span = (blocks + grid - 1) / grid * kQueryBlock;  // whole blocks
    HG_TRACE("k_unpermute", st);
    if (Map::kNeedsPos)
      k_scatter_counts<<<(unsigned)std::min<uint64_t>((q + 255) / 256, (uint64_t)di.sms * 16), 256, 0, st>>>(
          qi, qc, q, counts);
    else {
      if (Map::kSkewed) {
        set_smem_once(k_unpermute_bal, (size_t)kUnpermuteTile * 4);
        k_unpermute_bal<<<(unsigned)grid, kUnpermuteThreads, (size_t)kUnpermuteTile * 4, st>>>(
            qi, qc, GS, p.ng, (const uint16_t*)(ws + p.o_tc), p.ptile, q, span, counts);
      } else {  // even groups: one warp per group merges faster
        auto launch = [&](auto kern) {
          set_smem_once(kern, (size_t)kUnpermuteTile * 4);
          kern<<<(unsigned)grid, kUnpermuteThreads, (size_t)kUnpermuteTile * 4, st>>>(qi, qc, GS, p.ng, q, span,
                                                                                      counts);
        };
        if (p.ng <= 32) launch(k_unpermute<1, 8>);
        else if (p.ng <= 64) launch(k_unpermute<2, 4>);
        else if (p.ng <= 128) launch(k_unpermute<4, 2>);
        else launch(k_unpermute<8, 1>);
      }
    }
  }
  return last_launch_status();
}

bool make_slab_probe_plan(const hg_config* cfg, uint64_t table_n, uint64_t q, SlabProbePlan* p) {
  const uint64_t V = cfg->num_buckets;
  if (V <= (1ull << kBinnedProbeLog2) || q == 0) return false;
  const DevInfo& di = dev_info();
  const int kb = cfg->key_type == HG_KEY_U64 ? 8 : 4;
  p->V = V;
  p->q = q;
  p->Ls = kSlabProbeLog2;
  p->S = (uint32_t)((V + (1ull << p->Ls) - 1) >> p->Ls);
  const int sms = std::max(di.sms, 1);
  // chunks are whole blocks of queries, as in the binned probe (its merge
  // relies on it)
  uint64_t chunk = std::max<uint64_t>(kPartTile, (q + 2 * sms - 1) / (2 * sms));
  chunk = (chunk + kQueryBlock - 1) / kQueryBlock * kQueryBlock;
  p->chunk = chunk;
  p->G = (uint32_t)std::max<uint64_t>(1, (q + chunk - 1) / chunk);
  hg_config cs = *cfg;
  cs.num_buckets = 1ull << p->Ls;
  if (!make_probe_plan(&cs, table_n, q, &p->sub)) return false;
  size_t o = sizeof(WsHeader);
  p->o_H = o;   o = align_up(o + (size_t)p->G * p->S * 4);
  p->o_C = o;   o = align_up(o + (size_t)p->G * p->S * 4);
  p->o_CT = o;  o = align_up(o + (size_t)p->S * 4);
  p->o_GS = o;  o = align_up(o + ((size_t)p->S + 1) * 4);
  p->o_ovf = o; o = align_up(o + (size_t)p->S * 4 + 16);
  p->o_qk = o;  o = align_up(o + ((size_t)q + 16) * kb);
  p->o_qi = o;  o = align_up(o + ((size_t)q + 16) * 4);
  p->o_qc = o;  o = align_up(o + ((size_t)q + 16) * 4);
  p->ptile = query_tile(kb);
  p->o_tc = o;  o = align_up(o + ((size_t)(q + p->ptile - 1) / p->ptile) * p->S * 2);
  p->o_sub = o; o = align_up(o + p->sub.total);
  p->total = o;
  return true;
}

template <typename K, typename Map>
hg_status probe_slabs(const hg_config* cfg, const SlabProbePlan& p, const hg_table* t, const K* queries,
                      uint64_t q, uint32_t* counts, uint8_t* ws, cudaStream_t st, Map map) {
  WsHeader* hdr = (WsHeader*)ws;
  uint32_t* H = (uint32_t*)(ws + p.o_H);
  uint32_t* C = (uint32_t*)(ws + p.o_C);
  uint32_t* CT = (uint32_t*)(ws + p.o_CT);
  uint32_t* GS = (uint32_t*)(ws + p.o_GS);
  uint32_t* ovf = (uint32_t*)(ws + p.o_ovf);
  K* qk = (K*)(ws + p.o_qk);
  uint32_t* qi = (uint32_t*)(ws + p.o_qi);
  uint32_t* qc = (uint32_t*)(ws + p.o_qc);
  uint8_t* sub = ws + p.o_sub;
  const DevInfo& di = dev_info();
  // 1. queries grouped by slab (bucket >> Ls), in whole query blocks
  {
    const size_t sm = hist_stage_offset(p.S) + Map::kStageBytes;
    auto kern = k_hist<K, Map>;
    set_smem_once(kern, sm);
    HG_TRACE("k_hist_Q", st);
    kern<<<p.G, kHistThreads, sm, st>>>(queries, q, p.chunk, p.Ls, p.S, 0, p.S, H, C, map,
                                        (uint32_t)Map::kStageBytes, nullptr);
    colscan_launch(C, p.G, p.S, CT, st);
    k_scan_bins<<<1, 1024, 0, st>>>(CT, p.S, GS, 0xffffffffu, ovf, &hdr->ovf_count, ovf + p.S, 0, (uint32_t)q,
                                    HugeArgs{}, nullptr);
  }
  {
    PartArgs<K> pa{};
    pa.in_k = queries;
    pa.in_i = nullptr;  // ids = query positions
    pa.out_k = qk;
    pa.out_i = qi;
    pa.n = q;
    pa.chunk = p.chunk;
    pa.G = p.G;
    pa.s = p.Ls;
    pa.sshift = 0;
    pa.nbins = p.S;
    pa.nsb = p.S;
    pa.H = H;
    pa.C = C;
    pa.CT = CT;
    pa.BS = GS;
    pa.status = &hdr->status;
    pa.tile_counts = (uint16_t*)(ws + p.o_tc);
    HG_TRACE("k_partition_Q", st);
    partition_any_launch<K, Map, false, false, PartQ<K>>(pa, map, p.G, st);
  }
  if (cudaPeekAtLastError() != cudaSuccess) return last_launch_status();  // partition not launched
  // 2. slab query counts to the host, then the binned probe of every slab
  uint32_t hGS[257];
  if (cudaMemcpyAsync(hGS, GS, ((size_t)p.S + 1) * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) return HG_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return HG_ERR_CUDA;
  for (uint32_t sl = 0; sl < p.S; ++sl) {
    const uint64_t qs = hGS[sl + 1] - hGS[sl];
    if (qs == 0) continue;
    const uint64_t b0 = (uint64_t)sl << p.Ls;
    hg_config cs = *cfg;
    cs.num_buckets = std::min<uint64_t>(1ull << p.Ls, p.V - b0);
    ProbePlan ps{};
    if (!make_probe_plan(&cs, t->n, qs, &ps) || ps.total > p.sub.total) return HG_ERR_UNSUPPORTED;
    hg_table ts = *t;
    ts.d_offsets = t->d_offsets + b0;  // offsets are positions in the whole table's key array
    Map ms = map;
    ms.slab_base = (uint32_t)b0;
    if (cudaMemsetAsync(sub, 0, sizeof(WsHeader), st) != cudaSuccess) return HG_ERR_CUDA;
    hg_status rc = probe_binned_impl<K, Map>(ps, cs.num_buckets, &ts, qk + hGS[sl], qs, qc + hGS[sl], sub, st, ms);
    if (rc != HG_OK) return rc;
    k_carry_status<<<1, 1, 0, st>>>(&((WsHeader*)sub)->status, &hdr->status);
  }
  // 3. counts back to query order
  {
    const uint64_t blocks = (q + kQueryBlock - 1) / kQueryBlock;
    const uint64_t grid = std::max<uint64_t>(1, std::min<uint64_t>(blocks, (uint64_t)2 * di.sms));
    const uint64_t span = (blocks + grid - 1) / grid * kQueryBlock;
    HG_TRACE("k_unpermute", st);
    set_smem_once(k_unpermute_bal, (size_t)kUnpermuteTile * 4);  // a few slabs: a warp per group would idle most warps
    k_unpermute_bal<<<(unsigned)grid, kUnpermuteThreads, (size_t)kUnpermuteTile * 4, st>>>(
        qi, qc, GS, p.S, (const uint16_t*)(ws + p.o_tc), p.ptile, q, span, counts);
  }
  return last_launch_status();
}

// ===========================================================================
// LSD radix sort of uint64 keys (used for the learned map's key sample):
// eight stable passes of the same histogram -> scan -> stable tile partition
// pipeline, with the "bucket" of a key being one of its bytes.
// ===========================================================================
struct RadixByteMap {
  static constexpr bool kNeedsPos = false;
  static constexpr bool kSkewed = false;
  static constexpr size_t kStageBytes = 0;
  uint32_t shift;
  __device__ __forceinline__ void init() {}
  __device__ __forceinline__ void stage(uint8_t*, size_t) {}
  template <typename K>
  __device__ __forceinline__ uint32_t operator()(K key, uint32_t /*pos*/ = 0) const {
    return (uint32_t)(((uint64_t)key >> shift) & 255u);
  }
  __device__ __forceinline__ uint32_t out_id(uint32_t id) const { return id; }
};

static void radix_layout(uint64_t n, uint64_t* chunk, uint32_t* G, size_t* o) {
  const int sms = std::max(dev_info().sms, 1);
  uint64_t c = std::max<uint64_t>(kPartTile, (n + 2 * sms - 1) / (2 * sms));
  c = (c + 15) / 16 * 16;
  *chunk = c;
  *G = (uint32_t)std::max<uint64_t>(1, (n + c - 1) / c);
  size_t off = sizeof(WsHeader);
  o[0] = off; off = align_up(off + (size_t)*G * 256 * 4);  // H
  o[1] = off; off = align_up(off + (size_t)*G * 256 * 4);  // C
  o[2] = off; off = align_up(off + 256 * 4);               // column totals
  o[3] = off; off = align_up(off + 257 * 4);               // digit starts
  o[4] = off; off = align_up(off + 256 * 4 + 16);          // unused list + scratch word
  o[5] = off; off = align_up(off + (n + 16) * 8);          // ping-pong keys
  o[6] = off; off = align_up(off + (n + 16) * 4);          // payload (positions, unused)
  o[7] = off;
}

size_t radix_sort_workspace_bytes(uint64_t n) {
  uint64_t chunk;
  uint32_t G;
  size_t o[8];
  radix_layout(n, &chunk, &G, o);
  return o[7];
}

hg_status radix_sort_u64(uint64_t* keys, uint64_t n, uint8_t* ws, cudaStream_t st) {
  if (n <= 1) return HG_OK;
  uint64_t chunk;
  uint32_t G;
  size_t o[8];
  radix_layout(n, &chunk, &G, o);
  WsHeader* hdr = (WsHeader*)ws;
  uint32_t* H = (uint32_t*)(ws + o[0]);
  uint32_t* C = (uint32_t*)(ws + o[1]);
  uint32_t* CT = (uint32_t*)(ws + o[2]);
  uint32_t* BS = (uint32_t*)(ws + o[3]);
  uint32_t* ovf = (uint32_t*)(ws + o[4]);
  uint64_t* tmp = (uint64_t*)(ws + o[5]);
  uint32_t* ids = (uint32_t*)(ws + o[6]);
  uint64_t* src = keys;
  uint64_t* dst = tmp;
  const size_t psm = part_smem_bytes(8, false, part_ipt_keys<uint64_t>(), false, kPartNW);
  auto kp = k_partition<uint64_t, RadixByteMap, false, part_ipt_keys<uint64_t>(), kPartNW, part_minb_keys<uint64_t>()>;
  set_smem_once(kp, psm);
  auto kh = k_hist<uint64_t, RadixByteMap>;
  const size_t hsm = hist_stage_offset(256);
  set_smem_once(kh, hsm);
  for (uint32_t pass = 0; pass < 8; ++pass) {
    RadixByteMap map{8 * pass};
    {
      HG_TRACE("k_radix_hist", st);
      kh<<<G, kHistThreads, hsm, st>>>(src, n, chunk, 0, 256, 0, 256, H, C, map, 0u, nullptr);
    }
    {
      HG_TRACE("k_radix_scan", st);
      colscan_launch(C, G, 256, CT, st);
      k_scan_bins<<<1, 1024, 0, st>>>(CT, 256, BS, 0xffffffffu, ovf, &hdr->ovf_count, ovf + 256, 0, (uint32_t)n,
                                      HugeArgs{}, nullptr);
    }
    PartArgs<uint64_t> pa{};
    pa.in_k = src;
    pa.in_i = nullptr;
    pa.out_k = dst;
    pa.out_i = ids;
    pa.n = n;
    pa.chunk = chunk;
    pa.G = G;
    pa.s = 0;
    pa.sshift = 0;
    pa.nbins = 256;
    pa.nsb = 256;
    pa.H = H;
    pa.C = C;
    pa.CT = CT;
    pa.BS = BS;
    pa.status = &hdr->status;
    {
      HG_TRACE("k_radix_partition", st);
      kp<<<G, kPartNW * 32, psm, st>>>(pa, map);
    }
    uint64_t* t = src;
    src = dst;
    dst = t;
  }
  return last_launch_status();  // eight passes: the result is back in keys
}

// Explicit instantiations used by hg_api.cu (build entry point).
#define HG_INST(K, M)                                                                                   \
  template hg_status build_v2<K, M>(const Plan&, const K*, const uint32_t*, uint32_t*, K*, uint32_t*, \
                                    uint8_t*, cudaStream_t, M, uint32_t, bool);                         \
  template hg_status build_slabs<K, M>(const hg_config*, const SlabPlan&, const K*, const uint32_t*,  \
                                       uint32_t*, K*, uint32_t*, uint8_t*, cudaStream_t, M);            \
  template hg_status build_v1<K, M>(uint64_t, uint64_t, const K*, const uint32_t*, uint32_t*, K*,       \
                                    uint32_t*, uint8_t*, cudaStream_t, M);                              \
  template hg_status probe_slabs<K, M>(const hg_config*, const SlabProbePlan&, const hg_table*, const K*,  \
                                       uint64_t, uint32_t*, uint8_t*, cudaStream_t, M);                   \
  template hg_status probe_binned_impl<K, M>(const ProbePlan&, uint64_t, const hg_table*, const K*,     \
                                             uint64_t, uint32_t*, uint8_t*, cudaStream_t, M);
HG_INST(uint32_t, MurmurMap<true>)
HG_INST(uint64_t, MurmurMap<true>)
HG_INST(uint32_t, MurmurMap<false>)
HG_INST(uint64_t, MurmurMap<false>)
HG_INST(uint32_t, LearnedMap)
HG_INST(uint64_t, LearnedMap)
#undef HG_INST
// batched tables: V2 build and binned probe only (the map needs positions)
template hg_status build_v2<uint32_t, BatchedMap>(const Plan&, const uint32_t*, const uint32_t*, uint32_t*,
                                                  uint32_t*, uint32_t*, uint8_t*, cudaStream_t, BatchedMap,
                                                  uint32_t, bool);
template hg_status probe_binned_impl<uint32_t, BatchedMap>(const ProbePlan&, uint64_t, const hg_table*,
                                                           const uint32_t*, uint64_t, uint32_t*, uint8_t*,
                                                           cudaStream_t, BatchedMap);

}  // namespace hg
