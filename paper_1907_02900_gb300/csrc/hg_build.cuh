// Declarations shared between the build translation unit and the API layer.
#pragma once

#include "hg_device.cuh"

namespace hg {

constexpr int kHistThreads = 1024;
constexpr uint32_t kMaxBinsLog2 = 15;  // bins counted in one shared-memory histogram
constexpr uint32_t kMaxBinShift = 15;  // buckets per bin <= 2^15 (u16 local index, 128 KB cursors)
// Partition geometry.  Stable passes: warps per CTA, items per thread,
// resident CTAs per SM.
constexpr int kPartNW = 16;
template <typename K>
constexpr int part_ipt_keys() {  // pass A: tiles of 8192 4-byte or 2048 8-byte keys
  return sizeof(K) == 8 ? 4 : 16;
}
template <typename K>
constexpr int part_minb_keys() {
  return sizeof(K) == 8 ? 2 : 1;
}
constexpr int kPartIPTB = 6;  // pass B: 256-thread CTAs, up to four per SM
constexpr int kPartNWB = 8;
constexpr int kPartMinBlocksB = 4;
// Passes in any order: threads per CTA, items per thread, resident CTAs per
// SM, by measured sweeps (ms, build and probe of 2^28 uint32 keys, then of
// 2^26 uint64 keys under the learned map).
template <typename K>
struct PartA {  // input positions as ids: tiles of 12288; 20 items 1.02, 28 items 0.98, 2 CTAs of 20 items 1.31 / of 5632
  static constexpr int NT = 512, IPT = sizeof(K) == 8 ? 11 : 24, MINB = sizeof(K) == 8 ? 2 : 1;  // 0.96 / 0.47
};
template <typename K>
struct PartB {  // elements with ids: tiles of 4608 / 4096; 12 items 1.23, 16 items with one CTA 1.24 / 12 items 0.55
  static constexpr int NT = 512, IPT = sizeof(K) == 8 ? 8 : 9, MINB = 2;  // 1.11 / 0.46
};
template <typename K>
struct PartQ {  // queries: tiles of 8192 / 4096 (they divide kQueryBlock); two CTAs of 4096 1.07 / one of 8192 0.51
  static constexpr int NT = 512, IPT = sizeof(K) == 8 ? 8 : 16, MINB = sizeof(K) == 8 ? 2 : 1;  // 0.92 / 0.41
};
constexpr uint32_t kPartPiece = 8;  // pass B: most tiles a CTA takes at a time (1: 1.19 ms, 4: 1.11, 8: 1.08)
constexpr uint32_t kMaxItemsPerCta = 128;  // pass B work items one CTA may own
constexpr uint32_t kMaxBinsPerCta = 512;   // bins one bin-build CTA may own
constexpr int kPartTile = 4096;  // smallest chunk of keys
constexpr int kBinNW = 32;             // warps of the oversized-bin kernels (1024 threads)
constexpr int kBigTile = 2048;         // tile of the oversized-bin kernel
constexpr uint32_t kBinEmaxU32 = 9216;  // largest bin built in shared memory (uint32 keys)
constexpr uint32_t kBinEmaxU64 = 7168;  // same for uint64 keys
constexpr uint32_t kHugeSeg = 1u << 17;  // bins above this many edges are built by several CTAs, one per segment
constexpr uint64_t kHugeMinN = 1ull << 22;  // ... in builds of at least this many keys
constexpr uint32_t kV1Small = 32;      // V1 fix-up: longest bucket sorted by one thread
constexpr int kV1HeavyNW = 16;
constexpr int kV1HeavyIPT = 8;  // V1 fix-up of long buckets: tiles of 4096

// V2 launch plan and workspace layout.
struct Plan {
  int kb;            // key bytes
  uint64_t n, V;
  uint32_t s;        // log2(buckets per bin)
  uint32_t sshift;   // log2(bins per super-bin)
  uint32_t nbins, nsb;
  uint32_t G;        // input chunks of pass A
  uint64_t chunk;    // elements per chunk (multiple of 16)
  uint32_t emax;     // largest bin built in shared memory
  uint32_t tpb;      // threads per bin-build CTA asked for (512 or 1024; 0 = automatic)
  uint32_t max_rows; // segments of huge bins (bins above kHugeSeg edges), upper bound
  size_t o_H, o_C, o_CT, o_T, o_BS, o_ovf, o_hlist, o_rowdesc, o_rowcnt, o_bk, o_bi, total;
};

bool make_plan_v2(const hg_config* cfg, uint64_t n, Plan* p);
// Whether every bin of a uniform spread of the keys is expected to fit the
// shared-memory bin build (mean + 5 standard deviations of a Poisson count).
bool v2_plan_fits(const Plan& p);

// Builds whose buckets need more than 2^15 bins of shared-memory size relabel
// once more (Section 3.3, "Larger Inputs"): a stable partition of the keys by
// slab of 2^Ls buckets, then one two-level build (Alg. 2) per slab into its
// slice of the table.  The slab sizes are read back to the host between the
// two steps (one stream synchronisation).
struct SlabPlan {
  int kb;
  uint64_t n, V;
  uint32_t Ls, S, G;
  uint64_t chunk;
  Plan sub;  // plan of a slab holding all n keys: the bound of every slab build's workspace
  Plan wide;  // the table as one two-level build (total 0: too many bins)
  size_t o_H, o_C, o_CT, o_T, o_BS, o_ovf, o_k, o_i, o_sub, o_wcur, o_wsbs, total;
};
bool make_slab_plan(const hg_config* cfg, uint64_t n, SlabPlan* p);
template <typename K, typename Map>
hg_status build_slabs(const hg_config* cfg, const SlabPlan& p, const K* keys, const uint32_t* ids,
                      uint32_t* offsets, K* csr_k, uint32_t* csr_i, uint8_t* ws, cudaStream_t st, Map map);

// Binned probe: query groups by bucket range, workspace layout.
struct ProbePlan {
  uint32_t sg;   // group = bucket >> sg
  uint32_t ng;   // groups (<= 256)
  uint32_t G;    // query chunks
  uint64_t chunk;
  uint32_t ptile;  // queries per tile of the query partition
  size_t o_H, o_C, o_CT, o_GS, o_ovf, o_qk, o_qi, o_qc, o_tc, total;
};
bool make_probe_plan(const hg_config* cfg, uint64_t table_n, uint64_t q, ProbePlan* p);
// Binned probe of a table of more than 2^kBinnedProbeLog2 buckets: 256 query
// groups would leave each group a table slice too large for L2, so the
// queries are first grouped by slab of 2^kSlabProbeLog2 buckets, each slab's
// queries take the binned probe against the slab's part of the table, and
// the counts are merged back to query order.  The slab query counts are read
// back to the host between the two steps (one stream synchronisation).
// (2^30 queries of 2^31 buckets, slabs of 2^28 / 2^30: 22.9 / 24.7 ms.)
constexpr uint32_t kBinnedProbeLog2 = 30;
constexpr uint32_t kSlabProbeLog2 = 28;
struct SlabProbePlan {
  uint64_t V, q;
  uint32_t Ls, S, G;
  uint64_t chunk;
  uint32_t ptile;
  ProbePlan sub;  // plan of a slab holding all q queries: the bound of every slab probe's workspace
  size_t o_H, o_C, o_CT, o_GS, o_ovf, o_qk, o_qi, o_qc, o_tc, o_sub, total;
};
bool make_slab_probe_plan(const hg_config* cfg, uint64_t table_n, uint64_t q, SlabProbePlan* p);
template <typename K, typename Map>
hg_status probe_slabs(const hg_config* cfg, const SlabProbePlan& p, const hg_table* t, const K* queries,
                      uint64_t q, uint32_t* counts, uint8_t* ws, cudaStream_t st, Map map);
size_t radix_sort_workspace_bytes(uint64_t n);
hg_status radix_sort_u64(uint64_t* keys, uint64_t n, uint8_t* ws, cudaStream_t st);
template <typename K, typename Map>
hg_status probe_binned_impl(const ProbePlan& p, uint64_t V, const hg_table* t, const K* queries, uint64_t q,
                            uint32_t* counts, uint8_t* ws, cudaStream_t st, Map map);
size_t v1_workspace_bytes(int kb, uint64_t n, uint64_t V);

// pos_base is added to every CSR offset written (the position of element 0
// of these CSR arrays inside larger ones; 0 for a standalone table).
// positional_ids: the ids carried are distinct input positions, in input
// order (a slab of a larger build), so the partitions may rank tiles in any
// order, as with implicit ids.
template <typename K, typename Map>
hg_status build_v2(const Plan& p, const K* keys, const uint32_t* ids, uint32_t* offsets, K* csr_k,
                   uint32_t* csr_i, uint8_t* ws, cudaStream_t st, Map map, uint32_t pos_base = 0,
                   bool positional_ids = false);
template <typename K, typename Map>
hg_status build_v1(uint64_t n, uint64_t V, const K* keys, const uint32_t* ids, uint32_t* offsets,
                   K* csr_k, uint32_t* csr_i, uint8_t* ws, cudaStream_t st, Map map);

// Bucket-map construction on the host.
inline MurmurMap<true> make_murmur_pow2(uint32_t seed, uint64_t V) {  // powers of two up to 2^32
  MurmurMap<true> m{};
  m.seed = seed;
  m.mod.mask = (uint32_t)(V - 1);
  return m;
}
inline MurmurMap<false> make_murmur(uint32_t seed, uint64_t V) {  // any other V (< 2^32)
  MurmurMap<false> m{};
  m.seed = seed;
  m.mod.d = (uint32_t)V;
  fastmod_params((uint32_t)V, &m.mod.m, &m.mod.sh1, &m.mod.sh2);
  return m;
}
inline LearnedMap make_learned(const void* blob, uint64_t V) {
  LearnedMap m{};
  m.blob = (const uint8_t*)blob;
  m.Vcap = V;
  return m;
}

// Calls f(K{}, map) with the key type and map the config names.
template <typename F>
hg_status dispatch_key_map(const hg_config* cfg, F&& f) {
  if (cfg->map == HG_MAP_LEARNED) {
    LearnedMap m = make_learned(cfg->d_model, cfg->num_buckets);
    return cfg->key_type == HG_KEY_U64 ? f(uint64_t{}, m) : f(uint32_t{}, m);
  }
  const uint64_t V = cfg->num_buckets;
  if ((V & (V - 1)) == 0) {
    MurmurMap<true> m = make_murmur_pow2(cfg->seed, V);
    return cfg->key_type == HG_KEY_U64 ? f(uint64_t{}, m) : f(uint32_t{}, m);
  }
  MurmurMap<false> m = make_murmur(cfg->seed, V);
  return cfg->key_type == HG_KEY_U64 ? f(uint64_t{}, m) : f(uint32_t{}, m);
}

}  // namespace hg

namespace hg {
size_t join_workspace_bytes(uint64_t nA, uint64_t V);
template <typename K, typename Map>
hg_status join_count_impl(const hg_config* cfg, const hg_table* A, const hg_table* B, int64_t* d_total,
                          int64_t* d_bucket_counts, uint8_t* ws, cudaStream_t st, Map map);
template <typename K, typename Map>
hg_status join_materialize_impl(const hg_config* cfg, const hg_table* A, const hg_table* B, int64_t* outA,
                                int64_t* outB, uint64_t cap, int64_t* d_total, uint8_t* ws, cudaStream_t st,
                                Map map, bool after_count);
}  // namespace hg
