// Top-k compressor of Algorithm 2 (Section 2.4, Theorem 1), worker and server.
//
// Worker: keep the k entries of p = fl(fl(eta*g) + e) with the largest |p_j|
// (ties to the lower index), send them as (u32 index, f32 value) records in
// ascending index order, and keep e_j = p_j - p_j (+0) at the kept entries
// and e_j = p_j elsewhere.  |p_j| is ordered by its bit pattern with the sign
// cleared (a 31-bit key), so the k-th largest key T is found by counting,
// without sorting.
//
// Small problems (chip_ctas): one kernel, 1, 8 or 16 CTAs per worker that keep
// p on chip.  Large ones: five kernels (three where the candidates are few enough
// for one launch to do steps 3 to 5, topk_pick_kernel), one pass over the dense
// vectors:
//   1. sample (16 blocks per worker): p at 65,536 elements spread over the
//      vector; tau, a key that rather more than k of the d keys reach (1.3 k
//      for k = d / 100), is read off their ranks.
//   2. form (tiles of 4096 elements): p, h (optional), and the tile's
//      candidates -- the elements whose key is at least tau -- written in
//      index order to the tile's slot, with the tile's count.  e is written
//      as if every candidate were kept.
//   3. count: the candidates in 2048 bins relative to tau.
//   4. resolve: the counts give T's bin; the keys in the bin are counted one
//      by one and listed, those above it per group of tiles.
//   5. emit: T and the number of keys equal to T that are kept (the lowest
//      indices), the groups' places among the records, and the kept records,
//      at (number of keys > T before it) + min(number of keys == T before it,
//      the number kept); a candidate that is not kept gets its e_j = p_j (and
//      h_j) back.
// With k candidates or more T >= tau, so every key >= T was a candidate and T
// is exact.  With fewer, either p has fewer than k non-zero entries (tau is
// then 1 and they are the candidates: T is 0, and the first zeros fill the
// records), or the sample sat where p is larger than elsewhere: then every
// element becomes a candidate.  tau only decides how much work the first pass
// saves; the result is the same bit for bit.  Nothing carries over from call
// to call.
//   Sparse gradients are ordinary input (frozen layers, rows nobody looked
// up).  With tau = 0 for them and one CTA per worker for what the list does not
// hold, 3.6M x 8, k = d / 100, k / 2 non-zero entries took 9.6 ms, 1.1 k 199 us;
// now 135 and 73 (25M x 16: 64.8 ms and 2.19 ms; now 794 and 777 us).
//
// Server: w_j -= (sum over workers of the value recorded for j, absent
// workers as +0, in the library's pairwise order) / M at the indices some
// worker sent; elsewhere the sum is +0 and w is unchanged.  Where the records
// are dense enough (tile_server), a first kernel finds where each worker's
// records of each tile of indices start, a CTA per tile merges the workers'
// records of it in shared memory, and tiles with very many are shared out in
// parts by a third kernel.  Sparse records of up to 64
// workers: one thread per record in two launches, which scatter the values
// into a table and set the worker's bit in a per-index mask, then let the
// lowest worker of each index sum the index's values and update w_j.  Above
// 64 workers one thread per record searches the other workers' records of its
// tile.
#include <atomic>
#include <cmath>
#include <cstdlib>

#include <cooperative_groups.h>

#include "device_common.cuh"
#include "internal.cuh"

namespace dq {
namespace {

namespace cg = cooperative_groups;

constexpr int kTile = 4096;                                   // elements per tile
constexpr int kFormThreads = 256;                             // threads of a form block
constexpr int kFormRows = kTile / (4 * kFormThreads);         // float4 rows per form thread
constexpr int kSelThreads = 512;                              // threads of a select CTA
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kFineShift = 12, kFineBins = 1792;              // bins of 4096 keys from tau up (7/8 of a binade)
constexpr int kBins = kFineBins + 256;                        // first round: then one bin per exponent
constexpr int kBins2 = 1 << kFineShift;                       // second round
constexpr int kMaxGroups = 8192;                              // groups of tiles per worker, at most
constexpr int kChipThreads = 1024;                            // CTAs that keep their part of p on chip
constexpr int kGroup = 64;                                    // bins per coarse count
constexpr int kChipMax = 49152;                               // parameters of a part, at most
constexpr int kStateWords = 64;
constexpr int kFirst = 4, kBatch = 8;                         // rows of 32 candidates a warp loads at once
constexpr int kSampBlocks = 16;                               // sample blocks per worker
constexpr int kSampThreads = 256;
constexpr int kSampRuns = 8192;                               // sampled runs of 8 elements
constexpr int kSamples = 8 * kSampRuns;
constexpr int kSampBits = 14;                                 // key bits a block's estimate is resolved to
constexpr int kSrvTile = 256;                                 // indices per server tile
constexpr int kSrvThreads = 256;

// State words of a scratch row: the sample blocks' estimates of tau, then
// what one step of a call leaves for the next.
enum : int {
  ST_TAU = 0,
  ST_LISTED = kSampBlocks,    // keys of T's bin put into the list so far
  ST_ROUTE,                   // how step 5 goes on
  ST_BIN,                     // T's first-round bin
  ST_REST                     // k less the keys above it (ROUTE_ZERO: less the candidates)
};
enum : uint32_t {
  ROUTE_LIST = 0,   // T's bin is listed: every CTA finds T by itself
  ROUTE_BIN = 1,    // it holds too many keys: a cluster reads the candidates again
  ROUTE_SHORT = 2,  // there were too few candidates: every element is one now
  ROUTE_ZERO = 3    // the candidates are all non-zero keys, and fewer than k: T is 0
};

__host__ __device__ constexpr int64_t tiles_of(int64_t d) { return (d + kTile - 1) / kTile; }
__host__ __device__ constexpr int64_t round64(int64_t x) { return (x + 63) / 64 * 64; }

// Keys of T's bin a row lists: far more than it holds unless very many keys
// are nearly equal (about 0.0005 k ln-slopes of the distribution at T).
__host__ __device__ constexpr uint32_t list_cap(int64_t d) { return (uint32_t)(8192 + d / 128); }

// Steps 3 to 5 take a worker's tiles in at most kMaxGroups groups of 2^shift
// consecutive ones (one tile each up to d = 2^25).
__host__ __device__ constexpr int group_shift(int64_t d) {
  int s = 0;
  while (((tiles_of(d) - 1) >> s) + 1 > kMaxGroups) ++s;
  return s;
}
__host__ __device__ constexpr int groups_of(int64_t d) { return (int)(((tiles_of(d) - 1) >> group_shift(d)) + 1); }

// Per-worker scratch, in u32 words: state | first- and second-round counts |
// tile counts | the groups' counts or places (uint2) | the list of T's bin
// (uint2) | candidate slots (kTile uint2 per tile).  Step 1 clears the
// state's counters and the round counts; the rest is rewritten by every call
// before it is read.
constexpr int64_t kHistWords = kBins + kBins2;
__host__ __device__ constexpr int64_t head_words(int64_t d) {
  return kStateWords + kHistWords + round64(tiles_of(d)) + 2 * kMaxGroups + round64(2 * (int64_t)list_cap(d));
}
__host__ __device__ constexpr int64_t row_words(int64_t d) { return head_words(d) + 2 * tiles_of(d) * kTile; }
__host__ __device__ constexpr int64_t srv_tiles(int64_t d) { return (d + kSrvTile - 1) / kSrvTile; }

struct RowScratch {
  uint32_t* state;
  uint32_t* hist;
  uint32_t* hist2;
  uint32_t* cnt;
  uint2* before;
  uint2* list;
  uint2* cand;
};

__device__ __forceinline__ RowScratch row_scratch(void* base, int64_t d, int row) {
  uint32_t* p = reinterpret_cast<uint32_t*>(base) + (int64_t)row * row_words(d);
  RowScratch r;
  r.state = p;
  r.hist = r.state + kStateWords;
  r.hist2 = r.hist + kBins;
  r.cnt = r.hist2 + kBins2;
  r.before = reinterpret_cast<uint2*>(r.cnt + round64(tiles_of(d)));
  r.list = r.before + kMaxGroups;
  r.cand = reinterpret_cast<uint2*>(p + head_words(d));
  return r;
}

__device__ __forceinline__ uint32_t key_of(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
// tau of the call under way: the mean of the sample blocks' estimates, one to
// a lane (the form kernel has no registers for all of them in every thread);
// 1, every non-zero key, where a block found too few of them for an estimate.
// All lanes of a warp call it together.
__device__ __forceinline__ uint32_t call_tau(const uint32_t* state) {
  static_assert(kSampBlocks == 16 && ST_TAU == 0, "a sixteenth of each");
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t own = lane < (uint32_t)kSampBlocks ? __ldcg(state + lane) : ~0u;
  const uint32_t mean = __reduce_add_sync(kFullMask, lane < (uint32_t)kSampBlocks ? own >> 4 : 0u);
  return __any_sync(kFullMask, own == 0u) ? 1u : mean;
}
__device__ __forceinline__ uint32_t key_bits(uint32_t bits) { return bits & 0x7FFFFFFFu; }

// Block-wide exclusive scan of one value per thread; *total gets the sum.
// `warp_sums` is shared memory of NT/32 values.  Two barriers.
template <int NT, typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T* total, T* warp_sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const T y = __shfl_up_sync(kFullMask, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  T before = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    const T s = warp_sums[w];
    if (w < warp) before += s;
    sum += s;
  }
  __syncthreads();
  *total = sum;
  return before + x - v;
}

// First-round bin of a candidate: 1792 bins of 4096 keys from tau up, then
// the key's exponent.  The k-th largest key lies within 7/8 of a binade of
// tau unless the sample was far off, so that two rounds give it exactly.
__device__ __forceinline__ uint32_t first_bin(uint32_t key, uint32_t tau) {
  const uint32_t r = key - tau;
  return r < ((uint32_t)kFineBins << kFineShift) ? r >> kFineShift : (uint32_t)kFineBins + (key >> 23);
}

// ---------------------------------------------------------------------------
// 1. tau from a sample.  The vector's whole 8-element runs are cut into
// kSampRuns equal strata, and one run of each is read, at a place in the
// stratum that a multiplicative hash picks (so that no period of the vector
// lines up with the sample).  Block b of a worker takes the strata b, b + 16,
// ... and writes the largest key of kSampBits leading bits that at least
// `rank` of its samples reach.  The caller's rank is a sixteenth of the expected
// one of the k-th largest key, r = k kSamples / d, plus seven standard
// deviations sqrt(r) of a binomial count (2.5, when the eight elements of a
// run are always large together); tau is the mean of the blocks' estimates, which varies
// about as little as one estimate from all samples would, and the blocks need
// not wait for one another.  rank = 0: no sample, tau = 0.  Latency is all
// that counts here: 8 loads of 16 bytes in flight per thread, then a bisection
// over samples in registers.  The blocks also clear the row's counts.  They
// let the form kernel's blocks be scheduled at once, so that its first wave is
// in place when they end (it still waits for them before it reads anything;
// its loads before the wait instead measured the same: 3.6M x 8 79.9 us
// against 80.3, 25M x 16 822 / 826).
// 16 blocks of 256 threads, with the warps' counts in words of their own, take
// 8.4 us for 8 workers; 8 blocks of 512 with one shared counter took 10.8.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kSampThreads) topk_sample_kernel(const CompressArgs a, uint32_t rank, void* scratch) {
  dq_pdl_enter();
  dq_pdl_release();
  constexpr int kHalves = 2 * kSampRuns / kSampBlocks / kSampThreads;  // half runs (float4) per thread
  constexpr int kWarps = kSampThreads / 32;
  __shared__ __align__(16) uint32_t count[kSampBits][kWarps];
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const float* g = a.g + (int64_t)row * a.g_stride;
  const float* e = a.e + (int64_t)(worker - a.row0) * a.ld;
  const RowScratch rs = row_scratch(scratch, a.d, worker - a.row0);
  for (int i = blockIdx.x * kSampThreads + threadIdx.x; i < kHistWords; i += kSampBlocks * kSampThreads) rs.hist[i] = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) rs.state[ST_LISTED] = 0;
  if (rank == 0) {
    if (threadIdx.x == 0) rs.state[ST_TAU + blockIdx.x] = 0;
    return;
  }
  const int64_t runs = a.d >> 3;  // >= kSampRuns
  float4 gv[kHalves], ev[kHalves];
#pragma unroll
  for (int i = 0; i < kHalves; ++i) {
    const uint32_t s = (uint32_t)(i * (kSampThreads / 2) + (threadIdx.x >> 1)) * kSampBlocks + blockIdx.x;
    const int64_t lo = runs * s / kSampRuns, hi = runs * (s + 1) / kSampRuns;
    const int64_t at = lo + __umulhi(s * 0x9E3779B1u, (uint32_t)(hi - lo));
    const int64_t j = 8 * at + 4 * (threadIdx.x & 1);
    gv[i] = __ldcs(reinterpret_cast<const float4*>(g + j));
    ev[i] = __ldcs(reinterpret_cast<const float4*>(e + j));
  }
  uint32_t key[kHalves][4];
#pragma unroll
  for (int i = 0; i < kHalves; ++i) {
    key[i][0] = key_of(ef_p(a.lr, gv[i].x, ev[i].x));
    key[i][1] = key_of(ef_p(a.lr, gv[i].y, ev[i].y));
    key[i][2] = key_of(ef_p(a.lr, gv[i].z, ev[i].z));
    key[i][3] = key_of(ef_p(a.lr, gv[i].w, ev[i].w));
  }
  uint32_t tau = 0;
#pragma unroll 1
  for (int it = 0; it < kSampBits; ++it) {
    const uint32_t trial = tau | (1u << (30 - it));
    uint32_t n = 0;
#pragma unroll
    for (int i = 0; i < kHalves; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) n += key[i][q] >= trial ? 1u : 0u;
    n = __reduce_add_sync(kFullMask, n);
    if ((threadIdx.x & 31) == 0) count[it][threadIdx.x >> 5] = n;
    __syncthreads();
    n = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) n += count[it][w];
    if (n >= rank) tau = trial;
  }
  if (threadIdx.x == 0) rs.state[ST_TAU + blockIdx.x] = tau;
}

// ---------------------------------------------------------------------------
// 2. p = fl(fl(eta g) + e); e = p, or p - p at a candidate (key >= tau), and
// h = fl(fl(eta g) + e); steps 3 to 5 correct both at the candidates
// that are not kept, a fraction of them.  Element order in a tile: row i,
// thread t, component q is tile offset 4 * (i * 256 + t) + q, so warp w of
// row i covers the 128 consecutive offsets of group g = 8 i + w.  Candidate
// values wait in shared memory (flagged in a bitmask) until the block's one
// barrier; then each warp writes its groups' candidates to the tile's slot
// in index order.  (Adding them to the row's counts here instead of in a
// step of their own took the kernel from 0.74 to 1.6 ms at 16 x 25M, k = d /
// 100: the additions meet in the few cache lines of the bins just above tau.)
// ---------------------------------------------------------------------------
template <bool KEEP_H>
__global__ void __launch_bounds__(kFormThreads, 4) topk_form_kernel(const CompressArgs a, void* scratch) {
  dq_pdl_enter();
  constexpr int kGroups = kTile / 128;
  __shared__ float vstage[kTile];
  __shared__ uint32_t flags[kTile / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const float* g = a.g + (int64_t)row * a.g_stride;
  float* e = a.e + (int64_t)(worker - a.row0) * a.ld;
  float* h = KEEP_H ? a.h + (int64_t)(worker - a.row0) * a.ld : nullptr;
  RowScratch rs = row_scratch(scratch, a.d, worker - a.row0);
  const int64_t tile = blockIdx.x;
  const int64_t tile0 = tile * kTile;
  // the tile's loads on their way before tau's
  float4 gr[kFormRows], er[kFormRows];
#pragma unroll
  for (int i = 0; i < kFormRows; ++i) {
    const int64_t j = tile0 + 4 * (i * kFormThreads + (int)threadIdx.x);
    gr[i] = er[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j + 3 < a.d) {
      gr[i] = __ldcg(reinterpret_cast<const float4*>(g + j));
      er[i] = __ldcg(reinterpret_cast<const float4*>(e + j));
    }
  }
  const uint32_t tau = call_tau(rs.state);
#pragma unroll
  for (int i = 0; i < kFormRows; ++i) {
    const int off = 4 * (i * kFormThreads + (int)threadIdx.x);
    const int64_t j = tile0 + off;
    float v[4], en[4];
    uint32_t bits = 0;
    if (j + 3 < a.d) {
      const float gq[4] = {gr[i].x, gr[i].y, gr[i].z, gr[i].w};
      const float eq[4] = {er[i].x, er[i].y, er[i].z, er[i].w};
      float hv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float s = __fmul_rn(a.lr, gq[q]);
        v[q] = __fadd_rn(s, eq[q]);
        const bool c = key_of(v[q]) >= tau;
        if (c) bits |= 1u << q;
        en[q] = c ? __fsub_rn(v[q], v[q]) : v[q];
        hv[q] = __fadd_rn(s, en[q]);
      }
      __stcs(reinterpret_cast<float4*>(e + j), make_float4(en[0], en[1], en[2], en[3]));
      if constexpr (KEEP_H) __stcs(reinterpret_cast<float4*>(h + j), make_float4(hv[0], hv[1], hv[2], hv[3]));
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        v[q] = 0.f;
        if (j + q < a.d) {
          const float s = __fmul_rn(a.lr, g[j + q]);
          v[q] = __fadd_rn(s, e[j + q]);
          const bool c = key_of(v[q]) >= tau;
          if (c) bits |= 1u << q;
          en[q] = c ? __fsub_rn(v[q], v[q]) : v[q];
          e[j + q] = en[q];
          if constexpr (KEEP_H) h[j + q] = __fadd_rn(s, en[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if ((bits >> q) & 1u) vstage[off + q] = v[q];
    // 8 lanes' 4 flag bits form one 32-bit word of the tile's bitmask
    uint32_t word = bits << (4 * (lane & 7));
    word |= __shfl_xor_sync(kFullMask, word, 1);
    word |= __shfl_xor_sync(kFullMask, word, 2);
    word |= __shfl_xor_sync(kFullMask, word, 4);
    if ((lane & 7) == 0) flags[off >> 5] = word;
  }
  __syncthreads();
  // group offsets: every warp scans the 32 groups' counts (group = lane)
  uint32_t gc = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) gc += __popc(flags[lane * 4 + q]);
  uint32_t incl = gc;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFullMask, incl, o);
    if (lane >= o) incl += y;
  }
  const uint32_t total = __shfl_sync(kFullMask, incl, 31);
  uint2* slot = rs.cand + tile * kTile;
  static_assert(kGroups == kFormRows * (kFormThreads / 32), "one group per warp and row");
#pragma unroll
  for (int i = 0; i < kFormRows; ++i) {
    const int grp = i * (kFormThreads / 32) + warp;
    const uint32_t gbase = __shfl_sync(kFullMask, incl - gc, grp);
    const uint32_t lane_bits = (flags[grp * 4 + (lane >> 3)] >> (4 * (lane & 7))) & 0xFu;
    const uint32_t n = __popc(lane_bits);
    uint32_t x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFullMask, x, o);
      if (lane >= o) x += y;
    }
    uint32_t pos = gbase + x - n;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if ((lane_bits >> q) & 1u) {
        const int off = grp * 128 + lane * 4 + q;
        if (dq_in_bounds(pos < (uint32_t)kTile, a.err))  // a tile holds at most kTile candidates
          slot[pos] = make_uint2((uint32_t)(tile0 + off), __float_as_uint(vstage[off]));
        ++pos;
      }
    }
  }
  if (threadIdx.x == 0) rs.cnt[tile] = total;
}

// ---------------------------------------------------------------------------
// 3-5. Select T over the candidates and write the kept records: three grids of
// a.nworkers rows of CTAs, a warp per group of tiles, groups dealt out over
// the row's warps in turn (so that a stretch of the vector that holds most of
// the candidates is shared by all of them).  What a step has to know of the
// whole worker every CTA works out for itself from the counts of the step
// before, which costs less than a step between them.  (One launch, by a
// cluster of 8 CTAs per worker, is faster while a CTA's share fits on chip:
// topk_pick_kernel.  With 250,000 records of each of 16 workers it took twice as
// long.)
// ---------------------------------------------------------------------------
struct SelectTask {
  const CompressArgs& a;
  RowScratch rs;
  int64_t k;
  int64_t nt;
  int groups, shift;
  float* e;
  float* h;
  const float* g;
  uint2* rec;
  int warp0, nwarps;  // this warp's first group, and the stride
  int rows;           // rows of 32 candidates of a tile worth loading before its count is known
};

// The CTA that is the `slot`-th of `ctas` that share row `row`.
__device__ __forceinline__ SelectTask select_task(const CompressArgs& a, int64_t k, int rows, void* scratch, int row,
                                                  int slot, int ctas, int warps = kSelWarps) {
  const int worker = a.worker0 + row;
  const int64_t at = (int64_t)(worker - a.row0) * a.ld;
  return SelectTask{a, row_scratch(scratch, a.d, worker - a.row0), k, tiles_of(a.d), groups_of(a.d), group_shift(a.d),
                    a.e + at, a.h ? a.h + at : nullptr, a.g + (int64_t)row * a.g_stride,
                    reinterpret_cast<uint2*>(a.msg + (int64_t)row * a.msg_stride),
                    slot * warps + (int)(threadIdx.x >> 5), ctas * warps, rows};
}

// A tile's count and first rows of 32 candidates, loaded together (a slot has
// kTile entries, whatever the count) and ahead of their use.
struct TileAhead {
  uint32_t n;
  uint2 c[kFirst];
};

__device__ __forceinline__ TileAhead load_tile(const SelectTask& s, int64_t t) {
  TileAhead x;
  x.n = 0;
  if (t < s.nt) {
    const uint2* slot = s.rs.cand + t * kTile + (threadIdx.x & 31);
    x.n = __ldcg(s.rs.cnt + t);
#pragma unroll
    for (int u = 0; u < kFirst; ++u) x.c[u] = u < s.rows ? __ldcg(slot + 32 * u) : make_uint2(0u, 0u);
  }
  return x;
}

__device__ __forceinline__ TileAhead load_first(const SelectTask& s) {
  return load_tile(s, (int64_t)s.warp0 << s.shift);
}

// This warp's groups of tiles in turn, each tile's candidates in index order:
// start(group), row(candidate, valid) for rows of 32, finish(group), by the
// whole warp.  `cur` is the first tile; the next one loads while a tile is
// worked on.
template <typename Start, typename Row, typename Finish>
__device__ __forceinline__ void walk(const SelectTask& s, TileAhead cur, Start&& start, Row&& row, Finish&& finish) {
  const int lane = threadIdx.x & 31;
  const int64_t mask = ((int64_t)1 << s.shift) - 1;
  for (int64_t t = (int64_t)s.warp0 << s.shift; t < s.nt;) {
    const int group = (int)(t >> s.shift);
    int64_t next = t + 1;
    const bool ends = (next & mask) == 0 || next >= s.nt;
    if (ends) next = (int64_t)(group + s.nwarps) << s.shift;
    const TileAhead ahead = load_tile(s, next);
    if ((t & mask) == 0) start(group);
#pragma unroll
    for (int u = 0; u < kFirst; ++u)
      if (u < s.rows && 32 * u < cur.n) row(cur.c[u], 32 * u + lane < cur.n);
    const uint2* slot = s.rs.cand + t * kTile + lane;
    for (uint32_t o = 32 * s.rows; o < cur.n; o += 32 * kBatch) {
      uint2 c[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        c[u] = make_uint2(0u, 0u);
        if (o + 32 * u + lane < cur.n) c[u] = __ldcg(slot + o + 32 * u);
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u)
        if (o + 32 * u < cur.n) row(c[u], o + 32 * u + lane < cur.n);
    }
    if (ends) finish(group);
    t = next;
    cur = ahead;
  }
}

constexpr int kOwnList = 512;  // keys of T's bin a CTA collects before it adds them to the row's list

template <int NT>
struct SelectSmem {
  alignas(16) uint32_t hist[kBins2];  // this CTA's counts
  uint64_t scan[NT / 32];
  uint32_t warp_sums[NT / 32];
  uint32_t found[3];
  uint32_t list_at;
  uint32_t listed;
  uint2 list[NT == kSelThreads ? kOwnList : 1];
};

// The bin b of BINS counts with count(> b) < k_rem <= count(>= b), k_rem -
// count(> b) and count(b), in sm.found (as they were when there are fewer).
// Returns the sum of all counts.  load(i): the counts i .. i + 3.
template <int NT, int BINS, typename Load>
__device__ __forceinline__ uint32_t find_bin(SelectSmem<NT>& sm, uint32_t k_rem, Load&& load) {
  constexpr int kPer = BINS / NT;  // bins per thread, from the top down
  static_assert(kPer * NT == BINS && kPer % 4 == 0, "whole bins per thread, four at a time");
  const int first = BINS - ((int)threadIdx.x + 1) * kPer;
  uint32_t cnt[kPer], sum = 0;
#pragma unroll
  for (int q = 0; q < kPer; q += 4) {
    const uint4 x = load(first + q);
    cnt[q] = x.x;
    cnt[q + 1] = x.y;
    cnt[q + 2] = x.z;
    cnt[q + 3] = x.w;
  }
#pragma unroll
  for (int q = 0; q < kPer; ++q) sum += cnt[q];
  uint32_t total;
  uint32_t cum = block_exclusive_scan<NT>(sum, &total, sm.warp_sums);
#pragma unroll
  for (int q = kPer - 1; q >= 0; --q) {
    if (cum < k_rem && k_rem - cum <= cnt[q]) {
      sm.found[0] = (uint32_t)(first + q);
      sm.found[1] = k_rem - cum;
      sm.found[2] = cnt[q];
    }
    cum += cnt[q];
  }
  __syncthreads();
  return total;
}

// Counts that other CTAs' finished grid added to.
struct RowCounts {
  const uint32_t* counts;
  __device__ __forceinline__ uint4 operator()(int i) const {
    return __ldcg(reinterpret_cast<const uint4*>(counts + i));
  }
};
// This CTA's own counts.
struct OwnCounts {
  const uint32_t* counts;
  __device__ __forceinline__ uint4 operator()(int i) const { return *reinterpret_cast<const uint4*>(counts + i); }
};

template <int NT>
__device__ __forceinline__ void clear_hist(SelectSmem<NT>& sm, int bins) {
  for (int i = threadIdx.x; i < bins; i += NT) sm.hist[i] = 0;
  __syncthreads();
}

__device__ __forceinline__ void add_hist(const SelectSmem<kSelThreads>& sm, uint32_t* row_hist, int bins) {
  __syncthreads();
  for (int i = threadIdx.x; i < bins; i += kSelThreads) {
    const uint32_t n = sm.hist[i];
    if (n) atomicAdd(row_hist + i, n);
  }
}

// e_j = p_j (and h_j) again at a candidate that is not kept (p_j = +0: they
// hold it already).
__device__ __forceinline__ void put_back(const SelectTask& s, uint2 c) {
  if (c.y == 0) return;
  const float p = __uint_as_float(c.y);
  s.e[c.x] = p;
  if (s.h) s.h[c.x] = __fadd_rn(__fmul_rn(s.a.lr, s.g[c.x]), p);
}

__device__ __forceinline__ void put_on_list(const SelectTask& s, uint2 x) {
  const uint32_t at = atomicAdd(s.rs.state + ST_LISTED, 1u);
  if (dq_in_bounds(at < list_cap(s.a.d), s.a.err)) s.rs.list[at] = x;
}

// The second round over this task's groups, into sm.hist: the 4096 keys of
// the first round's bin, or (T is far above tau) the next 12 bits of the
// exponent's keys.  Also each group's number of keys above the bin, and
// (`listing`: the first round's count says that they fit) the row's list of
// the keys in it.
__device__ __forceinline__ void count_second(SelectSmem<kSelThreads>& sm, const SelectTask& s, const TileAhead& first,
                                             uint32_t tau, uint32_t bin, bool listing) {
  if (threadIdx.x == 0) sm.listed = 0;
  clear_hist(sm, kBins2);
  const int lane = threadIdx.x & 31;
  const bool fine = bin < (uint32_t)kFineBins;
  uint32_t above = 0, in_group = 0;
  walk(
      s, first, [&](int group) { above = 0, in_group = (uint32_t)group; },
      [&](uint2 c, bool valid) {
        const uint32_t key = key_bits(c.y);
        const uint32_t b = first_bin(key, tau);
        above += valid && b > bin ? 1u : 0u;
        const bool in = valid && b == bin;
        const uint32_t who = __ballot_sync(kFullMask, in);
        if (who) {  // about one candidate in 500
          if (in) atomicAdd(&sm.hist[(fine ? key - tau : key >> 11) & (kBins2 - 1)], 1u);
          if (listing) {
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(&sm.listed, (uint32_t)__popc(who));
            at = __shfl_sync(kFullMask, at, 0) + __popc(who & ((1u << lane) - 1u));
            if (in && at < (uint32_t)kOwnList) sm.list[at] = make_uint2(in_group, key);
            else if (in) put_on_list(s, make_uint2(in_group, key));
          }
        }
      },
      [&](int group) {
        above = __reduce_add_sync(kFullMask, above);
        if (lane == 0) s.rs.before[group] = make_uint2(above, 0u);
      });
  __syncthreads();
  const uint32_t own = min(sm.listed, (uint32_t)kOwnList);
  if (!own) return;
  if (threadIdx.x == 0) sm.list_at = atomicAdd(s.rs.state + ST_LISTED, own);
  __syncthreads();
  const uint32_t cap = list_cap(s.a.d);
  for (uint32_t i = threadIdx.x; i < own; i += kSelThreads)
    if (dq_in_bounds(sm.list_at + i < cap, s.a.err)) s.rs.list[sm.list_at + i] = sm.list[i];
}

__device__ __forceinline__ void count_first(SelectSmem<kSelThreads>& sm, const SelectTask& s, const TileAhead& first,
                                            uint32_t tau) {
  clear_hist(sm, kBins);
  walk(
      s, first, [](int) {},
      [&](uint2 c, bool valid) {
        if (valid) atomicAdd(&sm.hist[first_bin(key_bits(c.y), tau)], 1u);
      },
      [](int) {});
}

// The exclusive prefix of gt[] and eq[] over the groups; an odd number of
// groups per thread keeps the threads' shared-memory accesses on different
// banks.
__device__ __forceinline__ void group_places(SelectSmem<kSelThreads>& sm, int groups, uint32_t* gt, uint32_t* eq) {
  __syncthreads();
  const int per = ((groups + kSelThreads - 1) / kSelThreads) | 1;
  const int i0 = min((int)threadIdx.x * per, groups), i1 = min(i0 + per, groups);
  uint64_t sum = 0, total;  // keys above T | keys equal to T << 32, both below 2^32
  for (int i = i0; i < i1; ++i) sum += (uint64_t)gt[i] | (uint64_t)eq[i] << 32;
  uint64_t p = block_exclusive_scan<kSelThreads>(sum, &total, sm.scan);
  for (int i = i0; i < i1; ++i) {
    const uint64_t v = (uint64_t)gt[i] | (uint64_t)eq[i] << 32;
    gt[i] = (uint32_t)p;
    eq[i] = (uint32_t)(p >> 32);
    p += v;
  }
  __syncthreads();
}

// The records of this task's groups, and e and h at the candidates not kept;
// gt[], eq[]: the numbers of keys above and equal to T before each group.
__device__ __forceinline__ void emit_groups(const SelectTask& s, const TileAhead& first, uint32_t T, uint32_t need,
                                            const uint32_t* gt, const uint32_t* eq) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  uint2 before = make_uint2(0u, 0u);
  walk(
      s, first, [&](int group) { before = make_uint2(gt[group], eq[group]); },
      [&](uint2 c, bool valid) {
        const uint32_t key = key_bits(c.y);
        const uint32_t gts = __ballot_sync(kFullMask, valid && key > T);
        const uint32_t eqs = __ballot_sync(kFullMask, valid && key == T);
        const uint32_t tie = before.y + __popc(eqs & lt);
        if (valid) {
          if (key > T || (key == T && tie < need)) {
            const uint32_t pos = before.x + __popc(gts & lt) + min(tie, need);
            if (dq_in_bounds(pos < (uint64_t)s.k, s.a.err)) s.rec[pos] = c;  // always true; keeps the write inside
          } else {
            put_back(s, c);
          }
        }
        before.x += __popc(gts);
        before.y += __popc(eqs);
      },
      [](int) {});
}

// Every element of the tiles slot, slot + ctas, ... becomes a candidate, as if
// kept (p from e, and from the candidates there were); body(p) for each.
template <int NT, typename Body>
__device__ __forceinline__ void all_as_candidates(const SelectTask& s, int slot, int ctas, Body&& body) {
  for (int64_t t = slot; t < s.nt; t += ctas) {
    const uint32_t m = __ldcg(s.rs.cnt + t);
    uint2* tile = s.rs.cand + t * kTile;
    for (uint32_t i = threadIdx.x; i < m; i += NT) put_back(s, __ldcg(tile + i));
    __syncthreads();
    const int64_t j0 = t * kTile;
    const int n = (int)min64(kTile, s.a.d - j0);
    for (int i = threadIdx.x; i < n; i += NT) {
      const int64_t j = j0 + i;
      const float p = s.e[j], en = __fsub_rn(p, p);
      tile[i] = make_uint2((uint32_t)j, __float_as_uint(p));
      if (__float_as_uint(p) != 0u) {
        s.e[j] = en;
        if (s.h) s.h[j] = __fadd_rn(__fmul_rn(s.a.lr, s.g[j]), en);
      }
      body(p);
    }
    if (threadIdx.x == 0) s.rs.cnt[t] = (uint32_t)n;
  }
}

// 3. First round.
__global__ void __launch_bounds__(kSelThreads, 2) topk_count_kernel(const CompressArgs a, int rows, void* scratch) {
  dq_pdl_enter();
  __shared__ SelectSmem<kSelThreads> sm;
  const SelectTask s = select_task(a, 0, rows, scratch, blockIdx.y, blockIdx.x, gridDim.x);
  count_first(sm, s, load_first(s), call_tau(s.rs.state));
  add_hist(sm, s.rs.hist, kBins);
}

// 4. T's bin from the first-round counts, then the second round.  For a row
// with too few candidates instead: nothing where they are all the non-zero
// keys (T is 0); else every element becomes a candidate (as if kept), and the
// first round is made again over all of them, from 0 up.
__global__ void __launch_bounds__(kSelThreads, 2) topk_resolve_kernel(const CompressArgs a, int64_t k, int rows, void* scratch) {
  dq_pdl_enter();
  __shared__ SelectSmem<kSelThreads> sm;
  const SelectTask s = select_task(a, k, rows, scratch, blockIdx.y, blockIdx.x, gridDim.x);
  const TileAhead first = load_first(s);
  const uint32_t tau = call_tau(s.rs.state);
  const uint32_t n = find_bin<kSelThreads, kBins>(sm, (uint32_t)k, RowCounts{s.rs.hist});
  const bool too_few = (int64_t)n < k;
  const uint32_t bin = sm.found[0], rest = sm.found[1];
  const bool listing = sm.found[2] <= list_cap(a.d);
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    s.rs.state[ST_ROUTE] = too_few ? (tau == 1 ? ROUTE_ZERO : ROUTE_SHORT) : listing ? ROUTE_LIST : ROUTE_BIN;
    s.rs.state[ST_BIN] = bin;
    s.rs.state[ST_REST] = too_few ? (uint32_t)k - n : rest;
  }
  if (!too_few) {
    count_second(sm, s, first, tau, bin, listing);
    add_hist(sm, s.rs.hist2, kBins2);
    return;
  }
  if (tau == 1) return;
  clear_hist(sm, kBins);
  all_as_candidates<kSelThreads>(s, blockIdx.x, gridDim.x,
                                 [&](float p) { atomicAdd(&sm.hist[first_bin(key_of(p), 0)], 1u); });
  add_hist(sm, s.rs.hist2, kBins);
}

// 5. T from the second-round counts, the groups' places from their counts and
// the list, and the records.  Rows whose T is 0 need no counts at all.  Rows
// that take further passes over the candidates (T's bin holds more keys than
// the list: very many equal keys; or the sample was far off) are selected by a
// cluster of CTAs each afterwards, since the others cannot wait for one
// another.  Two: clusters of 4 or 8 made those rows up to 3 times as fast, but
// every call slower, as fewer CTAs fit at once (dcgan-sized, 3.6M x 8, k = d /
// 100: 80 us with 2, 82 with 4 or 8; 25M x 16 826 / 843 / 839).
constexpr int kEmitCluster = 2;

// T's last 11 bits where the second round has not settled them: the keys with
// the leading bits `high`.
__device__ __forceinline__ void third_round_add(uint32_t* hist, uint32_t key, uint32_t high) {
  if ((key >> 11) == high) atomicAdd(hist + (key & 2047u), 1u);
}

// The records of a row with fewer than k non-zero keys, its candidates: all of
// them, and the first `need` zeros in index order (their e = p - p is +0).
// place(group): the numbers of candidates and of zeros before it; shared: kTile
// / 32 words per warp.
template <typename Place>
__device__ __forceinline__ void emit_with_zeros(uint32_t* shared, const SelectTask& s, uint32_t need, Place&& place) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t* const bits = shared + (threadIdx.x >> 5) * (kTile / 32);  // the tile's candidates, a bit each
  auto put = [&](uint32_t pos, uint2 x) {
    if (dq_in_bounds(pos < (uint64_t)s.k, s.a.err)) s.rec[pos] = x;  // always true; keeps the write inside
  };
  for (int group = s.warp0; group < s.groups; group += s.nwarps) {
    const uint2 before = place(group);
    uint32_t above = before.x, zeros = before.y;
    const int64_t t1 = min64(s.nt, (int64_t)(group + 1) << s.shift);
    for (int64_t t = (int64_t)group << s.shift; t < t1; ++t) {
      const uint32_t n = __ldcg(s.rs.cnt + t);
      const uint2* slot = s.rs.cand + t * kTile;
      const int64_t j0 = t * kTile;
      const int size = (int)min64(kTile, s.a.d - j0);
      const bool some = zeros < need;  // of this tile's zeros are kept
      if (some) {
        for (int i = lane; i < kTile / 32; i += 32) bits[i] = 0;
        __syncwarp();
      }
      for (uint32_t o = lane; o < n; o += 32) {
        const uint2 x = __ldcg(slot + o);
        const uint32_t i = x.x - (uint32_t)j0;
        put(above + o + min(zeros + (i - o), need), x);
        if (some && dq_in_bounds(i < (uint32_t)kTile, s.a.err)) atomicOr(bits + (i >> 5), 1u << (i & 31));
      }
      __syncwarp();
      uint32_t at = above, z = zeros;
#pragma unroll 4
      for (int r = 0; some && r < size; r += 32) {
        const int64_t j = j0 + r + lane;
        const uint32_t here = bits[r >> 5];
        const uint32_t none = ~here & (size - r < 32 ? (1u << (size - r)) - 1u : kFullMask);
        const uint32_t tie = z + __popc(none & lt);
        if (((none >> lane) & 1u) && tie < need) {
          put(at + __popc(here & lt) + tie, make_uint2((uint32_t)j, __float_as_uint(s.e[j])));
          s.e[j] = 0.f;
          if (s.h) s.h[j] = __fadd_rn(__fmul_rn(s.a.lr, s.g[j]), 0.f);
        }
        at += __popc(here);
        z += __popc(none);
      }
      __syncwarp();
      above += n;
      zeros += (uint32_t)size - n;
    }
  }
}

// A ROUTE_BIN or ROUTE_SHORT row, by the CTAs of a cluster together.
// (A call, so that its registers are no burden to the rows without it.)
__device__ __noinline__ void select_by_cluster(SelectSmem<kSelThreads>& sm, const CompressArgs& a, int64_t k, int rows,
                                               void* scratch, int row, uint32_t* places) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int lane = threadIdx.x & 31;
  const SelectTask s = select_task(a, k, rows, scratch, row, rank, kEmitCluster);
  auto cluster_counts = [&](int i) {  // of sm.hist
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int r = 0; r < kEmitCluster; ++r) {
      const uint4 y = *cluster.map_shared_rank(reinterpret_cast<const uint4*>(sm.hist + i), r);
      x.x += y.x;
      x.y += y.y;
      x.z += y.z;
      x.w += y.w;
    }
    return x;
  };
  uint32_t tau, bin, rest;
  if (__ldcg(s.rs.state + ST_ROUTE) == ROUTE_SHORT) {
    tau = 0;
    find_bin<kSelThreads, kBins>(sm, (uint32_t)k, RowCounts{s.rs.hist2});
    bin = sm.found[0], rest = sm.found[1];
    count_second(sm, s, load_first(s), tau, bin, false);
    cluster.sync();
    find_bin<kSelThreads, kBins2>(sm, rest, cluster_counts);
  } else {
    tau = call_tau(s.rs.state);
    bin = __ldcg(s.rs.state + ST_BIN), rest = __ldcg(s.rs.state + ST_REST);
    find_bin<kSelThreads, kBins2>(sm, rest, RowCounts{s.rs.hist2});
  }
  const uint32_t digit = sm.found[0];
  uint32_t T = tau + (bin << kFineShift) + digit, need = sm.found[1];
  cluster.sync();
  if (bin >= (uint32_t)kFineBins) {
    const uint32_t high = ((bin - kFineBins) << 12) | digit;
    clear_hist(sm, 2048);
    walk(
        s, load_first(s), [](int) {},
        [&](uint2 c, bool valid) {
          if (valid) third_round_add(sm.hist, key_bits(c.y), high);
        },
        [](int) {});
    cluster.sync();
    find_bin<kSelThreads, 2048>(sm, need, cluster_counts);
    T = (high << 11) | sm.found[0];
    need = sm.found[1];
    cluster.sync();  // nobody leaves, or counts anew, while its counts are read
  }
  uint32_t gt = 0, eq = 0;
  walk(
      s, load_first(s), [&](int) { gt = 0, eq = 0; },
      [&](uint2 c, bool valid) {
        const uint32_t key = key_bits(c.y);
        gt += valid && key > T ? 1u : 0u;
        eq += valid && key == T ? 1u : 0u;
      },
      [&](int group) {
        gt = __reduce_add_sync(kFullMask, gt);
        eq = __reduce_add_sync(kFullMask, eq);
        if (lane == 0) s.rs.before[group] = make_uint2(gt, eq);
      });
  __threadfence();
  cluster.sync();
  for (int i = threadIdx.x; i < s.groups; i += kSelThreads) {
    const uint2 n = __ldcg(s.rs.before + i);
    places[i] = n.x;
    places[s.groups + i] = n.y;
  }
  group_places(sm, s.groups, places, places + s.groups);
  emit_groups(s, load_first(s), T, need, places, places + s.groups);
  __syncthreads();
}

__global__ void __launch_bounds__(kSelThreads, 2)
    topk_emit_kernel(const CompressArgs a, int64_t k, int rows, int ctas, void* scratch) {
  dq_pdl_enter();
  __shared__ SelectSmem<kSelThreads> sm;
  extern __shared__ uint32_t places[];
  const int row = (int)blockIdx.x / ctas;
  if (row < a.nworkers) {
    const SelectTask s = select_task(a, k, rows, scratch, row, (int)blockIdx.x - row * ctas, ctas);
    const TileAhead first = load_first(s);
    const uint32_t listed = s.rs.state[ST_LISTED], route = s.rs.state[ST_ROUTE];
    uint32_t* gt = places;
    uint32_t* eq = places + s.groups;
    if (route == ROUTE_ZERO) {
      for (int i = threadIdx.x; i < s.groups; i += kSelThreads) {
        uint32_t n = 0;
        const int64_t t0 = (int64_t)i << s.shift, t1 = min64(s.nt, (int64_t)(i + 1) << s.shift);
        for (int64_t t = t0; t < t1; ++t) n += __ldcg(s.rs.cnt + t);
        gt[i] = n;
        eq[i] = (uint32_t)(min64(t1 * kTile, a.d) - t0 * kTile) - n;
      }
      group_places(sm, s.groups, gt, eq);
      static_assert(kSelWarps * (kTile / 32) <= kBins2, "bits of a tile per warp");
      emit_with_zeros(sm.hist, s, s.rs.state[ST_REST], [&](int group) { return make_uint2(gt[group], eq[group]); });
    } else if (route == ROUTE_LIST) {
      for (int i = threadIdx.x; i < s.groups; i += kSelThreads) {
        gt[i] = s.rs.before[i].x;
        eq[i] = 0;
      }
      const uint2 early = s.rs.list[threadIdx.x];  // (the list holds at least 8192)
      auto for_listed = [&](auto&& body) {
        for (uint32_t i = threadIdx.x; i < listed; i += kSelThreads)
          body(i < (uint32_t)kSelThreads ? early : s.rs.list[i]);
      };
      find_bin<kSelThreads, kBins2>(sm, s.rs.state[ST_REST], RowCounts{s.rs.hist2});
      const uint32_t bin = s.rs.state[ST_BIN];
      uint32_t T = call_tau(s.rs.state) + (bin << kFineShift) + sm.found[0], need = sm.found[1];
      if (bin >= (uint32_t)kFineBins) {
        const uint32_t high = ((bin - kFineBins) << 12) | sm.found[0];
        __syncthreads();
        clear_hist(sm, 2048);
        for_listed([&](uint2 x) { third_round_add(sm.hist, x.y, high); });
        __syncthreads();
        find_bin<kSelThreads, 2048>(sm, need, OwnCounts{sm.hist});
        T = (high << 11) | sm.found[0];
        need = sm.found[1];
      }
      for_listed([&](uint2 x) {
        if (x.y > T) atomicAdd(gt + x.x, 1u);
        if (x.y == T) atomicAdd(eq + x.x, 1u);
      });
      group_places(sm, s.groups, gt, eq);
      emit_groups(s, first, T, need, gt, eq);
    }
  }
  for (int r = (int)blockIdx.x / kEmitCluster; r < a.nworkers; r += (int)gridDim.x / kEmitCluster) {
    const uint32_t route = __ldcg(row_scratch(scratch, a.d, a.worker0 + r - a.row0).state + ST_ROUTE);
    if (route == ROUTE_BIN || route == ROUTE_SHORT) {
      __syncthreads();
      select_by_cluster(sm, a, k, rows, scratch, r, places);
    }
  }
}

// ---------------------------------------------------------------------------
// The whole step of a worker in one launch, by C CTAs (one cluster) that keep
// p on chip: CTA r has the r-th part of the vector.  The digits of T (11 + 10
// + 10 bits) come from three counting rounds, the cluster's counts read
// through distributed shared memory; then e, h and the records, a warp per
// stretch of consecutive elements.  At these sizes launches and memory
// latency are most of the time.
// ---------------------------------------------------------------------------
struct ChipSmem {
  uint32_t hist[2048 + 1024 + 1024];            // the rounds' counts (read by the cluster)
  uint32_t coarse[(2048 + 1024 + 1024) / kGroup];  // sums of kGroup bins (read by the cluster)
  uint32_t found[3][4];                          // per round: bin, rest of k, lower ranks' keys above the bin and in it
  uint32_t warp_gt[kChipThreads / 32], warp_eq[kChipThreads / 32];
};

// Elements of a CTA's part: a multiple of 4.
__host__ __device__ constexpr int64_t chip_part(int64_t d, int ctas) { return ((d + ctas - 1) / ctas + 3) / 4 * 4; }

// One warp: the bin b of the cluster's summed counts with count(> b) < k_rem
// <= count(>= b): first its group, from every CTA's group sums, then the bin,
// from every CTA's counts of the group.  out: b, k_rem - count(> b), and the
// counts of the CTAs of lower rank in the bins above b and in b.
template <int C, int BINS>
__device__ __forceinline__ void cluster_find(uint32_t* hist, uint32_t* coarse, uint32_t k_rem, int rank, uint32_t* out) {
  constexpr int G = BINS / kGroup;
  static_assert(G <= 32 && kGroup == 64, "a group per lane, two bins per lane");
  cg::cluster_group cluster = cg::this_cluster();
  const int lane = threadIdx.x & 31;
  // the inclusive sums of two values from lane 0 up
  auto scan = [&](uint32_t& x, uint32_t& y) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t a = __shfl_up_sync(kFullMask, x, off), b = __shfl_up_sync(kFullMask, y, off);
      if (lane >= off) {
        x += a;
        y += b;
      }
    }
  };
  uint32_t all = 0, low = 0;  // of group G - 1 - lane
  if (lane < G) {
#pragma unroll
    for (int r = 0; r < C; ++r) {
      const uint32_t* at = coarse + G - 1 - lane;
      const uint32_t x = C == 1 ? *at : *cluster.map_shared_rank(at, r);
      if (r < rank) low += x;
      all += x;
    }
  }
  uint32_t cum = all, cum_low = low;
  scan(cum, cum_low);
  const uint32_t hit = __ballot_sync(kFullMask, cum - all < k_rem && k_rem <= cum);
  const int src = hit ? __ffs(hit) - 1 : 0;
  const uint32_t above = __shfl_sync(kFullMask, cum - all, src), above_low = __shfl_sync(kFullMask, cum_low - low, src);
  // bins 63 - 2 lane (y) and 62 - 2 lane (x) of the group
  const uint32_t bin = (uint32_t)(G - 1 - src) * kGroup + kGroup - 2 - 2 * lane;
  uint2 n = make_uint2(0u, 0u), m = n;
#pragma unroll
  for (int r = 0; r < C; ++r) {
    const uint2* at = reinterpret_cast<const uint2*>(hist + bin);
    const uint2 x = C == 1 ? *at : *cluster.map_shared_rank(at, r);
    if (r < rank) {
      m.x += x.x;
      m.y += x.y;
    }
    n.x += x.x;
    n.y += x.y;
  }
  cum = n.x + n.y;
  cum_low = m.x + m.y;
  scan(cum, cum_low);
  cum += above - n.x - n.y;  // keys above this lane's two bins
  cum_low += above_low - m.x - m.y;
  if (cum < k_rem && k_rem - cum <= n.y) {
    out[0] = bin + 1;
    out[1] = k_rem - cum;
    out[2] = cum_low;
    out[3] = m.y;
  } else if (cum + n.y < k_rem && k_rem - cum - n.y <= n.x) {
    out[0] = bin;
    out[1] = k_rem - cum - n.y;
    out[2] = cum_low + m.y;
    out[3] = m.x;
  }
}

// T, the number of keys equal to it that are kept, and the numbers of keys above
// and equal to T in the CTAs of lower rank, from keys spread over the cluster:
// the top digits' counts are in sm.hist, each_key(body) calls body(key) for this
// CTA's keys.  The caller arrives at a cluster barrier afterwards and waits at it
// before it leaves: until then its counts may be read.
struct Threshold {
  uint32_t T, need, gt_before, eq_before;
};
template <int C, typename EachKey>
__device__ __forceinline__ Threshold cluster_threshold(ChipSmem& sm, uint32_t k, int rank, EachKey&& each_key) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Threshold t{0u, k, 0u, 0u};
#pragma unroll
  for (int round = 0; round < 3; ++round) {
    uint32_t* hist = sm.hist + (round == 0 ? 0 : round == 1 ? 2048 : 3072);
    uint32_t* coarse = sm.coarse + (round == 0 ? 0 : round == 1 ? 2048 : 3072) / kGroup;
    const int low = 20 - 10 * round;  // key bits below this round's digit
    if (round > 0)
      each_key([&](uint32_t key) {
        if ((key >> (low + 10)) == t.T) atomicAdd(&hist[(key >> low) & 1023u], 1u);
      });
    __syncthreads();
    for (int group = warp; group < (round == 0 ? 2048 : 1024) / kGroup; group += kChipThreads / 32) {
      const uint32_t n = __reduce_add_sync(kFullMask, hist[group * kGroup + lane] + hist[group * kGroup + 32 + lane]);
      if (lane == 0) coarse[group] = n;
    }
    if constexpr (C > 1) cg::this_cluster().sync();
    else __syncthreads();
    if (warp == 0) {
      if (round == 0) cluster_find<C, 2048>(hist, coarse, t.need, rank, sm.found[round]);
      else cluster_find<C, 1024>(hist, coarse, t.need, rank, sm.found[round]);
    }
    __syncthreads();
    t.T = round == 0 ? sm.found[0][0] : t.T << 10 | sm.found[round][0];
    t.need = sm.found[round][1];
    t.gt_before += sm.found[round][2];
    t.eq_before = sm.found[round][3];
  }
  return t;
}

template <int C, bool KEEP_H>
__global__ void __launch_bounds__(kChipThreads, 1) topk_chip_kernel(const CompressArgs a, int64_t k) {
  dq_pdl_enter();
  extern __shared__ __align__(16) float p[];
  __shared__ __align__(16) ChipSmem sm;
  constexpr int kWarps = kChipThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = blockIdx.x;
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const int64_t part = chip_part(a.d, C);
  const int64_t first = min64(a.d, part * rank);
  const int d = (int)(min64(a.d, first + part) - first);  // elements of this part
  const float* g = a.g + (int64_t)row * a.g_stride + first;
  float* e = a.e + (int64_t)(worker - a.row0) * a.ld + first;
  float* h = KEEP_H ? a.h + (int64_t)(worker - a.row0) * a.ld + first : nullptr;
  uint2* rec = reinterpret_cast<uint2*>(a.msg + (int64_t)row * a.msg_stride);
  for (int i = threadIdx.x; i < 4096; i += kChipThreads) sm.hist[i] = 0;
  __syncthreads();
  // p, and the counts of its top 11 bits
  constexpr int kLoads = 4;  // loads of 16 bytes of each vector in flight
  for (int j0 = 4 * threadIdx.x; j0 < d; j0 += 4 * kLoads * kChipThreads) {
    float4 gv[kLoads], ev[kLoads];
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int j = j0 + 4 * i * kChipThreads;
      if (j + 3 < d) {
        gv[i] = __ldcs(reinterpret_cast<const float4*>(g + j));
        ev[i] = __ldcs(reinterpret_cast<const float4*>(e + j));
      }
    }
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int j = j0 + 4 * i * kChipThreads;
      float v[4];
      if (j + 3 < d) {
        const float sg[4] = {__fmul_rn(a.lr, gv[i].x), __fmul_rn(a.lr, gv[i].y), __fmul_rn(a.lr, gv[i].z),
                             __fmul_rn(a.lr, gv[i].w)};
        v[0] = __fadd_rn(sg[0], ev[i].x);
        v[1] = __fadd_rn(sg[1], ev[i].y);
        v[2] = __fadd_rn(sg[2], ev[i].z);
        v[3] = __fadd_rn(sg[3], ev[i].w);
        *reinterpret_cast<float4*>(p + j) = make_float4(v[0], v[1], v[2], v[3]);
        if constexpr (KEEP_H)  // as if nothing were kept
          *reinterpret_cast<float4*>(h + j) = make_float4(__fadd_rn(sg[0], v[0]), __fadd_rn(sg[1], v[1]),
                                                          __fadd_rn(sg[2], v[2]), __fadd_rn(sg[3], v[3]));
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (j + q < d) {
            const float sg = __fmul_rn(a.lr, g[j + q]);
            p[j + q] = v[q] = __fadd_rn(sg, e[j + q]);
            if constexpr (KEEP_H) h[j + q] = __fadd_rn(sg, v[q]);
          }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (j + q < d) atomicAdd(&sm.hist[key_of(v[q]) >> 20], 1u);
    }
  }
  const Threshold th = cluster_threshold<C>(sm, (uint32_t)k, rank, [&](auto&& body) {
    for (int j = threadIdx.x; j < d; j += kChipThreads) body(key_of(p[j]));
  });
  const uint32_t T = th.T, need = th.need;
  // every read of another CTA's shared memory is done: no CTA leaves before
  // all have said so
  if constexpr (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  // warp w takes the elements [w, w + 1) * stretch, 32 at a time
  const int stretch = (d + 32 * kWarps - 1) / (32 * kWarps) * 32;
  const int j0 = min(warp * stretch, d), j1 = min(j0 + stretch, d);
  uint32_t gt = 0, eq = 0;
  for (int j = j0 + lane; j < j1; j += 32) {
    const uint32_t key = key_of(p[j]);
    gt += key > T ? 1u : 0u;
    eq += key == T ? 1u : 0u;
  }
  gt = __reduce_add_sync(kFullMask, gt);
  eq = __reduce_add_sync(kFullMask, eq);
  if (lane == 0) {
    sm.warp_gt[warp] = gt;
    sm.warp_eq[warp] = eq;
  }
  __syncthreads();
  gt = th.gt_before + __reduce_add_sync(kFullMask, lane < warp ? sm.warp_gt[lane] : 0u);
  eq = th.eq_before + __reduce_add_sync(kFullMask, lane < warp ? sm.warp_eq[lane] : 0u);
  const uint32_t lt = (1u << lane) - 1u;
  for (int base = j0; base < j1; base += 32) {
    const int j = base + lane;
    const bool valid = j < j1;
    const float v = valid ? p[j] : 0.f;
    const uint32_t key = key_of(v);
    const uint32_t gts = __ballot_sync(kFullMask, valid && key > T);
    const uint32_t eqs = __ballot_sync(kFullMask, valid && key == T);
    const uint32_t tie = eq + __popc(eqs & lt);
    if (valid) {
      const bool kept = key > T || (key == T && tie < need);
      if (kept) {
        const uint32_t pos = gt + __popc(gts & lt) + min(tie, need);
        if (dq_in_bounds(pos < (uint64_t)k, a.err))  // always true; keeps the write inside the message
          rec[pos] = make_uint2((uint32_t)(first + j), __float_as_uint(v));
      }
      const float en = kept ? __fsub_rn(v, v) : v;
      e[j] = en;
      if constexpr (KEEP_H)
        if (kept) h[j] = __fadd_rn(__fmul_rn(a.lr, g[j]), en);
    }
    gt += __popc(gts);
    eq += __popc(eqs);
  }
  if constexpr (C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Steps 3 to 5 in one launch where a worker's candidates fit into the shared
// memory of a cluster (picks): the cluster's CTAs share them evenly, in index
// order, find T as above and write the records.  The three grids read the
// candidates three times, and at these sizes each of them is launch, first loads
// and barriers (3.6M x 8, k = d / 100, fresh gradients, the whole step: 101.5 us with
// three launches, 86.5 so).  What does not fit after all (many
// equal keys) is read from memory again in every round; with fewer than k
// candidates the zeros fill the records, or all elements become candidates.
// ---------------------------------------------------------------------------
constexpr int kPickCtas = 8;
constexpr int kPickTiles = 4096;  // tiles of a worker, at most
constexpr int kPickCap = 14336;   // candidates of a CTA in shared memory
static_assert(kPickCap * sizeof(uint2) + sizeof(ChipSmem) + (kPickTiles + 1 + kChipThreads / 32) * 4 < 227 * 1024, "fits");

__global__ void __launch_bounds__(kChipThreads, 1) topk_pick_kernel(const CompressArgs a, int64_t k, void* scratch) {
  dq_pdl_enter();
  extern __shared__ __align__(16) uint2 cand[];  // this CTA's first kPickCap candidates
  __shared__ __align__(16) ChipSmem sm;
  __shared__ uint32_t pre[kPickTiles + 1];       // candidates before each tile
  __shared__ uint32_t scan[kChipThreads / 32];
  constexpr int kWarps = kChipThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = blockIdx.x;
  const SelectTask s = select_task(a, k, 0, scratch, blockIdx.y, rank, kPickCtas, kWarps);
  const int nt = (int)s.nt;
  // the tiles' places
  auto place_tiles = [&]() -> uint32_t {
    constexpr int kPer = kPickTiles / kChipThreads;
    uint32_t c[kPer], sum = 0, total;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int t = (int)threadIdx.x * kPer + q;
      c[q] = t < nt ? __ldcg(s.rs.cnt + t) : 0u;
      sum += c[q];
    }
    uint32_t at = block_exclusive_scan<kChipThreads>(sum, &total, scan);
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int t = (int)threadIdx.x * kPer + q;
      if (t <= nt) pre[t] = at;
      at += c[q];
    }
    if (threadIdx.x == 0) pre[nt] = total;
    __syncthreads();
    return total;
  };
  const bool zeros_left = call_tau(s.rs.state) == 1u;
  for (int i = threadIdx.x; i < 4096; i += kChipThreads) sm.hist[i] = 0;
  uint32_t n = place_tiles();
  if ((int64_t)n < k && zeros_left) {  // the candidates are all non-zero keys: T is 0
    static_assert(kWarps * (kTile / 32) <= 4096, "bits of a tile per warp");
    emit_with_zeros(sm.hist, s, (uint32_t)k - n,
                    [&](int t) { return make_uint2(pre[t], (uint32_t)((int64_t)t * kTile) - pre[t]); });
    return;
  }
  if ((int64_t)n < k) {  // the sample was far off
    cg::this_cluster().sync();  // every CTA has read the counts, and so comes here too, before one changes
    all_as_candidates<kChipThreads>(s, rank, kPickCtas, [](float) {});
    __threadfence();
    cg::this_cluster().sync();
    n = place_tiles();
  }
  const uint32_t lo = (uint32_t)((uint64_t)n * rank / kPickCtas), hi = (uint32_t)((uint64_t)n * (rank + 1) / kPickCtas);
  const int m = (int)(hi - lo);
  // the f-th candidate: of the last tile with no more than f before it
  auto fetch = [&](uint32_t f) -> uint2 {
    int t = 0;
#pragma unroll
    for (int step = kPickTiles / 2; step >= 1; step >>= 1)
      if (t + step < nt && pre[t + step] <= f) t += step;
    return __ldcg(s.rs.cand + (int64_t)t * kTile + (f - pre[t]));
  };
  const int own = min(m, kPickCap);
  constexpr int kLoads = 4;
  for (int i0 = threadIdx.x; i0 < m; i0 += kLoads * kChipThreads) {
    uint2 x[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u)
      if (i0 + u * kChipThreads < m) x[u] = fetch(lo + i0 + u * kChipThreads);
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int i = i0 + u * kChipThreads;
      if (i >= m) continue;
      if (i < own) cand[i] = x[u];
      atomicAdd(&sm.hist[key_bits(x[u].y) >> 20], 1u);
    }
  }
  const Threshold th = cluster_threshold<kPickCtas>(sm, (uint32_t)k, rank, [&](auto&& body) {
    for (int i = threadIdx.x; i < own; i += kChipThreads) body(key_bits(cand[i].y));
    for (int i = own + (int)threadIdx.x; i < m; i += kChipThreads) body(key_bits(fetch(lo + i).y));
  });
  // no CTA leaves before all have read its counts
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  const uint32_t T = th.T, need = th.need;
  // warp w takes the candidates [w, w + 1) * stretch, 32 at a time
  const int stretch = (m + 32 * kWarps - 1) / (32 * kWarps) * 32;
  const int i0 = min(warp * stretch, m), i1 = min(i0 + stretch, m);
  uint32_t gt = 0, eq = 0;
  for (int i = i0 + lane; i < i1; i += 32) {
    const uint32_t key = key_bits(i < own ? cand[i].y : fetch(lo + i).y);
    gt += key > T ? 1u : 0u;
    eq += key == T ? 1u : 0u;
  }
  gt = __reduce_add_sync(kFullMask, gt);
  eq = __reduce_add_sync(kFullMask, eq);
  if (lane == 0) {
    sm.warp_gt[warp] = gt;
    sm.warp_eq[warp] = eq;
  }
  __syncthreads();
  gt = th.gt_before + __reduce_add_sync(kFullMask, lane < warp ? sm.warp_gt[lane] : 0u);
  eq = th.eq_before + __reduce_add_sync(kFullMask, lane < warp ? sm.warp_eq[lane] : 0u);
  const uint32_t lt = (1u << lane) - 1u;
  for (int base = i0; base < i1; base += 32) {
    const int i = base + lane;
    const bool valid = i < i1;
    uint2 c = make_uint2(0u, 0u);
    if (valid) c = i < own ? cand[i] : fetch(lo + i);
    const uint32_t key = key_bits(c.y);
    const uint32_t gts = __ballot_sync(kFullMask, valid && key > T);
    const uint32_t eqs = __ballot_sync(kFullMask, valid && key == T);
    const uint32_t tie = eq + __popc(eqs & lt);
    if (valid) {
      if (key > T || (key == T && tie < need)) {
        const uint32_t pos = gt + __popc(gts & lt) + min(tie, need);
        if (dq_in_bounds(pos < (uint64_t)k, a.err)) s.rec[pos] = c;  // always true; keeps the write inside
      } else {
        put_back(s, c);
      }
    }
    gt += __popc(gts);
    eq += __popc(eqs);
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Server.  starts[m][t] = first record of worker m whose index is in run t
// of kSrvTile indices or later (t in [0, nts]); record r writes the runs
// (run(r-1), run(r)], and the last record also (run(k-1), nts].  A thread takes
// kStartsPer consecutive records (25M x 16, k = d / 100: 22 us with one).
// ---------------------------------------------------------------------------
constexpr int kStartsPer = 4;

__global__ void __launch_bounds__(256) topk_server_starts_kernel(const ServerArgs s, uint32_t* starts, uint32_t* dense) {
  dq_pdl_enter();
  if (dense && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *dense = 0;
  const int m = blockIdx.y;
  const int64_t r0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kStartsPer;
  const int lane = threadIdx.x & 31;
  const int64_t nts = srv_tiles(s.d);
  const uint2* msg = reinterpret_cast<const uint2*>(s.msgs + (int64_t)m * s.msg_stride);
  uint32_t* st = starts + (int64_t)m * (nts + 1);
  // the runs of this thread's records (past the end: the last record's)
  int64_t run[kStartsPer];
  if (r0 + kStartsPer <= s.k) {
    static_assert(kStartsPer == 4, "two loads of two records");
    const uint4 a = __ldg(reinterpret_cast<const uint4*>(msg + r0)), b = __ldg(reinterpret_cast<const uint4*>(msg + r0 + 2));
    run[0] = a.x / kSrvTile;
    run[1] = a.z / kSrvTile;
    run[2] = b.x / kSrvTile;
    run[3] = b.z / kSrvTile;
  } else {
#pragma unroll
    for (int q = 0; q < kStartsPer; ++q) run[q] = msg[min64(r0 + q, s.k - 1)].x / kSrvTile;
  }
#pragma unroll
  for (int q = 0; q < kStartsPer; ++q) run[q] = min64(run[q], nts - 1);
  // the run before this thread's first record
  int64_t prev = __shfl_up_sync(kFullMask, run[kStartsPer - 1], 1);
  if (lane == 0) prev = r0 == 0 ? -1 : min64(msg[min64(r0, s.k) - 1].x / kSrvTile, nts - 1);
#pragma unroll
  for (int q = 0; q < kStartsPer; ++q) {
    // this record fills the runs (prev, run] with its number
    const int64_t r = r0 + q;
    const int64_t t_a = prev + 1, t_b = r < s.k ? run[q] : prev;
    for (int64_t t = t_a; t <= t_b && t < t_a + 32; ++t) st[t] = (uint32_t)r;
    // long stretches without records are written by the whole warp
    uint32_t longs = __ballot_sync(kFullMask, t_b - t_a >= 32);
    while (longs) {
      const int src = __ffs(longs) - 1;
      longs &= longs - 1;
      const int64_t a = __shfl_sync(kFullMask, t_a, src), bnd = __shfl_sync(kFullMask, t_b, src);
      const uint32_t val = (uint32_t)__shfl_sync(kFullMask, r, src);
      for (int64_t t = a + 32 + lane; t <= bnd; t += 32) st[t] = val;
    }
    // after the last record: the runs up to nts point past the end
    const uint32_t last = __ballot_sync(kFullMask, r == s.k - 1);
    if (last) {
      const int64_t a = __shfl_sync(kFullMask, t_b, __ffs(last) - 1) + 1;
      for (int64_t t = a + lane; t <= nts; t += 32) st[t] = (uint32_t)s.k;
    }
    prev = run[q];
  }
}

template <bool POW2>
__device__ __forceinline__ float srv_average(float acc, const ServerArgs& s) {
  if constexpr (POW2) return __fmul_rn(acc, s.inv_M);
  else return __fdiv_rn(acc, (float)s.M);
}

// Server for M <= kSrvMaskMaxM: two launches over the M * k records, with
// two tables in the scratch -- a worker mask per index (u32, u64 above 32
// workers; all zero between calls) and M values per index (never cleared).
//   1. scatter: record (m, r) with index j writes its value to entry (j, m)
//      and sets bit m of j's mask.
//   2. reduce: the record of the lowest worker in j's mask owns j.  It loads j's
//      values 16 bytes at a time where M is a multiple of 4 (one by one, M = 64, d = 100,000, k = d / 10,
//      the same indices: 28 us from warm caches, 15 so) and sums
//      the values of the workers in the mask, in worker order with the
//      absent workers as +0 leaves (the library's pairwise order), updates
//      w_j and clears j's mask.  The other records of j read its mask
//      before or after the owner clears it; either way their own bit is not
//      its lowest, so they do nothing.
// Indices nobody sent have the sum +0 and keep w_j; with store_q the q_hat
// buffer is cleared before the scatter.
// Bound by the tables' scattered sectors.  Consecutive blocks take the same
// stretch of records of the M workers in turn: the records are sorted, so the
// workers' blocks touch the same masks and values about the same time, while
// those are in L2 (worker after worker each swept the whole table through
// DRAM: 25M x 16, k = d / 100, 453 us against 282).
constexpr int kSrvMaskMaxM = 64;

template <typename Mask>
struct SrvTables {
  Mask* mask;   // d masks
  float* vals;  // worker m's value of index j at vals[j * M + m]
};

// Words of a mask: one bit per worker.
__host__ __device__ constexpr int srv_mask_words(int32_t nworkers) { return nworkers <= 32 ? 1 : 2; }

__host__ __device__ constexpr int64_t srv_mask_table_words(int64_t d, int32_t nworkers) {
  return (srv_mask_words(nworkers) + (int64_t)nworkers) * round64(d);
}

template <typename Mask>
inline SrvTables<Mask> srv_tables(void* scratch, int64_t d, int32_t rows) {
  uint32_t* base = reinterpret_cast<uint32_t*>(scratch) + row_words(d) * rows;
  return SrvTables<Mask>{reinterpret_cast<Mask*>(base),
                         reinterpret_cast<float*>(base + sizeof(Mask) / sizeof(uint32_t) * round64(d))};
}

// This thread's record: worker m's r-th.
struct SrvRecord {
  int m;
  int64_t r;
};
__device__ __forceinline__ SrvRecord srv_record(const ServerArgs& s) {
  return SrvRecord{(int)(blockIdx.x % (unsigned)s.M),
                   (int64_t)(blockIdx.x / (unsigned)s.M) * kSrvThreads + threadIdx.x};
}

template <typename Mask>
__global__ void __launch_bounds__(kSrvThreads) topk_server_scatter_kernel(const ServerArgs s, SrvTables<Mask> t) {
  dq_pdl_enter();
  const auto [m, r] = srv_record(s);
  if (r >= s.k) return;
  const uint2 rec = reinterpret_cast<const uint2*>(s.msgs + (int64_t)m * s.msg_stride)[r];
  // records come from the compressor and are below d
  if (!dq_in_bounds((int64_t)rec.x < s.d, s.err)) return;
  t.vals[(int64_t)rec.x * s.M + m] = __uint_as_float(rec.y);
  atomicOr(t.mask + rec.x, (Mask)1 << m);
}

// The sum at an index whose mask of workers is `mask`, by the owner with its
// value v; four(w, x): the values of workers w .. w + 3 (w + 1 for two workers
// in all; of those in the mask, anything for the others).
template <int P, typename Mask, typename Four>
__device__ __forceinline__ float owner_sum(Mask mask, float v, Four&& four) {
  if ((mask & (mask - 1u)) == 0u) return P == 1 ? v : __fadd_rn(v, 0.f);  // one value among +0 leaves
  // the padded tree itself: chunks of C leaves (workers), each summed
  // pairwise from its values (+0 where a worker is absent), then the
  // P / C chunk sums pairwise -- the chunks are the tree's subtrees
  constexpr int C = P < 16 ? P : 16, Q = C < 4 ? C : 4;
  float part[P / C];
#pragma unroll
  for (int c = 0; c < P / C; ++c) {
    const uint32_t bits = (uint32_t)(mask >> (C * c)) & (uint32_t)((1ull << C) - 1ull);
    float x[C];
#pragma unroll
    for (int u = 0; u < C; u += Q) {
      float y[4] = {};
      if ((bits >> u) & ((1u << Q) - 1u)) four(C * c + u, y);
#pragma unroll
      for (int q = 0; q < Q; ++q) x[u + q] = (bits >> (u + q)) & 1u ? y[q] : 0.f;
    }
#pragma unroll
    for (int width = C / 2; width >= 1; width /= 2)
#pragma unroll
      for (int i = 0; i < width; ++i) x[i] = __fadd_rn(x[2 * i], x[2 * i + 1]);
    part[c] = x[0];
  }
#pragma unroll
  for (int width = P / C / 2; width >= 1; width /= 2)
#pragma unroll
    for (int i = 0; i < width; ++i) part[i] = __fadd_rn(part[2 * i], part[2 * i + 1]);
  return part[0];
}

template <typename Mask, bool POW2, int P>
__global__ void __launch_bounds__(kSrvThreads) topk_server_reduce_kernel(const ServerArgs s, SrvTables<Mask> t) {
  dq_pdl_enter();
  const auto [m, r] = srv_record(s);
  if (r >= s.k) return;
  const uint2 rec = reinterpret_cast<const uint2*>(s.msgs + (int64_t)m * s.msg_stride)[r];
  const int64_t j = rec.x;
  if (j >= s.d) return;  // skipped by the scatter (and reported there by the checked build)
  const Mask mask = t.mask[j];
  // the owner: bit m set and no bit below it
  if (!((mask >> m) & 1u) || (mask & (((Mask)1 << m) - 1u))) return;
  const float* vals = t.vals + j * s.M;
  const bool whole = s.M % 4 == 0;  // rows of whole 16-byte words
  const float sum = owner_sum<P>(mask, __uint_as_float(rec.y), [&](int who, float (&x)[4]) {
    if (P >= 4 && whole) {
      const float4 v = *reinterpret_cast<const float4*>(vals + who);
      x[0] = v.x;
      x[1] = v.y;
      x[2] = v.z;
      x[3] = v.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < P && ((mask >> (who + q)) & 1u)) x[q] = vals[who + q];
    }
  });
  s.w[j] = server_out(s, s.w[j], srv_average<POW2>(sum, s));
  t.mask[j] = 0;
}

// Server for dense records (tile_server), M <= kSrvMaskMaxM, in two kernels.
// starts[m][t] tells where worker m's records of each run of kSrvTile indices
// are.
//   merge, a CTA per tile of kMergeRuns runs: up to kMergeCap records go to shared memory,
//     worker after worker, and set their worker's bit in their index's mask;
//     the record of the lowest worker of an index owns it.  A sole worker's
//     record updates w; the indices of several workers get rows of M values in
//     what the list leaves free, as many at a time as fit, which their records
//     fill and their owners sum.  A tile with more records goes on a list.
//   dense, over the list: a zeroed value per worker and index of some runs; the
//     records set theirs and every index sums its column (+0 where nobody sent
//     it, which leaves w as it is).  Records gather where a layer's gradients
//     are large, in a few tiles out of thousands, so those tiles are dealt out
//     in runs to a grid of their own (524,288 x 64, k = d / 10 in a tenth of
//     the vector: 392 us where the merge's CTAs did it themselves, 38 so).
//     An item's parameters and the next one's place in the messages load with
//     its records (25M x 16 in 64 layers, k = d / 100, some 560 dense tiles: 56
//     us one after the other, 37 so).
// Records and touched parameters are all they move, against the tables of the
// two kernels above, whose scattered sectors go through DRAM twice.  Latency
// bounds them: the loads of a thread's 8 records, and of the parameters it
// owns, are in flight together (one after the other: 25M x 16, k = d / 100,
// 143 us, 103 so).
constexpr int kMergeThreads = 256;
constexpr int kMergeCap = 2048;  // records in the list
constexpr int kMergeRuns = 16;   // runs per merge CTA
// Words for the rows of shared indices (what leaves 4 or, above 32 workers, 3
// CTAs per SM).
constexpr int merge_row_words(size_t mask_bytes) { return mask_bytes == 4 ? 2048 : 4096; }

// Shared memory of the merge kernel: the list, the rows, the masks and the rows'
// numbers.
constexpr size_t merge_smem(size_t mask_bytes) {
  return kMergeCap * sizeof(uint2) + merge_row_words(mask_bytes) * sizeof(float) +
         kMergeRuns * kSrvTile * (mask_bytes + sizeof(uint16_t));
}
// Runs of an item of the dense kernel, at most, and its shared memory.
constexpr int dense_runs(int P) { return P >= 32 ? 1 : P >= 4 ? 48 / P : 16; }
constexpr size_t dense_smem(int M, int P) { return (size_t)M * dense_runs(P) * kSrvTile * sizeof(float); }

// Whether these kernels run.  They look at every tile in three launches, so
// they want many records, in a vector of many tiles (us from cold caches, the
// tables' kernels / these; indices spread evenly, gathered in a tenth of the
// vector, the same for all workers):
//   3.6M x 8, 1 %, 288,000 records    27 / 23   14 / 20   16 / 19
//   25M x 4, 0.2 %, 200,000           29 / 45   19 / 36   16 / 49
//   25M x 16, 0.2 %, 800,000          98 / 62   55 / 48   23 / 60
//   3.6M x 32, 1 %, 1,152,000         89 / 53   47 / 23   27 / 37
//   10M x 16, 1 %, 1,600,000         119 / 51   66 / 44   35 / 40
//   25M x 16, 1 %, 4,000,000         282 / 103 155 / 78   74 / 82
//   1.05M x 64, 10 %, 6,710,848      231 / 71  133 / 80   98 / 70
//   25M x 1, 3 %, 750,000             72 / 42   17 / 33   72 / 42
//   10M x 2, 3 %, 600,000             45 / 32   16 / 29   39 / 31
// and from warm ones
//   524,288 x 24, 10 %, 1,258,000     34 / 19   19 / 20   18 / 19
//   524,288 x 48, 10 %, 2,516,000     82 / 29   38 / 45   35 / 29
//   524,288 x 64, 10 %, 3,355,000    111 / 33   50 / 38   48 / 33
// Over 2600 such cases the line below has the least loss on either side of it.
bool tile_server(int64_t d, int64_t k, int nworkers) {
  const double records = (double)k * nworkers, least = d >= 1'000'000 ? 700e3 : 1e6;
  return nworkers <= kSrvMaskMaxM && d >= 500'000 && records >= least && records >= 0.03 * (double)d;
}

// Server scratch of the two kernels, after the starts: the number of tiles on
// the list, then the tiles.
__host__ __device__ constexpr int64_t starts_words(int64_t d, int32_t nworkers) {
  return round64((int64_t)nworkers * (srv_tiles(d) + 1));
}
__host__ __device__ constexpr int64_t dense_list_words(int64_t d) {
  return 64 + round64((srv_tiles(d) + kMergeRuns - 1) / kMergeRuns);
}

template <typename Mask, bool POW2, int P>
__global__ void __launch_bounds__(kMergeThreads, 4)
    topk_server_merge_kernel(const ServerArgs s, const uint32_t* starts, uint32_t* dense) {
  dq_pdl_enter();
  constexpr int kIndices = kMergeRuns * kSrvTile;
  constexpr uint32_t kNone = ~0u;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  uint2* list = reinterpret_cast<uint2*>(tile_smem);             // {index in the tile | worker << 16, value}
  float* rows = reinterpret_cast<float*>(list + kMergeCap);      // M values per row
  Mask* mask = reinterpret_cast<Mask*>(rows + merge_row_words(sizeof(Mask)));
  uint16_t* row_of = reinterpret_cast<uint16_t*>(mask + kIndices);  // of a shared index
  __shared__ uint32_t nshared;
  __shared__ uint32_t first[P];                                  // each worker's first record of the tile
  __shared__ uint32_t off[P + 1];                                // the tile's records of the workers before it
  const int64_t nts = srv_tiles(s.d);
  const int64_t run0 = (int64_t)blockIdx.x * kMergeRuns, run1 = min64(run0 + kMergeRuns, nts);
  const int64_t t0 = run0 * kSrvTile;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    uint32_t before = 0;
    for (int m0 = 0; m0 < s.M; m0 += 32) {
      const int m = m0 + lane;
      uint32_t lo = 0, hi = 0;
      if (m < s.M) {
        lo = (uint32_t)min64(starts[(int64_t)m * (nts + 1) + run0], s.k);
        hi = (uint32_t)min64(starts[(int64_t)m * (nts + 1) + run1], s.k);
      }
      const uint32_t n = hi > lo ? hi - lo : 0u;
      uint32_t x = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFullMask, x, o);
        if (lane >= o) x += y;
      }
      if (m < s.M) {
        first[m] = lo;
        off[m] = before + x - n;
      }
      before += __shfl_sync(kFullMask, x, 31);
    }
    if (lane == 0) off[s.M] = before;
  }
  for (int i = threadIdx.x; i < kIndices; i += kMergeThreads) mask[i] = 0;
  if (threadIdx.x == 0) nshared = 0;
  __syncthreads();
  const uint32_t n = off[s.M];
  if (n == 0) return;
  if (n > (uint32_t)kMergeCap) {
    if (threadIdx.x == 0) dense[64 + atomicAdd(dense, 1u)] = blockIdx.x;
    return;
  }
  // this thread's records, their loads in flight together
  constexpr int kMine = kMergeCap / kMergeThreads;
  uint2 mine[kMine];  // {index, value}, then {index in the tile | worker << 16, value}
  int who[kMine];
#pragma unroll
  for (int u = 0; u < kMine; ++u) {
    const uint32_t f = threadIdx.x + u * kMergeThreads;
    int m = 0;  // the worker: off[m] <= f < off[m + 1]
#pragma unroll
    for (int step = P / 2; step >= 1; step >>= 1)
      if (m + step < s.M && off[m + step] <= f) m += step;
    who[u] = m;
    if (f < n) mine[u] = reinterpret_cast<const uint2*>(s.msgs + (int64_t)m * s.msg_stride)[first[m] + (f - off[m])];
  }
#pragma unroll
  for (int u = 0; u < kMine; ++u) {
    const uint32_t f = threadIdx.x + u * kMergeThreads;
    if (f >= n) {
      mine[u].x = kNone;
      continue;
    }
    // (records come from the compressor: sorted, and below d)
    const int64_t i = (int64_t)mine[u].x - t0;
    const bool here = dq_in_bounds(i >= 0 && i < kIndices && (int64_t)mine[u].x < s.d, s.err);
    mine[u].x = here ? (uint32_t)i | (uint32_t)who[u] << 16 : kNone;
    list[f] = mine[u];
    if (here) atomicOr(mask + i, (Mask)1 << who[u]);
  }
  __syncthreads();
  // sole workers' indices: their parameters in flight together
  float wv[kMine];
#pragma unroll
  for (int u = 0; u < kMine; ++u) {
    if (mine[u].x == kNone) continue;
    const uint32_t i = mine[u].x & 0xFFFFu;
    const int m = (int)(mine[u].x >> 16);
    const Mask bits = mask[i];
    if (bits == (Mask)1 << m) {
      wv[u] = s.w[t0 + i];
    } else {
      if (!(bits & (((Mask)1 << m) - 1u))) row_of[i] = (uint16_t)atomicAdd(&nshared, 1u);  // the lowest worker's
      mine[u].x = kNone;
    }
  }
#pragma unroll
  for (int u = 0; u < kMine; ++u) {
    if (mine[u].x == kNone) continue;
    const float v = __uint_as_float(mine[u].y), sum = P == 1 ? v : __fadd_rn(v, 0.f);  // among +0 leaves
    s.w[t0 + (mine[u].x & 0xFFFFu)] = server_out(s, wv[u], srv_average<POW2>(sum, s));
  }
  __syncthreads();
  const uint32_t at_once = merge_row_words(sizeof(Mask)) / (uint32_t)s.M, shared = nshared;
  for (uint32_t row0 = 0; row0 < shared; row0 += at_once) {
    // body(row, record, index, worker, mask) for the records of these rows
    auto for_shared = [&](auto&& body) {
      for (uint32_t f = threadIdx.x; f < n; f += kMergeThreads) {
        const uint2 e = list[f];
        if (e.x == kNone) continue;
        const uint32_t i = e.x & 0xFFFFu;
        const int m = (int)(e.x >> 16);
        const Mask bits = mask[i];
        if (bits == (Mask)1 << m) continue;
        const uint32_t row = row_of[i] - row0;
        if (row < at_once) body(row, e.y, i, m, bits);
      }
      __syncthreads();
    };
    for_shared([&](uint32_t row, uint32_t v, uint32_t, int m, Mask) { rows[row * s.M + m] = __uint_as_float(v); });
    for_shared([&](uint32_t row, uint32_t v, uint32_t i, int m, Mask bits) {
      if (bits & (((Mask)1 << m) - 1u)) return;
      const float sum = owner_sum<P>(bits, __uint_as_float(v), [&](int who, float (&x)[4]) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < P && who + q < s.M) x[q] = rows[row * s.M + who + q];
      });
      s.w[t0 + i] = server_out(s, s.w[t0 + i], srv_average<POW2>(sum, s));
    });
  }
}

template <bool POW2, int P>
__global__ void __launch_bounds__(kMergeThreads, 4)
    topk_server_dense_kernel(const ServerArgs s, const uint32_t* starts, const uint32_t* dense) {
  dq_pdl_enter();
  extern __shared__ __align__(16) float table[];  // M rows of values
  const int64_t nts = srv_tiles(s.d);
  __shared__ uint32_t first[P], past[P];          // each worker's records of the item
  // warps per worker, or workers per warp; of those so many at a time, and so
  // many rows of 32 records of each, that 8 loads are in flight
  constexpr int kWarps = kMergeThreads / 32, kShare = P < kWarps ? kWarps / P : 1;
  constexpr int kWorkers = P < kWarps ? 1 : P / kWarps, kTake = kWorkers < 4 ? kWorkers : 4, kAhead = 8 / kTake;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // as many runs per item as leave two items to every CTA
  const int64_t tiles = dense[0];
  const int per = (int)max64(1, min64(dense_runs(P), tiles * kMergeRuns / (2 * (int64_t)gridDim.x)));
  const int row = per * kSrvTile;
  const int items_per = (kMergeRuns + per - 1) / per;  // of a tile
  const int64_t items = tiles * items_per;
  // the runs [run0, run1) of an item (empty past the vector's end)
  struct Item {
    int64_t run0, run1;
  };
  auto item_at = [&](int64_t item) {
    const int64_t run0 = (int64_t)dense[64 + item / items_per] * kMergeRuns + (item % items_per) * per;
    const int64_t tile_end = (run0 / kMergeRuns + 1) * kMergeRuns;
    return Item{run0, max64(run0, min64(min64(run0 + per, tile_end), nts))};
  };
  // thread m's share of the next item's table of contents: worker m's records
  uint32_t lo = 0, hi = 0;
  auto load_records = [&](const Item& x) {
    lo = hi = 0;
    if ((int)threadIdx.x >= s.M || x.run0 >= nts) return;
    const uint32_t* st = starts + (int64_t)threadIdx.x * (nts + 1);
    lo = st[x.run0];
    hi = st[x.run1];
  };
  if (blockIdx.x >= items) return;
  Item next = item_at(blockIdx.x);
  load_records(next);
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const Item now = next;
    const int64_t t0 = now.run0 * kSrvTile;
    const int width = (int)max64(0, min64((now.run1 - now.run0) * kSrvTile, s.d - t0));
    if ((int)threadIdx.x < s.M) {
      first[threadIdx.x] = (uint32_t)min64(lo, s.k);
      past[threadIdx.x] = (uint32_t)min64(hi, s.k);
    }
    for (int i = threadIdx.x; i < s.M * (row / 4); i += kMergeThreads)
      reinterpret_cast<float4*>(table)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    // the parameters, and the next item's, on their way with the records
    float wv[dense_runs(P)];
#pragma unroll
    for (int u = 0; u < dense_runs(P); ++u) {
      const int i = threadIdx.x + u * kMergeThreads;
      wv[u] = i < width && !s.store_q ? s.w[t0 + i] : 0.f;
    }
    if (item + gridDim.x < items) {
      next = item_at(item + gridDim.x);
      load_records(next);
    }
#pragma unroll 1
    for (int w0 = 0; w0 < kWorkers; w0 += kTake) {
      // (records come from the compressor: sorted, and below d, so that an item
      // has no more of a worker's than indices)
      uint32_t at[kTake];
      int left[kTake];
      bool more = false;
#pragma unroll
      for (int t = 0; t < kTake; ++t) {
        const int m = warp / kShare + kWarps * (w0 + t), skip = 32 * (warp % kShare) + lane;
        at[t] = 0;
        left[t] = 0;
        if (m < s.M && past[m] > first[m]) {
          at[t] = first[m] + skip;
          left[t] = (int)min(past[m] - first[m], (uint32_t)row) - skip;
        }
        more = more || left[t] > 0;
      }
      while (more) {
        more = false;
        uint2 rec[kTake][kAhead];
#pragma unroll
        for (int t = 0; t < kTake; ++t) {
          const uint2* msg = reinterpret_cast<const uint2*>(
                                 s.msgs + (int64_t)(warp / kShare + kWarps * (w0 + t)) * s.msg_stride) + at[t];
#pragma unroll
          for (int u = 0; u < kAhead; ++u)
            if (32 * kShare * u < left[t]) rec[t][u] = msg[32 * kShare * u];
        }
#pragma unroll
        for (int t = 0; t < kTake; ++t) {
          float* values = table + (warp / kShare + kWarps * (w0 + t)) * row;
#pragma unroll
          for (int u = 0; u < kAhead; ++u)
            if (32 * kShare * u < left[t]) {
              const int64_t i = (int64_t)rec[t][u].x - t0;
              if (dq_in_bounds(i >= 0 && i < width, s.err)) values[i] = __uint_as_float(rec[t][u].y);
            }
          at[t] += 32 * kShare * kAhead;
          left[t] -= 32 * kShare * kAhead;
          more = more || left[t] > 0;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < dense_runs(P); ++w) {
      const int i = threadIdx.x + w * kMergeThreads;
      if (i >= width) break;
      // the padded tree, in chunks of up to 16 workers
      constexpr int C = P < 16 ? P : 16;
      float part_sum[P / C];
#pragma unroll
      for (int c = 0; c < P / C; ++c) {
        float x[C];
#pragma unroll
        for (int u = 0; u < C; ++u) x[u] = C * c + u < s.M ? table[(C * c + u) * row + i] : 0.f;
        part_sum[c] = pairwise_n<C>(x);
      }
      const float sum = pairwise_n<P / C>(part_sum);
      s.w[t0 + i] = server_out(s, wv[w], srv_average<POW2>(sum, s));
    }
    __syncthreads();
  }
}

// One thread per record of every worker.  The record of the lowest worker
// holding index j owns j: it sums the values recorded for j over all M
// workers (absent ones as +0 leaves) in the library's pairwise order and
// applies w_j -= sum / M; the others find an earlier worker holding j and
// stop.  Each search looks only at the other worker's
// records in j's tile of kSrvTile indices (the starts table), and the
// searches in kSrvGroup workers' lists advance in lockstep so that their
// loads are in flight together.
constexpr int kSrvGroup = 8;

template <bool POW2>
__global__ void __launch_bounds__(kSrvThreads) topk_server_owner_kernel(const ServerArgs s, const uint32_t* starts) {
  dq_pdl_enter();
  const int64_t id = (int64_t)blockIdx.x * kSrvThreads + threadIdx.x;
  if (id >= (int64_t)s.M * s.k) return;
  const int m = (int)(id / s.k);
  const int64_t r = id - (int64_t)m * s.k;
  const uint2 mine = reinterpret_cast<const uint2*>(s.msgs + (int64_t)m * s.msg_stride)[r];
  const uint32_t j = mine.x;
  if (!dq_in_bounds((int64_t)j < s.d, s.err)) return;  // records come from the compressor and are < d
  const int64_t nts = srv_tiles(s.d);
  const int64_t t = j / kSrvTile;
  PairwiseAcc<13> sum;  // M <= 4096
  for (int m2 = 0; m2 < m; ++m2) sum.push(0.f);  // no earlier worker holds j (else it owns j)
  sum.push(__uint_as_float(mine.y));
  for (int m0 = 0; m0 < s.M; m0 += kSrvGroup) {
    uint32_t lo[kSrvGroup], hi[kSrvGroup], end[kSrvGroup];
#pragma unroll
    for (int u = 0; u < kSrvGroup; ++u) {
      const int m2 = m0 + u;
      lo[u] = hi[u] = 0;
      if (m2 < s.M && m2 != m) {
        const uint32_t* st = starts + (int64_t)m2 * (nts + 1);
        lo[u] = (uint32_t)min64(st[t], s.k);
        hi[u] = (uint32_t)min64(st[t + 1], s.k);
      }
      end[u] = hi[u];
    }
    // lower bound of j in every range, one halving step for all at a time
    bool active = true;
    while (active) {
      uint32_t x[kSrvGroup];
#pragma unroll
      for (int u = 0; u < kSrvGroup; ++u) {
        x[u] = 0;
        if (lo[u] < hi[u]) {
          const uint2* rec = reinterpret_cast<const uint2*>(s.msgs + (int64_t)(m0 + u) * s.msg_stride);
          x[u] = rec[lo[u] + ((hi[u] - lo[u]) >> 1)].x;
        }
      }
      active = false;
#pragma unroll
      for (int u = 0; u < kSrvGroup; ++u) {
        if (lo[u] < hi[u]) {
          const uint32_t mid = lo[u] + ((hi[u] - lo[u]) >> 1);
          if (x[u] < j) lo[u] = mid + 1;
          else hi[u] = mid;
          active |= lo[u] < hi[u];
        }
      }
    }
    float val[kSrvGroup];
    bool has[kSrvGroup];
#pragma unroll
    for (int u = 0; u < kSrvGroup; ++u) {
      has[u] = false;
      val[u] = 0.f;
      if (lo[u] < end[u]) {
        const uint2* rec = reinterpret_cast<const uint2*>(s.msgs + (int64_t)(m0 + u) * s.msg_stride);
        const uint2 x = rec[lo[u]];
        has[u] = x.x == j;
        val[u] = __uint_as_float(x.y);
      }
    }
#pragma unroll
    for (int u = 0; u < kSrvGroup; ++u) {
      if (has[u] && m0 + u < m) return;  // an earlier worker owns j
      if (m0 + u > m && m0 + u < s.M) sum.push(has[u] ? val[u] : 0.f);
    }
  }
  s.w[j] = __fsub_rn(s.w[j], srv_average<POW2>(sum.result(), s));
}

}  // namespace

size_t topk_scratch_bytes(int64_t d, int64_t k, int32_t rows, int32_t nworkers) {
  // the server's tables: masks and values, or the record starts of every
  // run of kSrvTile indices (dense records; more than kSrvMaskMaxM workers);
  // none for 0
  const int64_t server_words = nworkers <= 0 ? 0
                               : nworkers <= kSrvMaskMaxM && !tile_server(d, k, nworkers)
                                   ? srv_mask_table_words(d, nworkers)
                                   : starts_words(d, nworkers) + dense_list_words(d);
  return (size_t)(row_words(d) * rows + server_words) * 4u;
}

// Rank in a sample block that its estimate of tau has to reach, or 0 where
// every non-zero element is a candidate instead: k is so near d that a sample
// rules nothing out, or the vector is smaller than the sample.
static uint32_t sample_rank(int64_t d, int64_t k) {
  const double expected = (double)k * kSamples / (double)d;
  if (d < kSamples) return 0;
  const double rank = std::ceil((expected + 7.0 * std::sqrt(expected) + 12.0) / kSampBlocks);
  return rank < (double)(kSamples / kSampBlocks) ? (uint32_t)rank : 0u;
}

// CTAs per worker of steps 3 to 5: a warp per group of tiles, but no more
// than two CTAs per SM in all, which fit at once, so that each reads the
// row's counts and clears its own once.
static unsigned select_blocks(int64_t d, int nworkers) {
  const int64_t need = (groups_of(d) + kSelWarps - 1) / kSelWarps;
  const int64_t most = (2 * 152 + nworkers - 1) / nworkers;
  return (unsigned)(need < most ? need : most);
}

// Allows `kernel` its dynamic shared memory beyond 48 KB (and, for clusters of
// more than 8 CTAs, their size).  The attributes belong to the function on the
// current device, so that they were set is remembered per device ordinal.
// Several host threads may race to set them; setting them twice is harmless.
template <typename K>
static cudaError_t allow_smem(K kernel, size_t bytes, int cluster, std::atomic<bool> (&done)[kKeptDevices]) {
  int dev = 0;
  cudaError_t st = cudaGetDevice(&dev);
  if (st != cudaSuccess) return st;
  const bool known = dev >= 0 && dev < kKeptDevices;
  if (known && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
  st = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (st == cudaSuccess && cluster > 8)
    st = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (st == cudaSuccess && known) done[dev].store(true, std::memory_order_release);
  return st;
}

// The kernel that keeps p on chip in C CTAs, and the attributes it needs.
template <int C>
static cudaError_t launch_chip(bool keep_h, const CompressArgs& a, int64_t k, cudaStream_t stream) {
  static std::atomic<bool> done[2][kKeptDevices];
  auto go = [&](auto kernel, std::atomic<bool> (&set)[kKeptDevices]) -> cudaError_t {
    const cudaError_t st = allow_smem(kernel, kChipMax * sizeof(float), C, set);
    if (st != cudaSuccess) return st;
    const size_t need = (size_t)chip_part(a.d, C) * sizeof(float);
    return launch_pdl_cluster(kernel, C, dim3((unsigned)C, (unsigned)a.nworkers), dim3(kChipThreads), need, stream, a, k);
  };
  return keep_h ? go(topk_chip_kernel<C, true>, done[0]) : go(topk_chip_kernel<C, false>, done[1]);
}

// Clusters of C CTAs of `kernel` that fit on the current device at once (for the
// on-chip kernel 152, 15 and 7 of 1, 8 and 16 CTAs on a whole GB300); less, or 0,
// on a part of one, where the launch would fail.  Asked once per device.  (Test
// hook: DQGAN_TEST_NO_CLUSTERS in the environment then makes it 0 for more than
// one CTA.)
template <int C, typename K>
static int resident_clusters(K kernel, size_t smem, std::atomic<bool> (&done)[kKeptDevices],
                             std::atomic<int> (&kept)[kKeptDevices]) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kKeptDevices) return 0;
  int n = kept[dev].load(std::memory_order_acquire);  // plus 1
  if (n == 0) {
    int fit = 0;
    if (C > 1 && std::getenv("DQGAN_TEST_NO_CLUSTERS")) {
      fit = 0;
    } else if (allow_smem(kernel, smem, C, done) == cudaSuccess) {
      if constexpr (C == 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kernel, kChipThreads, smem) != cudaSuccess) fit = 0;
        fit *= device_sms();
      } else {
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(C);
        lc.blockDim = dim3(kChipThreads);
        lc.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = C;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        lc.attrs = &attr;
        lc.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&fit, kernel, &lc) != cudaSuccess) fit = 0;
      }
    }
    cudaGetLastError();  // a form that does not fit is not an error of the call
    n = fit + 1;
    kept[dev].store(n, std::memory_order_release);
  }
  return n - 1;
}

template <int C>
static int chip_resident() {
  static std::atomic<bool> done[kKeptDevices];
  static std::atomic<int> kept[kKeptDevices];
  return resident_clusters<C>(topk_chip_kernel<C, true>, kChipMax * sizeof(float), done, kept);
}

// CTAs per worker of the kernel that keeps p on chip, or 0 where the five
// kernels are taken: the least of the times that fit what was measured (us,
// k = d / 100, d from 4096 to 786,432, 1 to 64 workers).  On chip, a wave of
// as many workers as are resident costs a fixed latency and 0.45 per 1024
// elements of a part; the five kernels cost 20, their memory traffic, and a
// little for every worker's sample.  E.g. one worker, d = 65,536: 9.1 with 16
// CTAs (9.9 with 8, 21 with the five kernels); 16 workers of 65,536: 24 with 8
// CTAs, 31 with 16, 30 with the five; 64 workers of 32,768: 26 with 1, 50 with
// 8.  (Each with its server step.)  Below kSamples the five kernels have no
// sample, every non-zero element is a candidate, and they cost some 50 more.
static int chip_ctas(int64_t d, int nworkers) {
  double best = 20.0 + 2.2e-6 * (double)d * nworkers + 0.15 * nworkers + (d < kSamples ? 50.0 : 0.0);
  int ctas = 0;
  auto consider = [&](int n, int resident, double latency) {
    const int64_t part = chip_part(d, n);
    if (part > kChipMax || resident == 0) return;
    const double t = ((nworkers + resident - 1) / resident) * (latency + 0.45 * (double)part / 1024.0);
    if (t < best) {
      best = t;
      ctas = n;
    }
  };
  consider(1, chip_resident<1>(), 4.0);
  consider(8, chip_resident<8>(), 6.8);
  consider(16, chip_resident<16>(), 7.5);
  return ctas;
}

// Whether the selection is one launch (topk_pick_kernel): the candidates that
// the sample leads one to expect fit on chip, with a tenth to spare, every
// worker's cluster fits the device at once, and they are so few that 8 CTAs per
// worker read them as fast as the grids of the three launches do.  Worker step,
// one launch / three (us, layers of different scale; k: candidates): 600,000 x 1,
// 6000: 18.2 / 21.2; 1M x 1, 10,000: 18.9 / 21.7, 100,000: 33.1 / 40.9; 1M x 8, 10,000:
// 30.9 / 34.6; 1M x 16 (two waves) 57.1 / 54.0; 3.6M x 1, 18,000 (26,000): 24.9 / 25.5,
// 36,000 (46,000): 28.5 / 26.4; 3.6M x 4, 36,000: 47.8 / 48.1; 3.6M x 8, 36,000: 77.0 / 79.9,
// 72,000 (87,000): 84.8 / 84.8; 3.6M x 15, 72,000: 132 / 142; 14M x 2, 28,000: 74.2 / 75.5.
static bool picks(const CompressArgs& a, int64_t k) {
  static std::atomic<bool> done[kKeptDevices];
  static std::atomic<int> kept[kKeptDevices];
  const double candidates = (double)sample_rank(a.d, k) * kSampBlocks * (double)a.d / kSamples;
  const double most = a.d <= 1'200'000 ? kPickCtas * kPickCap / 1.1
                                       : fmin(kPickCtas * kPickCap / 1.1, 25e3 * (1.0 + 0.25 * a.nworkers));
  return candidates > 0 && candidates <= most && tiles_of(a.d) <= kPickTiles &&
         a.nworkers <= resident_clusters<kPickCtas>(topk_pick_kernel, kPickCap * sizeof(uint2), done, kept);
}

cudaError_t launch_topk_compress(const CompressArgs& a, int64_t k, bool keep_h, void* scratch,
                                 cudaStream_t stream, uint64_t* launches) {
  static std::atomic<bool> emit_done[kKeptDevices];
  const unsigned rows = (unsigned)a.nworkers;
  cudaError_t st = cudaSuccess;
  auto launched = [&](cudaError_t r) {
    st = r;
    if (st == cudaSuccess) *launches += 1;
    return st == cudaSuccess;
  };
  switch (chip_ctas(a.d, a.nworkers)) {
    case 1: launched(launch_chip<1>(keep_h, a, k, stream)); return st;
    case 8: launched(launch_chip<8>(keep_h, a, k, stream)); return st;
    case 16: launched(launch_chip<16>(keep_h, a, k, stream)); return st;
  }
  const dim3 tiles((unsigned)tiles_of(a.d), rows), select(select_blocks(a.d, a.nworkers), rows);
  if (picks(a, k)) {
    static std::atomic<bool> pick_done[kKeptDevices];
    constexpr size_t smem = kPickCap * sizeof(uint2);
    if ((st = allow_smem(topk_pick_kernel, smem, kPickCtas, pick_done)) != cudaSuccess) return st;
    (void)(launched(launch_pdl(topk_sample_kernel, dim3(kSampBlocks, rows), dim3(kSampThreads), 0, stream, a,
                               sample_rank(a.d, k), scratch)) &&
           launched(launch_pdl(keep_h ? topk_form_kernel<true> : topk_form_kernel<false>, tiles, dim3(kFormThreads), 0,
                               stream, a, scratch)) &&
           launched(launch_pdl_cluster(topk_pick_kernel, kPickCtas, dim3(kPickCtas, rows), dim3(kChipThreads), smem, stream,
                                       a, k, scratch)));
    return st;
  }
  // the rows that a tile with its share of 1.3 k candidates has
  const int64_t mean = 1 + 13 * k / (320 * tiles_of(a.d));
  const int ahead = (int)(mean < kFirst ? mean : kFirst);
  const size_t places = groups_of(a.d) * 2 * sizeof(uint32_t);
  // (with a cluster for every row that needs one, where they fit at once)
  const unsigned least = kEmitCluster * rows < 2 * 152 ? kEmitCluster * rows : 2 * 152;
  const unsigned emit = ((select.x * rows > least ? select.x * rows : least) + kEmitCluster - 1) / kEmitCluster * kEmitCluster;
  if ((st = allow_smem(topk_emit_kernel, kMaxGroups * 2 * sizeof(uint32_t), 1, emit_done)) != cudaSuccess) return st;
  (void)(launched(launch_pdl(topk_sample_kernel, dim3(kSampBlocks, rows), dim3(kSampThreads), 0, stream, a,
                             sample_rank(a.d, k), scratch)) &&
         launched(launch_pdl(keep_h ? topk_form_kernel<true> : topk_form_kernel<false>, tiles, dim3(kFormThreads), 0,
                             stream, a, scratch)) &&
         launched(launch_pdl(topk_count_kernel, select, dim3(kSelThreads), 0, stream, a, ahead, scratch)) &&
         launched(launch_pdl(topk_resolve_kernel, select, dim3(kSelThreads), 0, stream, a, k, ahead, scratch)) &&
         launched(launch_pdl_cluster(topk_emit_kernel, kEmitCluster, dim3(emit), dim3(kSelThreads), places, stream, a, k,
                                     ahead, (int)select.x, scratch)));
  return st;
}

static cudaError_t launch_tile_server(const ServerArgs& s, const uint32_t* starts, uint32_t* dense, cudaStream_t stream,
                                      uint64_t* launches) {
  const int64_t tiles = (srv_tiles(s.d) + kMergeRuns - 1) / kMergeRuns;
  auto go = [&](auto merge, auto dense_kernel, size_t mask_bytes, int P,
                std::atomic<bool> (&done)[2][kKeptDevices]) -> cudaError_t {
    cudaError_t st = allow_smem(merge, merge_smem(mask_bytes), 1, done[0]);
    if (st == cudaSuccess) st = allow_smem(dense_kernel, dense_smem(P, P), 1, done[1]);
    if (st == cudaSuccess)
      st = launch_pdl(merge, dim3((unsigned)tiles), dim3(kMergeThreads), merge_smem(mask_bytes), stream, s, starts, dense);
    if (st != cudaSuccess) return st;
    *launches += 1;
    const int64_t items = tiles * kMergeRuns, most = 152 * (s.M > 56 ? 3 : 4);  // CTAs that fit at once
    st = launch_pdl(dense_kernel, dim3((unsigned)(items < most ? items : most)), dim3(kMergeThreads), dense_smem(s.M, P),
                    stream, s, starts, (const uint32_t*)dense);
    *launches += st == cudaSuccess ? 1 : 0;
    return st;
  };
  switch (next_pow2(s.M)) {
#define DQ_TILE(P, MASK)                                                                                    \
  case P: {                                                                                                 \
    static std::atomic<bool> done[2][2][kKeptDevices];                                                      \
    return s.M_pow2 ? go(topk_server_merge_kernel<MASK, true, P>, topk_server_dense_kernel<true, P>,        \
                         sizeof(MASK), P, done[0])                                                          \
                    : go(topk_server_merge_kernel<MASK, false, P>, topk_server_dense_kernel<false, P>,      \
                         sizeof(MASK), P, done[1]);                                                         \
  }
    DQ_TILE(1, uint32_t) DQ_TILE(2, uint32_t) DQ_TILE(4, uint32_t) DQ_TILE(8, uint32_t) DQ_TILE(16, uint32_t)
    DQ_TILE(32, uint32_t) DQ_TILE(64, unsigned long long)
#undef DQ_TILE
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_topk_server(const ServerArgs& s, void* scratch, int32_t rows, cudaStream_t stream,
                                uint64_t* launches) {
  if (s.store_q) {  // the dense q_hat buffer: +0 wherever nobody sent an index
    if (s.M > kSrvMaskMaxM) return cudaErrorNotSupported;  // the owner kernel is sparse
    const cudaError_t st = cudaMemsetAsync(s.w, 0, (size_t)s.d * sizeof(float), stream);
    if (st != cudaSuccess) return st;
  }
  uint32_t* starts = reinterpret_cast<uint32_t*>(scratch) + row_words(s.d) * rows;
  const dim3 starts_grid((unsigned)((s.k + 256 * kStartsPer - 1) / (256 * kStartsPer)), (unsigned)s.M);
  if (tile_server(s.d, s.k, s.M)) {
    uint32_t* dense = starts + starts_words(s.d, s.M);
    const cudaError_t st = launch_pdl(topk_server_starts_kernel, starts_grid, dim3(256), 0, stream, s, starts, dense);
    if (st != cudaSuccess) return st;
    *launches += 1;
    return launch_tile_server(s, starts, dense, stream, launches);
  }
  if (s.M <= kSrvMaskMaxM) {
    const dim3 grid((unsigned)((s.k + kSrvThreads - 1) / kSrvThreads * s.M));
    const auto t32 = srv_tables<uint32_t>(scratch, s.d, rows);
    const auto t64 = srv_tables<unsigned long long>(scratch, s.d, rows);
    const bool narrow = srv_mask_words(s.M) == 1;
    cudaError_t st =
        narrow ? launch_pdl(topk_server_scatter_kernel<uint32_t>, grid, dim3(kSrvThreads), 0, stream, s, t32)
               : launch_pdl(topk_server_scatter_kernel<unsigned long long>, grid, dim3(kSrvThreads), 0, stream, s, t64);
    if (st != cudaSuccess) return st;
    auto go = [&](auto kernel, auto t) { return launch_pdl(kernel, grid, dim3(kSrvThreads), 0, stream, s, t); };
    st = cudaErrorInvalidValue;
    switch (next_pow2(s.M)) {
#define DQ_TOPK_REDUCE(P)                                                 \
  case P:                                                                 \
    st = s.M_pow2 ? go(topk_server_reduce_kernel<uint32_t, true, P>, t32) \
                  : go(topk_server_reduce_kernel<uint32_t, false, P>, t32); \
    break;
      DQ_TOPK_REDUCE(1) DQ_TOPK_REDUCE(2) DQ_TOPK_REDUCE(4) DQ_TOPK_REDUCE(8) DQ_TOPK_REDUCE(16)
      DQ_TOPK_REDUCE(32)
#undef DQ_TOPK_REDUCE
      case 64:
        st = s.M_pow2 ? go(topk_server_reduce_kernel<unsigned long long, true, 64>, t64)
                      : go(topk_server_reduce_kernel<unsigned long long, false, 64>, t64);
        break;
    }
    // (a failure here would leave the scatter's mask bits set; the launch has
    // the scatter's grid and block, which were just accepted)
    *launches += st == cudaSuccess ? 2 : 1;
    return st;
  }
  const int64_t n = (int64_t)s.M * s.k;
  launch_pdl(topk_server_starts_kernel, starts_grid, dim3(256), 0, stream, s, starts, (uint32_t*)nullptr);
  const unsigned blocks = (unsigned)((n + kSrvThreads - 1) / kSrvThreads);
  if (s.M_pow2) launch_pdl(topk_server_owner_kernel<true>, dim3(blocks), dim3(kSrvThreads), 0, stream, s, starts);
  else launch_pdl(topk_server_owner_kernel<false>, dim3(blocks), dim3(kSrvThreads), 0, stream, s, starts);
  *launches += 2;
  return cudaGetLastError();
}

}  // namespace dq
