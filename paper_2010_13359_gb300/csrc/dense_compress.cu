// Worker side of Algorithm 2 (DQGAN) for the dense compressors: fused
//   p = fl(fl(eta * g) + e)            error feedback
//   Q(p) and its packed message         scaled sign / b-bit stochastic / identity
//   e = fl(p - Q(p))                    residual, written in place
//   h = fl(fl(eta * g) + e)             lookahead offset (optional)
// in one pass over g and e.
//
// Mapping: a bucket is cut into 4-element chunks; a warp reads rows of 32
// consecutive chunks (512 contiguous bytes) with 128-bit loads and keeps them
// in registers until the bucket's scale is known, so g and e are read once
// and e is written once.  The bucket's l1 sum is taken in the library's fixed
// order: lane l adds the chunk sums ((|a0|+|a1|)+|a2|)+|a3| of chunks
// l, l+32, l+64, ... in increasing order, then five xor-shuffle rounds with
// partners 16, 8, 4, 2, 1 combine the 32 lane totals.  The max-abs scale of
// the stochastic quantiser is exact in any order.
#include <type_traits>

#include "device_common.cuh"

namespace dq {
namespace {

// Loads this thread's CPL chunks c = c0 + 32 i of the bucket [base, end)
// and forms p.  Elements outside the bucket read as 0 and give p = 0.  sg (if
// HOLD) receives fl(eta * g) for the lookahead.
template <int CPL, bool HOLD>
__device__ __forceinline__ void load_and_form(const CompressArgs& a, const float* g, const float* e,
                                              int64_t base, int64_t end, int c0, bool full,
                                              float (&p)[CPL][4], float (&sg)[HOLD ? CPL : 1][4]) {
  const int nchunk = a.bucket >> 2;
  if (full) {
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
      const int c = c0 + 32 * i;
      float4 gv = make_float4(0.f, 0.f, 0.f, 0.f), ev = gv;
      if (c < nchunk) {
        gv = ld_stream4(g + base + 4 * c);
        ev = ld_stream4(e + base + 4 * c);
      }
      const float gq[4] = {gv.x, gv.y, gv.z, gv.w};
      const float eq[4] = {ev.x, ev.y, ev.z, ev.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float s = __fmul_rn(a.lr, gq[q]);
        p[i][q] = (c < nchunk) ? __fadd_rn(s, eq[q]) : 0.f;
        if constexpr (HOLD) sg[i][q] = s;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
      const int c = c0 + 32 * i;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t j = base + 4 * c + q;
        const bool ok = (c < nchunk) && (j < end);
        const float gq = ok ? g[j] : 0.f;
        const float eq = ok ? e[j] : 0.f;
        const float s = __fmul_rn(a.lr, gq);
        p[i][q] = ok ? __fadd_rn(s, eq) : 0.f;
        if constexpr (HOLD) sg[i][q] = s;
      }
    }
  }
}

// Stores the new residual (and lookahead offset) of one chunk.
template <bool KEEP_H, bool HOLD, int CPL>
__device__ __forceinline__ void store_chunk(const CompressArgs& a, const float* g, float* e, float* h,
                                            int64_t j, bool full, int nvalid, const float (&en)[4],
                                            const float (&sg)[HOLD ? CPL : 1][4], int i) {
  if (full) {
    st_stream4(e + j, make_float4(en[0], en[1], en[2], en[3]));
    if constexpr (KEEP_H) {
      float s4[4];
      if constexpr (HOLD) {
#pragma unroll
        for (int q = 0; q < 4; ++q) s4[q] = sg[i][q];
      } else {
        const float4 gv = __ldg(reinterpret_cast<const float4*>(g + j));
        s4[0] = __fmul_rn(a.lr, gv.x);
        s4[1] = __fmul_rn(a.lr, gv.y);
        s4[2] = __fmul_rn(a.lr, gv.z);
        s4[3] = __fmul_rn(a.lr, gv.w);
      }
      st_stream4(h + j, make_float4(__fadd_rn(s4[0], en[0]), __fadd_rn(s4[1], en[1]),
                                    __fadd_rn(s4[2], en[2]), __fadd_rn(s4[3], en[3])));
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (q < nvalid) {
        e[j + q] = en[q];
        if constexpr (KEEP_H) {
          float s;
          if constexpr (HOLD) s = sg[i][q];
          else s = __fmul_rn(a.lr, g[j + q]);
          h[j + q] = __fadd_rn(s, en[q]);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Scaled sign, s_b = ||p_b||_1 / n_b (Section 2.4; error-feedback sign
// compressor of Section 3.1).  Bit = (p < 0); Q(p) = bit ? -s_b : s_b.
//
// WPB warps share a bucket (4 for 4096, 2 for 2048, 1 up to 1024); each
// thread holds CPT chunks in registers.  Warp w of a bucket owns the chunk
// rows w*CPT .. w*CPT+CPT-1 (row r = chunks 32r .. 32r+31, contiguous in
// memory), so lane l holds the chunk sums of positions r of the l1 chain
// "lane l adds chunks l, l+32, l+64, ... in order".  With one warp the chain
// runs in registers; with several, the chunk sums go through shared memory
// and warp 0 runs the chains, so the sum is the same whatever WPB is.
// ---------------------------------------------------------------------------

template <int CPT, int WPB, bool KEEP_H, bool SEG>
__global__ void __launch_bounds__(32 * WPB * (WPB < 4 ? 4 / WPB : 1))
sign_compress_kernel(const CompressArgs a) {
  dq_pdl_enter();
  constexpr bool HOLD = KEEP_H && CPT <= 8;
  constexpr int BPC = WPB < 4 ? 4 / WPB : 1;  // buckets per CTA (CTA = max(4, WPB) warps)
  constexpr int CHAIN = 32 * CPT * WPB;
  __shared__ float chain[WPB > 1 ? BPC * CHAIN : 1];
  __shared__ float scale_sh[BPC];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int slot = warp / WPB;  // bucket within the CTA
  const int wib = warp % WPB;   // warp within the bucket
  const int64_t b = (int64_t)blockIdx.x * BPC + slot;
  const bool valid = b < a.nb;
  if (WPB == 1 && !valid) return;  // no barriers below for a single warp per bucket
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const float* g = a.g + (int64_t)row * a.g_stride;
  float* e = a.e + (int64_t)(worker - a.row0) * a.ld;
  float* h = KEEP_H ? a.h + (int64_t)(worker - a.row0) * a.ld : nullptr;
  uint8_t* msg = a.msg + (int64_t)row * a.msg_stride;

  // flat buckets: [b n, b n + n) clipped to d; layer buckets (SEG): the table
  const int64_t base = SEG ? (valid ? a.bstart[b] : 0) : b * a.bucket;
  const int64_t end = SEG ? (valid ? a.bstart[b + 1] : 0) : a.d;  // elements at or past `end` are not this bucket's
  const int64_t count = SEG ? end - base : (valid ? min64((int64_t)a.bucket, a.d - base) : 0);
  const bool full = (count == a.bucket);
  const int nchunk = a.bucket >> 2;
  const int row0 = wib * CPT;  // first chunk row of this warp

  float p[CPT][4];
  float sg[HOLD ? CPT : 1][4];
  if (valid) {
    load_and_form<CPT, HOLD>(a, g, e, base, end, 32 * row0 + lane, full, p, sg);
  } else {
#pragma unroll
    for (int i = 0; i < CPT; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) p[i][q] = 0.f;
  }

  float s;
  if constexpr (WPB == 1) {
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < CPT; ++i)
      acc = __fadd_rn(acc, __fadd_rn(__fadd_rn(__fadd_rn(fabsf(p[i][0]), fabsf(p[i][1])), fabsf(p[i][2])),
                                     fabsf(p[i][3])));
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(kFullMask, acc, off));
    s = __fdiv_rn(acc, (float)count);
  } else {
    float* ch = chain + slot * CHAIN;
#pragma unroll
    for (int i = 0; i < CPT; ++i)
      ch[(row0 + i) * 32 + lane] =
          __fadd_rn(__fadd_rn(__fadd_rn(fabsf(p[i][0]), fabsf(p[i][1])), fabsf(p[i][2])), fabsf(p[i][3]));
    __syncthreads();
    if (wib == 0) {
      float acc = 0.f;
#pragma unroll 8
      for (int r = 0; r < CPT * WPB; ++r) acc = __fadd_rn(acc, ch[r * 32 + lane]);
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(kFullMask, acc, off));
      if (lane == 0) scale_sh[slot] = valid ? __fdiv_rn(acc, (float)count) : 0.f;
    }
    __syncthreads();
    s = scale_sh[slot];
    if (!valid) return;
  }
  if (wib == 0 && lane == 0) reinterpret_cast<float*>(msg)[b] = s;

  uint32_t* words = reinterpret_cast<uint32_t*>(msg + a.off_payload);
  const int64_t word0 = base >> 5;
  const int64_t word_end = SEG ? (end + 31) >> 5 : (a.d + 31) >> 5;  // buckets start on word boundaries
  const int words_in_bucket = a.bucket >> 5;
#pragma unroll
  for (int i = 0; i < CPT; ++i) {
    const uint32_t wv = pack_sign_row(p[i][0], p[i][1], p[i][2], p[i][3], lane);
    if ((lane & 3) == 0 && lane < 16) {
      const int wib_word = 4 * (row0 + i) + (lane >> 2);
      if (wib_word < words_in_bucket && word0 + wib_word < word_end) words[word0 + wib_word] = wv;
    }
    const int c = 32 * (row0 + i) + lane;
    if (c < nchunk) {
      const int64_t j = base + 4 * c;
      const int nvalid = (int)min64(4, end - j);
      if (nvalid > 0) {
        float en[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) en[q] = __fsub_rn(p[i][q], p[i][q] < 0.f ? -s : s);
        store_chunk<KEEP_H, HOLD, CPT>(a, g, e, h, j, full, nvalid, en, sg, i);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// b-bit stochastic quantiser of Hou et al. (Section 2.4, proof of Theorem 2),
// and QSGD's variant with the l2 scale (Eq. (qsgd)):
// s_b = max |p_j| (or ||p_b||_2), levels B_r = r / K, K = 2^(b-1) - 1; |p_j| K / s_b rounds
// up from r = floor(.) iff u < frac(.), u the 24-bit Philox4x32-10 draw of
// counter (j div 4, worker, step, 0x51) word j mod 4; code = K +- level.
// ---------------------------------------------------------------------------
// Code words of b = 2 and 4 from the chunks' pieces (row i: chunks 32 i + lane,
// 4 b bits each): 8 / b neighbouring lanes' pieces of a row make a word.
// put(i, first, word): the word of row i that starts at lane `first`.  Lanes
// that share words swap pieces so that each ends with whole words of a row of
// its own: one shuffle for two rows (b = 4), two for four (b = 2), instead of
// one or two per row.  (Giving each lane consecutive chunks needs no shuffle,
// but spreads each of a warp's loads over lines 64 bytes apart: b = 4, 512 per
// scale, 25M x 16 took 877 us against 746 so, and 3.6M x 8 with the gradients
// in pinned host memory 1134 against 550.)
template <int BITS, int CPT, typename Put>
__device__ __forceinline__ void pack_rows(const uint32_t (&piece)[CPT], int lane, Put&& put) {
  if constexpr (BITS == 4 && CPT % 2 == 0) {
    const bool odd = lane & 1;
#pragma unroll
    for (int i = 0; i < CPT; i += 2) {
      const uint32_t got = __shfl_xor_sync(kFullMask, odd ? piece[i] : piece[i + 1], 1);
      put(odd ? i + 1 : i, lane & ~1, odd ? got | piece[i + 1] << 16 : piece[i] | got << 16);
    }
  } else if constexpr (BITS == 4) {
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      const uint32_t got = __shfl_xor_sync(kFullMask, piece[i], 1);
      if ((lane & 1) == 0) put(i, lane, piece[i] | got << 16);
    }
  } else if constexpr (BITS == 2 && CPT % 4 == 0) {
    // a 4 x 4 transpose of bytes over 4 lanes: byte r of a lane is its piece
    // of row i + r, and lane q of the four ends with row i + q
    const bool hi2 = lane & 2, hi1 = lane & 1;
#pragma unroll
    for (int i = 0; i < CPT; i += 4) {
      const uint32_t rows01 = piece[i] | piece[i + 1] << 8, rows23 = piece[i + 2] | piece[i + 3] << 8;
      const uint32_t got2 = __shfl_xor_sync(kFullMask, hi2 ? rows01 : rows23, 2);
      // two rows: bytes {row a, row a + 1} of the lower lane, then of the upper
      const uint32_t two = hi2 ? got2 | rows23 << 16 : rows01 | got2 << 16;
      const uint32_t even = __byte_perm(two, 0u, 0x4420), odd = __byte_perm(two, 0u, 0x4431);
      const uint32_t got1 = __shfl_xor_sync(kFullMask, hi1 ? even : odd, 1);
      put(i + (lane & 3), lane & ~3, __byte_perm(hi1 ? got1 : even, hi1 ? odd : got1, 0x5140));
    }
  } else if constexpr (BITS == 2) {
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      uint32_t wv = piece[i] << (8 * (lane & 3));
      wv |= __shfl_xor_sync(kFullMask, wv, 1);
      wv |= __shfl_xor_sync(kFullMask, wv, 2);
      if ((lane & 3) == 0) put(i, lane, wv);
    }
  }
}

// L2 = false: s_b = max |p_j| (Hou et al.); L2 = true: s_b = fl(sqrt(sum p_j^2))
// (QSGD), the sum of squares in the fixed chain order of the scaled sign.
template <int CPT, int WPB, int BITS, bool KEEP_H, bool L2, bool SEG>
__global__ void __launch_bounds__(32 * WPB * (WPB < 4 ? 4 / WPB : 1))
squant_compress_kernel(const CompressArgs a) {
  dq_pdl_enter();
  constexpr int K = (1 << (BITS - 1)) - 1;
  constexpr bool HOLD = KEEP_H && CPT <= 8;
  constexpr int BPC = WPB < 4 ? 4 / WPB : 1;  // buckets per CTA (CTA = max(4, WPB) warps)
  constexpr int CHAIN = 32 * CPT * WPB;
  __shared__ float level_value[K + 1];        // fl(r / K)
  __shared__ float warp_max[2][BPC * WPB];  // by turns: a bucket's maxima may still be read when the next one's come
  __shared__ float chain[(L2 && WPB > 1) ? BPC * CHAIN : 1];
  for (int r = threadIdx.x; r <= K; r += blockDim.x) level_value[r] = __fdiv_rn((float)r, (float)K);
  __syncthreads();

  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int slot = warp / WPB;  // bucket within the CTA
  const int wib = warp % WPB;   // warp within the bucket
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const float* g = a.g + (int64_t)row * a.g_stride;
  float* e = a.e + (int64_t)(worker - a.row0) * a.ld;
  float* h = KEEP_H ? a.h + (int64_t)(worker - a.row0) * a.ld : nullptr;
  uint8_t* msg = a.msg + (int64_t)row * a.msg_stride;

  // The grid is persistent: a warp (a CTA, where several warps share a
  // bucket) takes buckets b, b + stride, ... (the level table above is built
  // once per CTA, not once per bucket) and, with layer segments, loads the
  // next bucket's bounds from the table while it quantises this one, so the
  // data loads of a bucket never wait for the table.
  const int64_t bstride = (int64_t)gridDim.x * BPC;
  int64_t b = (int64_t)blockIdx.x * BPC + slot;
  int64_t next_base = 0, next_end = 0;
  if (SEG && b < a.nb) {
    next_base = a.bstart[b];
    next_end = a.bstart[b + 1];
  }
  int turn = 0;
  for (;; b += bstride, turn ^= 1) {
  const bool valid = b < a.nb;
  if (WPB == 1 ? !valid : b - slot >= a.nb) return;  // (several warps: the whole CTA leaves together)

  // flat buckets: [b n, b n + n) clipped to d; layer buckets (SEG): the table
  int64_t base, end;  // elements at or past `end` are not this bucket's
  if constexpr (SEG) {
    base = valid ? next_base : 0;
    end = valid ? next_end : 0;
    if (b + bstride < a.nb) {
      next_base = a.bstart[b + bstride];
      next_end = a.bstart[b + bstride + 1];
    }
  } else {
    base = b * a.bucket;
    end = a.d;
  }
  const int64_t count = SEG ? end - base : (valid ? min64((int64_t)a.bucket, a.d - base) : 0);
  const bool full = (count == a.bucket);
  const int nchunk = a.bucket >> 2;
  const int row0 = wib * CPT;  // first chunk row of this warp

  float p[CPT][4];
  float sg[HOLD ? CPT : 1][4];
  if (valid) {
    load_and_form<CPT, HOLD>(a, g, e, base, end, 32 * row0 + lane, full, p, sg);
  } else {
#pragma unroll
    for (int i = 0; i < CPT; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) p[i][q] = 0.f;
  }

  float mx = 0.f;
  if constexpr (!L2) {
    // s = max |p| over the bucket (exact in any order)
#pragma unroll
    for (int i = 0; i < CPT; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) mx = fmaxf(mx, fabsf(p[i][q]));
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, off));
    if constexpr (WPB > 1) {
      if (lane == 0) warp_max[turn][warp] = mx;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < WPB; ++w) mx = fmaxf(mx, warp_max[turn][slot * WPB + w]);
      if (!valid) continue;
    }
  } else {
    // s = sqrt of the sum of squares in the chain order
    float cs[CPT];
#pragma unroll
    for (int i = 0; i < CPT; ++i)
      cs[i] = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(p[i][0], p[i][0]), __fmul_rn(p[i][1], p[i][1])),
                                  __fmul_rn(p[i][2], p[i][2])),
                        __fmul_rn(p[i][3], p[i][3]));
    float acc = 0.f;
    if constexpr (WPB == 1) {
#pragma unroll
      for (int i = 0; i < CPT; ++i) acc = __fadd_rn(acc, cs[i]);
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(kFullMask, acc, off));
      mx = __fsqrt_rn(acc);
    } else {
      float* ch = chain + slot * CHAIN;
#pragma unroll
      for (int i = 0; i < CPT; ++i) ch[(row0 + i) * 32 + lane] = cs[i];
      __syncthreads();
      if (wib == 0) {
#pragma unroll 8
        for (int r = 0; r < CPT * WPB; ++r) acc = __fadd_rn(acc, ch[r * 32 + lane]);
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(kFullMask, acc, off));
        if (lane == 0) warp_max[0][slot * WPB] = __fsqrt_rn(acc);
      }
      __syncthreads();
      mx = warp_max[0][slot * WPB];
      if (!valid) continue;
    }
  }
  const float s = mx;
  if (wib == 0 && lane == 0) reinterpret_cast<float*>(msg)[b] = s;
  const float inv = (s > 0.f) ? __fdiv_rn((float)K, s) : 0.f;

  uint32_t* words = reinterpret_cast<uint32_t*>(msg + a.off_payload);
  const int64_t nwords = (a.d * BITS + 31) >> 5;
  // a code word holds 32 / BITS elements of one bucket (buckets start on
  // multiples of 32): write the words that start inside this bucket
  auto put_word = [&](int c_first, uint32_t wv) {
    const int64_t widx = ((base >> 2) + c_first) >> (BITS == 8 ? 0 : BITS == 4 ? 1 : 2);
    if (c_first < nchunk && widx < nwords && (!SEG || widx * (32 / BITS) < end)) words[widx] = wv;
  };
  uint32_t piece[CPT];  // the chunks' 4 * BITS code bits
  // (a whole bucket that fills the lanes' rows needs no test per element)
  auto quantise = [&](auto all) {
#pragma unroll
    for (int i = 0; i < CPT; ++i) {
      const int c = 32 * (row0 + i) + lane;
      const int64_t j = base + 4 * c;
      const int nvalid = all ? 4 : (c < nchunk) ? (int)max64(0, min64(4, end - j)) : 0;
      // global chunk index = Philox counter word 0
      const uint4 r4 = philox4x32_10(make_uint4((uint32_t)(j >> 2), (uint32_t)worker, a.step, kSquantTag),
                                     a.seed_lo, a.seed_hi);
      const uint32_t rq[4] = {r4.x, r4.y, r4.z, r4.w};
      piece[i] = 0;
      float en[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        int code;
        squant_element<K>(p[i][q], s, inv, rq[q], level_value, &code, &en[q]);
        if (q < nvalid) piece[i] |= (uint32_t)code << (q * BITS);
      }
      if constexpr (BITS == 8) put_word(c, piece[i]);
      if (nvalid > 0) store_chunk<KEEP_H, HOLD, CPT>(a, g, e, h, j, all || full, nvalid, en, sg, i);
    }
  };
  if (full && nchunk == 32 * CPT * WPB) quantise(std::true_type{});
  else quantise(std::false_type{});
  pack_rows<BITS, CPT>(piece, lane, [&](int i, int first, uint32_t wv) { put_word(32 * (row0 + i) + first, wv); });
  }
}

// ---------------------------------------------------------------------------
// Buckets of 32, 64 and 128: a warp takes the buckets of a span of 512 elements
// at a time, as four rows of 32 chunks; LPB lanes (8, 16 or 32) of a row make a
// bucket.  Flat buckets are consecutive elements; layer buckets (SEG) start
// where the table says.  The lanes of a bucket reduce among themselves, in
// the fixed order of the wider kernels: the rounds they leave out (partners
// 16 and 8) add the +0 of lanes that a bucket of 32 or 64 does not reach.
// Against a warp per bucket, every lane has work and eight loads of 16 bytes
// in flight whatever the bucket (d = 10M, 16 workers: sign, 32 / 128 per scale,
// 981 / 302 -> 293 / 290 us; 8-bit codes 1373 / 374 -> 338 / 350; layer buckets
// of 64, 8 bits, 746 -> 374).  At 256 per scale the warp per bucket is as good.
// ---------------------------------------------------------------------------
constexpr int kSpan = 512;
constexpr int kSpanRows = kSpan / 128;

// Where this lane's chunks of a span lie: row i's from element j[i], nv[i] of
// its four in the bucket.
struct SpanAt {
  int64_t j[kSpanRows];
  int nv[kSpanRows];
};

template <int LPB, bool SEG>
struct SpanBuckets {
  static constexpr int kBucket = LPB * 4;
  static constexpr int kPerSpan = kSpan / kBucket;
  // the bucket of row i of span `span` in this lane
  static __device__ __forceinline__ int64_t bucket(int64_t span, int i, int lane) {
    return span * kPerSpan + i * (32 / LPB) + lane / LPB;
  }
  static __device__ __forceinline__ SpanAt at(const CompressArgs& a, int64_t span, int lane) {
    SpanAt s;
#pragma unroll
    for (int i = 0; i < kSpanRows; ++i) {
      int64_t first, end;
      if constexpr (SEG) {
        const int64_t b = bucket(span, i, lane);
        first = b < a.nb ? a.bstart[b] : 0;
        end = b < a.nb ? a.bstart[b + 1] : 0;
      } else {
        first = bucket(span, i, lane) * kBucket;
        end = a.d;
      }
      s.j[i] = first + 4 * (lane % LPB);
      s.nv[i] = (int)max64(0, min64(4, end - s.j[i]));
    }
    return s;
  }
};

// p (and fl(eta g)) of this lane's chunks; 0 past a bucket's end.
template <bool KEEP_H>
__device__ __forceinline__ void load_span(const CompressArgs& a, const float* g, const float* e, const SpanAt& at,
                                          bool full, float (&p)[kSpanRows][4], float (&sg)[KEEP_H ? kSpanRows : 1][4]) {
  float gq[kSpanRows][4], eq[kSpanRows][4];
#pragma unroll
  for (int i = 0; i < kSpanRows; ++i) {
    if (full) {
      const float4 x = ld_stream4(g + at.j[i]), y = ld_stream4(e + at.j[i]);
      gq[i][0] = x.x; gq[i][1] = x.y; gq[i][2] = x.z; gq[i][3] = x.w;
      eq[i][0] = y.x; eq[i][1] = y.y; eq[i][2] = y.z; eq[i][3] = y.w;
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        gq[i][q] = q < at.nv[i] ? g[at.j[i] + q] : 0.f;
        eq[i][q] = q < at.nv[i] ? e[at.j[i] + q] : 0.f;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kSpanRows; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float s = __fmul_rn(a.lr, gq[i][q]);
      p[i][q] = full || q < at.nv[i] ? __fadd_rn(s, eq[i][q]) : 0.f;
      if constexpr (KEEP_H) sg[i][q] = s;
    }
}

// Whether a span holds whole buckets only (the same in every lane).
__device__ __forceinline__ bool span_full(const SpanAt& at) {
  bool all = true;
#pragma unroll
  for (int i = 0; i < kSpanRows; ++i) all = all && at.nv[i] == 4;
  return __all_sync(kFullMask, all);
}

template <int LPB, bool KEEP_H, bool SEG>
__global__ void __launch_bounds__(128) sign_compress_rows_kernel(const CompressArgs a) {
  dq_pdl_enter();
  using Buckets = SpanBuckets<LPB, SEG>;
  constexpr int kBucket = Buckets::kBucket;
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const float* g = a.g + (int64_t)row * a.g_stride;
  float* e = a.e + (int64_t)(worker - a.row0) * a.ld;
  float* h = KEEP_H ? a.h + (int64_t)(worker - a.row0) * a.ld : nullptr;
  uint8_t* msg = a.msg + (int64_t)row * a.msg_stride;
  uint32_t* words = reinterpret_cast<uint32_t*>(msg + a.off_payload);
  const int64_t spans = (a.nb + Buckets::kPerSpan - 1) / Buckets::kPerSpan;
  for (int64_t span = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5); span < spans; span += (int64_t)gridDim.x * 4) {
    const SpanAt at = Buckets::at(a, span, lane);
    const bool full = SEG ? span_full(at) : (span + 1) * kSpan <= a.d;
    float p[kSpanRows][4], sg[KEEP_H ? kSpanRows : 1][4];
    load_span<KEEP_H>(a, g, e, at, full, p, sg);
    float s[kSpanRows];
#pragma unroll
    for (int i = 0; i < kSpanRows; ++i) {
      float acc = chunk_abs_sum(p[i][0], p[i][1], p[i][2], p[i][3]);
#pragma unroll
      for (int off = LPB / 2; off >= 1; off >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(kFullMask, acc, off));
      // elements of this lane's bucket (1 where there is none)
      int count = kBucket;
      if (!full) {
        count = at.nv[i];
#pragma unroll
        for (int off = LPB / 2; off >= 1; off >>= 1) count += __shfl_xor_sync(kFullMask, count, off);
        count = max(count, 1);
      }
      s[i] = __fdiv_rn(acc, (float)count);
      const int64_t b = Buckets::bucket(span, i, lane);
      if ((lane & (LPB - 1)) == 0 && (full || b < a.nb)) reinterpret_cast<float*>(msg)[b] = s[i];
    }
#pragma unroll
    for (int i = 0; i < kSpanRows; ++i) {
      const uint32_t wv = pack_sign_row(p[i][0], p[i][1], p[i][2], p[i][3], lane);
      // lane 4 u has the word of the chunks in lanes 8 u ..
      const int64_t j = at.j[i];
      const int nvalid = full ? 4 : at.nv[i];
      const int from = 8 * (lane >> 2) & 31;
      const int64_t jw = SEG ? __shfl_sync(kFullMask, j, from) : j + 4 * (from - lane);
      const bool there = full || __shfl_sync(kFullMask, nvalid, from) > 0;
      if ((lane & 3) == 0 && lane < 16 && there) words[jw >> 5] = wv;
      if (nvalid > 0) {
        float en[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) en[q] = __fsub_rn(p[i][q], p[i][q] < 0.f ? -s[i] : s[i]);
        store_chunk<KEEP_H, KEEP_H, kSpanRows>(a, g, e, h, j, full, nvalid, en, sg, i);
      }
    }
  }
}

template <int LPB, int BITS, bool KEEP_H, bool L2, bool SEG>
__global__ void __launch_bounds__(128) squant_compress_rows_kernel(const CompressArgs a) {
  dq_pdl_enter();
  constexpr int K = (1 << (BITS - 1)) - 1;
  using Buckets = SpanBuckets<LPB, SEG>;
  __shared__ float level_value[K + 1];  // fl(r / K)
  for (int r = threadIdx.x; r <= K; r += blockDim.x) level_value[r] = __fdiv_rn((float)r, (float)K);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const float* g = a.g + (int64_t)row * a.g_stride;
  float* e = a.e + (int64_t)(worker - a.row0) * a.ld;
  float* h = KEEP_H ? a.h + (int64_t)(worker - a.row0) * a.ld : nullptr;
  uint8_t* msg = a.msg + (int64_t)row * a.msg_stride;
  uint32_t* words = reinterpret_cast<uint32_t*>(msg + a.off_payload);
  const int64_t spans = (a.nb + Buckets::kPerSpan - 1) / Buckets::kPerSpan;
  for (int64_t span = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5); span < spans; span += (int64_t)gridDim.x * 4) {
    const SpanAt at = Buckets::at(a, span, lane);
    const bool full = SEG ? span_full(at) : (span + 1) * kSpan <= a.d;
    float p[kSpanRows][4], sg[KEEP_H ? kSpanRows : 1][4];
    load_span<KEEP_H>(a, g, e, at, full, p, sg);
    float s[kSpanRows], inv[kSpanRows];
#pragma unroll
    for (int i = 0; i < kSpanRows; ++i) {
      const float(&v)[4] = p[i];
      float x;
      if constexpr (L2)
        x = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(v[0], v[0]), __fmul_rn(v[1], v[1])), __fmul_rn(v[2], v[2])),
                      __fmul_rn(v[3], v[3]));
      else
        x = fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3])));
#pragma unroll
      for (int off = LPB / 2; off >= 1; off >>= 1) {
        const float y = __shfl_xor_sync(kFullMask, x, off);
        x = L2 ? __fadd_rn(x, y) : fmaxf(x, y);
      }
      if constexpr (L2) x = __fsqrt_rn(x);
      const int64_t b = Buckets::bucket(span, i, lane);
      if ((lane & (LPB - 1)) == 0 && (full || b < a.nb)) reinterpret_cast<float*>(msg)[b] = x;
      s[i] = x;
      inv[i] = (x > 0.f) ? __fdiv_rn((float)K, x) : 0.f;
    }
    // the code word of row i that starts at lane `first` of this lane's bucket
    auto put_word = [&](int i, int first, uint32_t wv) {
      int64_t j = at.j[0];
#pragma unroll
      for (int r = 1; r < kSpanRows; ++r)
        if (i == r) j = at.j[r];
      j -= 4 * (lane - first);
      bool there = true;
      if (!full) {
        int64_t end = SEG ? 0 : a.d;
        if constexpr (SEG) {
          const int64_t b = Buckets::bucket(span, i, lane);
          end = b < a.nb ? a.bstart[b + 1] : 0;
        }
        there = j < end;
      }
      if (there) words[j >> (BITS == 8 ? 2 : BITS == 4 ? 3 : 4)] = wv;
    };
    uint32_t piece[kSpanRows];  // the chunks' 4 * BITS code bits
#pragma unroll
    for (int i = 0; i < kSpanRows; ++i) {
      const int64_t j = at.j[i];
      const int nvalid = full ? 4 : at.nv[i];
      // global chunk index = Philox counter word 0
      const uint4 r4 = philox4x32_10(make_uint4((uint32_t)(j >> 2), (uint32_t)worker, a.step, kSquantTag),
                                     a.seed_lo, a.seed_hi);
      const uint32_t rq[4] = {r4.x, r4.y, r4.z, r4.w};
      piece[i] = 0;
      float en[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        int code;
        squant_element<K>(p[i][q], s[i], inv[i], rq[q], level_value, &code, &en[q]);
        if (q < nvalid) piece[i] |= (uint32_t)code << (q * BITS);
      }
      if constexpr (BITS == 8) put_word(i, lane, piece[i]);
      if (nvalid > 0) store_chunk<KEEP_H, KEEP_H, kSpanRows>(a, g, e, h, j, full, nvalid, en, sg, i);
    }
    pack_rows<BITS, kSpanRows>(piece, lane, put_word);
  }
}

// ---------------------------------------------------------------------------
// Identity: the message is p itself and e = fl(p - p) = 0.
// ---------------------------------------------------------------------------
template <bool KEEP_H>
__global__ void __launch_bounds__(256)
identity_compress_kernel(const CompressArgs a) {
  dq_pdl_enter();
  const int row = blockIdx.y;
  const int worker = a.worker0 + row;
  const float* g = a.g + (int64_t)row * a.g_stride;
  float* e = a.e + (int64_t)(worker - a.row0) * a.ld;
  float* h = KEEP_H ? a.h + (int64_t)(worker - a.row0) * a.ld : nullptr;
  float* vals = reinterpret_cast<float*>(a.msg + (int64_t)row * a.msg_stride);
  const int64_t nchunks = (a.d + 3) >> 2;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nchunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = 4 * c;
    if (j + 3 < a.d) {
      const float4 gv = ld_stream4(g + j);
      const float4 ev = ld_stream4(e + j);
      const float gq[4] = {gv.x, gv.y, gv.z, gv.w};
      const float eq[4] = {ev.x, ev.y, ev.z, ev.w};
      float pv[4], en[4], hv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float s = __fmul_rn(a.lr, gq[q]);
        pv[q] = __fadd_rn(s, eq[q]);
        en[q] = __fsub_rn(pv[q], pv[q]);
        hv[q] = __fadd_rn(s, en[q]);
      }
      st_stream4(vals + j, make_float4(pv[0], pv[1], pv[2], pv[3]));
      st_stream4(e + j, make_float4(en[0], en[1], en[2], en[3]));
      if constexpr (KEEP_H) st_stream4(h + j, make_float4(hv[0], hv[1], hv[2], hv[3]));
    } else {
      for (int64_t jj = j; jj < a.d; ++jj) {
        const float s = __fmul_rn(a.lr, g[jj]);
        const float pv = __fadd_rn(s, e[jj]);
        const float en = __fsub_rn(pv, pv);
        vals[jj] = pv;
        e[jj] = en;
        if constexpr (KEEP_H) h[jj] = __fadd_rn(s, en);
      }
    }
  }
}

// CTAs of a persistent kernel per row: about four waves of resident CTAs in
// all rows, no more than `need`.
int64_t persistent_blocks(int64_t need, int threads, int nworkers) {
  const int sms = device_sms();
  if (sms <= 0) return need;
  const int64_t cap = ((int64_t)sms * 4 * (2048 / threads) + nworkers - 1) / nworkers;
  return need < cap ? need : max64(cap, 1);
}

template <int CPT, int WPB>
cudaError_t sign_dispatch_keep(const CompressArgs& a, bool keep_h, cudaStream_t stream) {
  constexpr int BPC = WPB < 4 ? 4 / WPB : 1;
  constexpr int THREADS = 32 * WPB * BPC;
  const dim3 grid((unsigned)((a.nb + BPC - 1) / BPC), (unsigned)a.nworkers);
  const bool seg = a.bstart != nullptr;
  if (keep_h) {
    if (seg) launch_pdl(sign_compress_kernel<CPT, WPB, true, true>, grid, dim3(THREADS), 0, stream, a);
    else launch_pdl(sign_compress_kernel<CPT, WPB, true, false>, grid, dim3(THREADS), 0, stream, a);
  } else {
    if (seg) launch_pdl(sign_compress_kernel<CPT, WPB, false, true>, grid, dim3(THREADS), 0, stream, a);
    else launch_pdl(sign_compress_kernel<CPT, WPB, false, false>, grid, dim3(THREADS), 0, stream, a);
  }
  return cudaGetLastError();
}

template <int CPT, int WPB, int BITS, bool L2>
cudaError_t squant_dispatch_keep(const CompressArgs& a, bool keep_h, cudaStream_t stream) {
  constexpr int BPC = WPB < 4 ? 4 / WPB : 1;
  constexpr int THREADS = 32 * WPB * BPC;
  const bool seg = a.bstart != nullptr;
  const int64_t gx = persistent_blocks((a.nb + BPC - 1) / BPC, THREADS, a.nworkers);
  const dim3 grid((unsigned)gx, (unsigned)a.nworkers);
  if (keep_h) {
    if (seg) launch_pdl(squant_compress_kernel<CPT, WPB, BITS, true, L2, true>, grid, dim3(THREADS), 0, stream, a);
    else launch_pdl(squant_compress_kernel<CPT, WPB, BITS, true, L2, false>, grid, dim3(THREADS), 0, stream, a);
  } else {
    if (seg) launch_pdl(squant_compress_kernel<CPT, WPB, BITS, false, L2, true>, grid, dim3(THREADS), 0, stream, a);
    else launch_pdl(squant_compress_kernel<CPT, WPB, BITS, false, L2, false>, grid, dim3(THREADS), 0, stream, a);
  }
  return cudaGetLastError();
}

template <int CPT, int WPB>
cudaError_t squant_dispatch_bits(const CompressArgs& a, bool keep_h, bool l2, cudaStream_t stream) {
  switch (a.bits) {
    case 2: return l2 ? squant_dispatch_keep<CPT, WPB, 2, true>(a, keep_h, stream)
                      : squant_dispatch_keep<CPT, WPB, 2, false>(a, keep_h, stream);
    case 4: return l2 ? squant_dispatch_keep<CPT, WPB, 4, true>(a, keep_h, stream)
                      : squant_dispatch_keep<CPT, WPB, 4, false>(a, keep_h, stream);
    case 8: return l2 ? squant_dispatch_keep<CPT, WPB, 8, true>(a, keep_h, stream)
                      : squant_dispatch_keep<CPT, WPB, 8, false>(a, keep_h, stream);
  }
  return cudaErrorInvalidValue;
}

// Whether a bucket of 128 goes to the rows kernels: a span per warp leaves a
// quarter of the warps, and while those do not fill the GPU the latency counts.
// Time of the rows kernels over that of a warp per bucket, by buckets of all
// workers (the same for 1 to 64 workers): sign 1.10 at 4096, 1.13 at 8192, 0.95
// at 16,384, 1.00 at 24,576, 0.94 at 32,768 and 65,536 (with layers 1.25, 1.26, 1.03,
// 1.08, 1.04, 1.00); quantisers 1.17 at 4096, 0.99 at 8192, 0.83 at 16,384, 0.82 at
// 32,768, 0.90 at 65,536 (with layers 1.28, 1.02, 0.91, 0.86, 0.92).
bool rows_pay(const CompressArgs& a, int64_t least) { return a.nb * a.nworkers >= least; }
constexpr int64_t kSignRowsLeast = 32768, kQuantRowsLeast = 10240;

// The grid of the rows kernels: 4 warps per CTA, a span per warp at a time.
dim3 rows_grid(const CompressArgs& a) {
  const int64_t per_span = kSpan / a.bucket;
  const int64_t need = ((a.nb + per_span - 1) / per_span + 3) / 4;
  return dim3((unsigned)persistent_blocks(need, 128, a.nworkers), (unsigned)a.nworkers);
}

template <int LPB>
cudaError_t sign_rows_dispatch(const CompressArgs& a, bool keep_h, cudaStream_t stream) {
  auto go = [&](auto kernel) { return launch_pdl(kernel, rows_grid(a), dim3(128), 0, stream, a); };
  if (a.bstart)
    return keep_h ? go(sign_compress_rows_kernel<LPB, true, true>)
                  : go(sign_compress_rows_kernel<LPB, false, true>);
  return keep_h ? go(sign_compress_rows_kernel<LPB, true, false>)
                : go(sign_compress_rows_kernel<LPB, false, false>);
}

template <int LPB, int BITS, bool L2>
cudaError_t squant_rows_dispatch_keep(const CompressArgs& a, bool keep_h, cudaStream_t stream) {
  auto go = [&](auto kernel) { return launch_pdl(kernel, rows_grid(a), dim3(128), 0, stream, a); };
  if (a.bstart)
    return keep_h ? go(squant_compress_rows_kernel<LPB, BITS, true, L2, true>)
                  : go(squant_compress_rows_kernel<LPB, BITS, false, L2, true>);
  return keep_h ? go(squant_compress_rows_kernel<LPB, BITS, true, L2, false>)
                : go(squant_compress_rows_kernel<LPB, BITS, false, L2, false>);
}

template <int LPB>
cudaError_t squant_rows_dispatch(const CompressArgs& a, bool keep_h, bool l2, cudaStream_t stream) {
  switch (a.bits) {
    case 2: return l2 ? squant_rows_dispatch_keep<LPB, 2, true>(a, keep_h, stream)
                      : squant_rows_dispatch_keep<LPB, 2, false>(a, keep_h, stream);
    case 4: return l2 ? squant_rows_dispatch_keep<LPB, 4, true>(a, keep_h, stream)
                      : squant_rows_dispatch_keep<LPB, 4, false>(a, keep_h, stream);
    case 8: return l2 ? squant_rows_dispatch_keep<LPB, 8, true>(a, keep_h, stream)
                      : squant_rows_dispatch_keep<LPB, 8, false>(a, keep_h, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_sign_compress(const CompressArgs& a, bool keep_h, cudaStream_t stream,
                                 uint64_t* launches) {
  cudaError_t st;
  switch (a.bucket) {
    case 32: st = sign_rows_dispatch<8>(a, keep_h, stream); break;
    case 64: st = sign_rows_dispatch<16>(a, keep_h, stream); break;
    case 128:
      st = rows_pay(a, kSignRowsLeast) ? sign_rows_dispatch<32>(a, keep_h, stream)
                                       : sign_dispatch_keep<1, 1>(a, keep_h, stream);
      break;
    case 256: st = sign_dispatch_keep<2, 1>(a, keep_h, stream); break;
    case 512: st = sign_dispatch_keep<4, 1>(a, keep_h, stream); break;
    case 1024: st = sign_dispatch_keep<2, 4>(a, keep_h, stream); break;
    case 2048: st = sign_dispatch_keep<2, 8>(a, keep_h, stream); break;
    case 4096: st = sign_dispatch_keep<2, 16>(a, keep_h, stream); break;
    default: return cudaErrorInvalidValue;
  }
  *launches += 1;
  return st;
}

cudaError_t launch_squant_compress(const CompressArgs& a, bool keep_h, bool l2, cudaStream_t stream,
                                   uint64_t* launches) {
  cudaError_t st;
  switch (a.bucket) {
    case 32: st = squant_rows_dispatch<8>(a, keep_h, l2, stream); break;
    case 64: st = squant_rows_dispatch<16>(a, keep_h, l2, stream); break;
    case 128:
      st = rows_pay(a, kQuantRowsLeast) ? squant_rows_dispatch<32>(a, keep_h, l2, stream)
                                        : squant_dispatch_bits<1, 1>(a, keep_h, l2, stream);
      break;
    case 256: st = squant_dispatch_bits<2, 1>(a, keep_h, l2, stream); break;
    case 512: st = squant_dispatch_bits<4, 1>(a, keep_h, l2, stream); break;
    case 1024: st = squant_dispatch_bits<8, 1>(a, keep_h, l2, stream); break;
    case 2048: st = squant_dispatch_bits<4, 4>(a, keep_h, l2, stream); break;
    case 4096: st = squant_dispatch_bits<4, 8>(a, keep_h, l2, stream); break;
    default: return cudaErrorInvalidValue;
  }
  *launches += 1;
  return st;
}

cudaError_t launch_identity_compress(const CompressArgs& a, bool keep_h, cudaStream_t stream,
                                     uint64_t* launches) {
  const int64_t nchunks = (a.d + 3) / 4;
  const int64_t blocks = min64((nchunks + 255) / 256, 152 * 8);
  const dim3 grid((unsigned)max64(blocks, 1), (unsigned)a.nworkers);
  if (keep_h) launch_pdl(identity_compress_kernel<true>, grid, dim3(256), 0, stream, a);
  else launch_pdl(identity_compress_kernel<false>, grid, dim3(256), 0, stream, a);
  *launches += 1;
  return cudaGetLastError();
}

}  // namespace dq
