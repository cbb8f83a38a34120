// k_tcgen05.cu -- split-precision products of the factored form on the tensor cores (tc_gemm.h).
//
// C = scale * A B^T for FP64 matrices A (M x K) and B (N x K), both K-contiguous, through integer slices
// held in FP16 (every slice is an integer times a power of two, so the FP16 values are exact):
//   x = 2^e (s0 2^-8 + t1 2^-20 + t2 2^-32),  e per row,  |s0| <= 255, |t1|, |t2| <= 2048,
// as planes a0 = s0, a1 = t1 / 2^12, a2 = t2 / 2^24 (subnormal FP16 below 2^-14, still exact), so that
// a_i b_j carries its weight whichever operand it comes from.  Per 128-deep K chunk the tensor cores
// accumulate in TMEM (FP32):
//   L0  = sum a0 b0                      (products < 2^16, 128 of them: exact in FP32)
//   L12 = sum a0 b1 + a0 b2 + a1 b0 + a1 b1 + a2 b0
// and the epilogue warps drain each chunk into registers: L0 into an int32 running sum (exact for
// K <= 32768), L12 into an FP32 running sum.  The tile is written as C = scale 2^(ea+eb-16) (T0 + T12) in
// FP64.  The leading term is exact whatever rounding the tensor core applies to its FP32 sums; the rest
// carries 2^-12 of the weight.  The representation error is about 2^-33 of the row maxima; the dropped
// products (a1 b2, a2 b1, a2 b2) are about 2^-29 of them.
// The tensor core's FP32 accumulation truncates (measured against an emulation), so L12's smaller terms are
// cut at the scale of its s0 t1 terms, and the truncation error of a chunk grows with the chunk's depth:
// hence chunks of 128 rather than the 512 that L0's exactness would allow.  The eight-product variant keeps
// a1 b2 and a2 b1 as well and splits L12 into L1 = a0 b1 + a1 b0 and L2 (the rest, in its own accumulator),
// C from T0 + (T1 + T2): wide outputs in two launches, (T0, T1) and then T2 added to C (both exact multiples of
// one power of two with a sum below 53 bits, so C is that of one launch bit for bit), as TMEM double-buffers
// three accumulators for 64 columns only, and an MMA of 64 columns issues no faster than one of 128: the two
// products of 180 functions compressed at 1e-8 took 16.2 ms in one launch each of
// 64 columns and take 12.6 ms in four of 128.
//
// Chunks lie at multiples of 128 of the natural K, also where a step table leaves steps of them out (the
// zero blocks of K by parity, below): what is left out adds zeros, so every sum is the dense product's bit
// for bit.
#include "tc_gemm.h"

namespace lrtei {
namespace tc {

// f in FP64 from its bits: conversions to FP64 run at two a clock and SM.
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f), E = (b >> 23) & 0xFFu;
  if (E == 0 || E == 0xFFu) return (double)f;  // zero, subnormal, infinity, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + (896u << 20))), (int)(b << 29));
}

// (T0 + T12 / 2^12) 2^k in integer arithmetic (this device's FP64 rate would make an FP64
// epilogue a visible part of the GEMM): X = T0 2^21 + round(T12 2^9) is an integer below 2^53
// (|T0| < 2^31; |T12| < 2^36 for K <= 32768), so X 2^(k-21) is exact in FP64 and is built from
// its bits.  Rounding T12 to 2^-9 moves the result by at most 2^-22 of a unit of T0, far below
// the 2^-33 representation error of the operands.  Results below the normal range flush to 0.
// round(f 2^9) as an integer, from the bits of the FP32 value f.
__device__ __forceinline__ int64_t round_2p9(float f) {
  const uint32_t fb = __float_as_uint(f);
  const int fe = (int)((fb >> 23) & 0xFFu);
  int64_t q = 0;
  if (fe != 0) {  // zero or subnormal f is below the 2^-9 resolution
    const int64_t m = (int64_t)((fb & 0x7FFFFFu) | 0x800000u);
    const int sh = fe - 127 - 23 + 9;  // f 2^9 = m 2^sh
    if (sh >= 0)
      q = m << min(sh, 27);  // q < 2^51 (|f| < 2^42)
    else if (sh > -26)
      q = (m + (1LL << (-sh - 1))) >> (-sh);
    if (fb >> 31) q = -q;
  }
  return q;
}

// t2: a second FP32 sum of the same weight as t12 (the three-accumulator scheme), else 0.
__device__ __forceinline__ double combine_pow2(int t0, float t12, int k, float t2 = 0.f) {
  const int64_t X = ((int64_t)t0 << 21) + round_2p9(t12) + round_2p9(t2);
  if (X == 0) return 0.0;
  const uint64_t a = (uint64_t)(X < 0 ? -X : X);
  const int lz = __clzll((long long)a);    // a < 2^53: lz >= 11
  const uint64_t mant = a << (lz - 11);    // leading one at bit 52
  const int E = 1023 + (63 - lz) + k - 21;  // X 2^(k-21) = 1.f 2^(E-1023)
  if (E <= 0) return 0.0;
  const uint64_t bits = ((uint64_t)(X < 0) << 63) | ((uint64_t)min(E, 2046) << 52) | (mant & ((1ULL << 52) - 1));
  return __longlong_as_double((long long)bits);
}

// f = i + l / 2^21 for |f| < 2^23 by two additions to powers of two: i is even, |l| <= 2^21 rounded to nearest, halves
// away from zero as f counts.
__device__ __forceinline__ void split_2p21(float f, int& i, int& l) {
  const float m = f + 25165824.f;  // 1.5 2^24: the last place is 2
  i = 2 * (__float_as_int(m) - 0x4BC00000);
  const float r = f - (m - 25165824.f), n = __fmaf_rn(r, 0x1p21f, 12582912.f);
  l = __float_as_int(n) - 0x4B400000;
  const float d = __fmaf_rn(r, 0x1p21f, -(n - 12582912.f));  // what the rounding (halves to even) left
  l += d == copysignf(0.5f, f) ? (__float_as_int(f) >> 31) | 1 : 0;
}

// combine_pow2(t0, 4096 t1, k, 4096 t2) in 32-bit words, the same bits: X = S 2^21 + L with S = T0 + the whole parts
// (|T0| <= 255^2 K, |T1| < 256 K, K <= 32768: within 32 bits).  For the products whose tiles are mostly epilogue (few
// steps, or two launches): X of the exchange, 90 orbitals of 180 functions in two blocks, 1.77 -> 1.52 ms; the compressed
// B of 180 functions unchanged to 0.8 % faster.  Not for the others: alike at 180 functions, 128.7 -> 131.4 us for the B of 45.
__device__ __forceinline__ double combine_words(int t0, float t1, int k, float t2 = 0.f, bool two = false) {
  int i, L;
  split_2p21(t1, i, L);
  int S = t0 + i;
  if (two) {
    int i2, l2;
    split_2p21(t2, i2, l2);
    S += i2;
    L += l2;
  }
  S += L >> 21;
  L &= 0x1FFFFF;
  const int neg = S >> 31;  // -1: two's complement of the 53 bits
  S = (S ^ neg) + (L == 0 ? neg & 1 : 0);
  L = ((L ^ neg) - neg) & 0x1FFFFF;
  const uint32_t low = (uint32_t)L << 11;  // S : low, the leading one moved to the top
  const bool big = S != 0;
  const uint32_t top = big ? (uint32_t)S : low, rest = big ? low : 0u;
  const int lz = __clz((int)top);
  const uint32_t h = __funnelshift_l(rest, top, lz), l = rest << (lz & 31);
  const int E = (big ? 1023 + 52 - 21 : 1023 + 20 - 21) + k - lz;
  const uint32_t hi = ((uint32_t)neg & 0x80000000u) | (uint32_t)min(E, 2046) << 20 | (h >> 11 & 0xFFFFFu);
  const bool zero = E <= 0 || top == 0;
  return __hiloint2double((int)(zero ? 0u : hi), (int)(zero ? 0u : __funnelshift_r(l, h, 11)));
}

// eight_hi and eight_lo: the two launches of eight products on 128 columns.
enum class Scheme { six, eight, eight_hi, eight_lo, plain };

// SWAP: the sums of B A^T, a_i b_j in the order of b_i a_j (FP32 sums depend on it).
template <int BN_, Scheme M, bool LIST_, bool SWAP = false>
struct Split {
  static constexpr bool P8 = M == Scheme::eight, PLAIN = M == Scheme::plain, HI = M == Scheme::eight_hi,
                        LO = M == Scheme::eight_lo, ONE = PLAIN || LO;  // ONE: a single FP32 accumulator
  static constexpr int BN = BN_, NP = PLAIN ? 1 : HI ? 2 : 3, PT = PLAIN ? 1 : 3, NACC = ONE ? 1 : P8 ? 3 : 2, KS = PLAIN ? 8 : 2;
  // KS: two steps a stage, half the barrier rounds; plain operands, whose step is one MMA, a whole chunk (ten rows
  // of B_u of 60 functions, n = 11: G 21 -> 13 us, B_u 24 -> 16, together with an epilogue without FP64)
  static constexpr int UNIT = 8, CHUNK = 8;  // 128 deep
  static constexpr bool BF16 = PLAIN, ACCUM = LO, LIST = LIST_;

  static __device__ __forceinline__ void mma(uint32_t d0, uint64_t a0, uint64_t b0, uint32_t idesc, uint32_t first) {
    if constexpr (PLAIN) {
      mma_bf16(d0, a0, b0, idesc, first);
    } else {
      constexpr uint64_t AS = (128 * 32) >> 4, BS = (BN * 32) >> 4;  // from plane to plane
      const uint32_t d1 = d0 + BN, d2 = P8 ? d0 + 2 * BN : d1;
      const uint64_t a1 = a0 + AS, a2 = a0 + 2 * AS, b1 = b0 + BS, b2 = b0 + 2 * BS;
      const uint32_t d2s = LO ? d0 : d2;
      // grouped by A slice so that each is read from shared memory once per k step; with eight products the
      // smaller terms go to their own accumulator d2, so that the tensor core's truncating FP32 accumulation
      // cuts them at their own scale
      if constexpr (SWAP) {
        if constexpr (!LO) {
          mma_bf16_a<ACol::fill>(d0, a0, b0, idesc, first);
          mma_bf16(d1, a1, b0, idesc, first);
        }
        if constexpr (!HI) mma_bf16(P8 || LO ? d2s : d1, a2, b0, idesc, P8 || LO ? first : 1u);
        if constexpr (!LO) mma_bf16(d1, a0, b1, idesc, 1u);
        if constexpr (!HI) {
          mma_bf16(d2s, a1, b1, idesc, 1u);
          mma_bf16(d2s, a0, b2, idesc, 1u);
        }
        if constexpr (P8 || LO) {
          mma_bf16(d2s, a1, b2, idesc, 1u);
          mma_bf16(d2s, a2, b1, idesc, 1u);
        }
        return;
      }
      if constexpr (HI) {
        mma_bf16_a<ACol::fill>(d0, a0, b0, idesc, first);
        mma_bf16_a<ACol::lastuse>(d1, a0, b1, idesc, first);
        mma_bf16(d1, a1, b0, idesc, 1u);
        return;
      }
      if constexpr (LO) {
        mma_bf16(d0, a0, b2, idesc, first);
        mma_bf16(d0, a1, b1, idesc, 1u);
        mma_bf16_a<ACol::fill>(d0, a2, b0, idesc, 1u);
        mma_bf16_a<ACol::lastuse>(d0, a2, b1, idesc, 1u);
        mma_bf16(d0, a1, b2, idesc, 1u);
        return;
      }
      mma_bf16_a<ACol::fill>(d0, a0, b0, idesc, first);
      mma_bf16_a<ACol::use>(d1, a0, b1, idesc, first);
      mma_bf16_a<ACol::lastuse>(d2, a0, b2, idesc, P8 ? first : 1u);
      mma_bf16_a<ACol::fill>(d1, a1, b0, idesc, 1u);
      mma_bf16_a<ACol::lastuse>(d2, a1, b1, idesc, 1u);
      if constexpr (P8) {
        mma_bf16_a<ACol::fill>(d2, a2, b0, idesc, 1u);
        mma_bf16_a<ACol::lastuse>(d2, a2, b1, idesc, 1u);
        mma_bf16(d2, a1, b2, idesc, 1u);
      } else {
        mma_bf16(d1, a2, b0, idesc, 1u);
      }
    }
  }

  template <int QC>
  struct Sums {
    int T0[ONE ? 1 : QC];
    float T1[QC], T2[P8 ? QC : 1];
    __device__ __forceinline__ void clear() {
#pragma unroll
      for (int j = 0; j < QC; ++j) {
        if constexpr (!ONE) T0[j] = 0;
        T1[j] = 0.f;
        if constexpr (P8) T2[j] = 0.f;
      }
    }
    __device__ __forceinline__ void drain(uint32_t t) {
#pragma unroll
      for (int j0 = 0; j0 < QC; j0 += 8) {  // the loads of an 8-column group are in flight together
        uint32_t r[8], q[8];
        if constexpr (!ONE) tmem_ld8(t + j0, r);
        tmem_ld8(t + (ONE ? 0 : BN) + j0, q);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if constexpr (!ONE) T0[j0 + j] += __float2int_rn(__uint_as_float(r[j]));
          T1[j0 + j] += __uint_as_float(q[j]);
        }
        if constexpr (P8) {
          tmem_ld8(t + 2 * BN + j0, q);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j) T2[j0 + j] += __uint_as_float(q[j]);
        }
      }
    }
    template <int C>
    __device__ __forceinline__ void hold(int j0) {
      if constexpr (!ONE) {
#pragma unroll
        for (int j = 0; j < C; ++j) {
          asm volatile("" : "+r"(T0[j0 + j]), "+f"(T1[j0 + j]) : : "memory");
          if constexpr (P8) asm volatile("" : "+f"(T2[j0 + j]) : : "memory");
        }
      }
    }
    // The planes' weights make T1 and T2 those of the sums of s0 t1 over 2^12.
    __device__ __forceinline__ double value(int j, int k, double scale) const {
      if constexpr (PLAIN) return scale == 1.0 ? widen(T1[j]) : scale * widen(T1[j]);  // k is 16 (k_plain_rows)
      const int t0 = LO ? 0 : T0[ONE ? 0 : j];
      const float t2 = P8 ? T2[P8 ? j : 0] : 0.f;
      const double v = SWAP || HI || LO ? combine_words(t0, T1[j], k - 16, t2, P8)
                                        : combine_pow2(t0, T1[j] * 4096.f, k - 16, t2 * 4096.f);
      return scale == 1.0 ? v : scale * v;
    }
  };
};

// Tile width: 128 columns for wide outputs (a 128 x 64 MMA is bound by its operand reads from shared memory and
// by its issue); plain BF16 takes 64.
static int tile_n(int64_t N, bool plain) { return N <= 32 ? 32 : (N <= 64 || plain) ? 64 : 128; }
// Of 128 and 64 columns the ones whose waves take less.  A 64-column tile takes ~0.72 of a 128-column one (its
// MMAs half, the reads of A and the latencies the same): 64 where they fill SMs that 128 leave idle.  1035 pairs,
// 2197 deep: B_u (45 tiles of 128) 48 -> 42 us; G (180) stays at two waves of 128, 63 us.
static int tile_of_waves(int BN, int64_t tiles128, int64_t tiles64) {
  if (BN != 128) return BN;
  const int64_t sms = 152, w128 = (tiles128 + sms - 1) / sms, w64 = (tiles64 + sms - 1) / sms;
  return 72 * w64 < 100 * w128 ? 64 : 128;
}

// The same for eight products of M rows and N columns, which are one launch in 64-column tiles and two in 128-column
// ones.  Up to 128 columns the left operand's bytes count: three planes once (the second tile finds them in L2) against
// two and three.  J-builds of 100 densities, 120 functions, n = 16: 495 us in two launches, 309 in one; of 65 densities, 90
// functions, n = 12: 178, 115; exchange of 180 functions and 90 orbitals, n = 10: 1.07 ms, 0.85.
static int tile_of_rows(int BN, int64_t M, int64_t N, int64_t splits) {
  if (BN == 128 && N <= 128) return 64;
  const int64_t tiles = (M + 127) / 128 * splits;
  return tile_of_waves(BN, tiles * ((N + 127) / 128), tiles * ((N + 63) / 64));
}

template <bool LIST, bool SWAP>
static lrtei_status run_as(const tcg::Params& p, int BN, bool plain, bool eight, cudaStream_t st) {
  if (plain)
    return BN == 64 ? tcg::launch<Split<64, Scheme::plain, LIST>>(p, st) : tcg::launch<Split<32, Scheme::plain, LIST>>(p, st);
  if (eight && BN == 128) {
    tcg::Params q = p;
    q.mirror = 0;
    const lrtei_status s = tcg::launch<Split<128, Scheme::eight_hi, LIST, SWAP>>(q, st);
    if (s != LRTEI_OK) return s;
    q.mirror = p.mirror;
    q.accumulate = 1;
    return tcg::launch<Split<128, Scheme::eight_lo, LIST, SWAP>>(q, st);
  }
  if (eight)
    return BN == 64 ? tcg::launch<Split<64, Scheme::eight, LIST, SWAP>>(p, st) : tcg::launch<Split<32, Scheme::eight, LIST, SWAP>>(p, st);
  if (BN == 128) return tcg::launch<Split<128, Scheme::six, LIST, SWAP>>(p, st);
  return BN == 64 ? tcg::launch<Split<64, Scheme::six, LIST, SWAP>>(p, st) : tcg::launch<Split<32, Scheme::six, LIST, SWAP>>(p, st);
}
static lrtei_status run(const tcg::Params& p, int BN, bool plain, bool eight, cudaStream_t st, bool swap = false) {
  ProfScope ps("tc_gemm", st);
  if (p.seg[0].tab) return run_as<true, false>(p, BN, plain, eight, st);
  return swap ? run_as<false, true>(p, BN, plain, eight, st) : run_as<false, false>(p, BN, plain, eight, st);
}

// What the products share: operands, output (or split partials) and checks.  units: 128-deep chunks of K.
static lrtei_status fill(tcg::Params& p, const SplitMatrix& A, const SplitMatrix& B, int BN, int64_t units, double scale,
                         double* d_C, int64_t ldc, bool transpose_out, int& splits, int64_t c_rows, int64_t c_cols,
                         double* d_part, int* d_status) {
  if (A.plain != B.plain || A.eight != B.eight) {
    set_error("tc_gemm: operands must share one precision scheme");
    return LRTEI_ERR_ARG;
  }
  if (A.tile != 128 || B.tile % BN != 0) {
    set_error("tc_gemm: operand tiles of %d and %d rows for %d columns", A.tile, B.tile, BN);
    return LRTEI_ERR_ARG;
  }
  splits = (int)std::max<int64_t>(1, std::min<int64_t>(splits, units));
  const int64_t per = (units + splits - 1) / splits;
  if (per * 128 > 32768) {
    set_error("tc_gemm: more than 32768 K per split (use more splits)");
    return LRTEI_ERR_UNSUPPORTED;
  }
  splits = (int)((units + per - 1) / per);
  if (splits > 1 && !d_part) {
    set_error("tc_gemm: split-K needs a partial buffer");
    return LRTEI_ERR_ARG;
  }
  p.splits = splits;
  p.a = reinterpret_cast<const uint8_t*>(A.d);
  p.b = reinterpret_cast<const uint8_t*>(B.d);
  p.a_steps = A.kpad / tcg::KB;
  p.b_steps = B.kpad / tcg::KB;
  p.b_tile = B.tile;
  p.ea = A.expo;
  p.eb = B.expo;
  p.scale = scale;
  p.transpose_out = transpose_out ? 1 : 0;
  p.C = splits > 1 ? d_part : d_C;
  p.ldc = splits > 1 ? c_cols : ldc;
  p.split_stride = splits > 1 ? c_rows * c_cols : 0;
  p.status = d_status;
  p.align = tc::store_align(p.C, p.ldc);
  p.test_stall = tcg::test_stall_cycles();
  return LRTEI_OK;
}

static lrtei_status reduce(const double* part, int splits, int64_t rows, int64_t cols, double* C, int64_t ldc,
                           cudaStream_t st) {
  launch_reduce_splits(part, splits, rows * cols, rows, cols, cols, C, ldc, st);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? LRTEI_OK : cuda_fail(e, "reduce_splits");
}

}  // namespace tc

lrtei_status tc_gemm(const SplitMatrix& A, int64_t a_row0, const SplitMatrix& B, int64_t M, int64_t N, double scale,
                     double* d_C, int64_t ldc, bool transpose_out, bool symmetric_upper, int splits, double* d_part,
                     int* d_status, cudaStream_t st) {
  if (A.kpad != B.kpad || A.kpad % 128 != 0) {
    set_error("tc_gemm: operands must share a K padded to a multiple of 128");
    return LRTEI_ERR_ARG;
  }
  if (symmetric_upper && (M != N || a_row0 != 0)) {
    set_error("tc_gemm: symmetric mode needs a square output");
    return LRTEI_ERR_ARG;
  }
  if (symmetric_upper) return tc_gemm_sym_band(A, B, 0, N, N, d_C, ldc, d_status, st);
  const int m_lo = (int)(a_row0 % 128), units = (int)(A.kpad / 128);
  int BN = tc::tile_n(N, A.plain);
  if (A.eight) BN = tc::tile_of_rows(BN, M + m_lo, N, splits);
  tcg::Params p{};
  const int64_t c_rows = transpose_out ? N : M, c_cols = transpose_out ? M : N;
  lrtei_status s = tc::fill(p, A, B, BN, units, scale, d_C, ldc, transpose_out, splits, c_rows, c_cols, d_part, d_status);
  if (s != LRTEI_OK) return s;
  p.nseg = 1;
  p.seg[0] = {a_row0 - m_lo, 0, M + m_lo, N, transpose_out ? -m_lo : -m_lo * p.ldc, 0, 0, 0, units,
              (int)((M + m_lo + 127) / 128), (int)((N + BN - 1) / BN), m_lo, A.steps(), nullptr};
  p.nitems = (int64_t)p.seg[0].tiles_m * p.seg[0].tiles_n;
  s = tc::run(p, BN, A.plain, A.eight, st);
  if (s != LRTEI_OK || splits == 1) return s;
  return tc::reduce(d_part, splits, c_rows, c_cols, d_C, ldc, st);
}

// C = A B^T for few rows A and many rows B, with B as the left operand of the tensor cores: its rows fill the 128 of
// a tile and the few of A its columns, 32, 64 or 128 of them, so that the drains and the epilogue run over live
// elements and a warp's stores along a row of C are one contiguous run.  53 rows by 2.5 M of 180: 1.5 ms with A on the left, 0.78 this
// way (2.9 GB of B); 10 rows by 437 k of 75: 264 us, 84.
lrtei_status tc_gemm_few(const SplitMatrix& A, const SplitMatrix& B, int64_t M, int64_t N, double* d_C, int64_t ldc,
                         int* d_status, cudaStream_t st) {
  if (A.kpad != B.kpad || A.kpad % 128 != 0) {
    set_error("tc_gemm_few: operands must share a K padded to a multiple of 128");
    return LRTEI_ERR_ARG;
  }
  const int units = (int)(A.kpad / 128);
  int splits = 1, BN = tc::tile_n(M, A.plain);
  if (A.eight) BN = tc::tile_of_rows(BN, N, M, 1);
  tcg::Params p{};
  lrtei_status s = tc::fill(p, B, A, BN, units, 1.0, d_C, ldc, true, splits, M, N, nullptr, d_status);
  if (s != LRTEI_OK) return s;
  p.nseg = 1;
  p.seg[0] = {0, 0, N, M, 0, 0, 0, 0, units, (int)((N + 127) / 128), (int)((M + BN - 1) / BN), 0, A.steps(), nullptr};
  p.nitems = (int64_t)p.seg[0].tiles_m * p.seg[0].tiles_n;
  return tc::run(p, BN, A.plain, A.eight, st, true);
}

// Several products C_i = A_i B_i^T of rows of A and B in one launch (their tiles share the last waves).
lrtei_status tc_gemm_blocks(const SplitMatrix& A, const SplitMatrix& B, const std::vector<TcBlock>& blocks, double* d_C,
                            int64_t ldc, int* d_status, cudaStream_t st) {
  if (A.kpad != B.kpad || A.kpad % 128 != 0 || blocks.size() > (size_t)tcg::kMaxSeg) {
    set_error("tc_gemm_blocks: operands must share a K padded to a multiple of 128, at most %d blocks", tcg::kMaxSeg);
    return LRTEI_ERR_ARG;
  }
  int64_t nmax = 0;
  for (const TcBlock& b : blocks) nmax = std::max(nmax, b.N);
  const int BN = tc::tile_n(nmax, A.plain), units = (int)(A.kpad / 128);
  tcg::Params p{};
  int splits = 1;
  lrtei_status s = tc::fill(p, A, B, BN, units, 1.0, d_C, ldc, false, splits, 0, 0, nullptr, d_status);
  if (s != LRTEI_OK) return s;
  for (const TcBlock& b : blocks) {
    if (b.M <= 0 || b.N <= 0) continue;
    const int m_lo = (int)(b.a_row0 % 128);
    tcg::Seg& o = p.seg[p.nseg++];
    o = {b.a_row0 - m_lo, b.b_row0, b.M + m_lo, b.N, b.c_off - m_lo * p.ldc, p.nitems, 0, 0, units,
         (int)((b.M + m_lo + 127) / 128), (int)((b.N + BN - 1) / BN), m_lo, A.steps(), nullptr};
    p.nitems += (int64_t)o.tiles_m * o.tiles_n;
  }
  return tc::run(p, BN, A.plain, A.eight, st);
}

lrtei_status tc_gemm_sym_band(const SplitMatrix& A, const SplitMatrix& B, int64_t row0, int64_t row1, int64_t N,
                              double* d_C, int64_t ldc, int* d_status, cudaStream_t st) {
  if (row0 % 128 != 0 || row0 >= row1 || row1 > N || (row1 < N && row1 % 128 != 0) || A.rows < row1 - row0 ||
      A.kpad != B.kpad || A.kpad % 128 != 0) {
    set_error("tc_gemm_sym_band: rows [%lld, %lld) are not a 128-aligned band of %lld", (long long)row0,
              (long long)row1, (long long)N);
    return LRTEI_ERR_ARG;
  }
  // upper-triangular enumeration in 128 x 128 blocks (128 / BN tiles each); A holds rows [row0, row1) only
  const int64_t nb = (N + 127) / 128, b0 = row0 / 128, b1 = (row1 + 127) / 128;
  const int64_t blocks = (nb - b0) * (nb - b0 + 1) / 2 - (nb - b1) * (nb - b1 + 1) / 2;
  const int BN = tc::tile_of_waves(tc::tile_n(std::max<int64_t>(N, 65), A.plain), blocks, 2 * blocks);
  const int units = (int)(A.kpad / 128);
  tcg::Params p{};
  int splits = 1;
  lrtei_status s = tc::fill(p, A, B, BN, units, 1.0, d_C, ldc, false, splits, N, N, nullptr, d_status);
  if (s != LRTEI_OK) return s;
  p.symmetric = p.mirror = 1;
  p.nseg = 1;
  p.blk0 = b0;
  p.blk1 = b1;
  p.nb = nb;
  p.seg[0] = {-row0, 0, row1, N, 0, 0, 0, 0, units, (int)(b1 - b0), (int)nb, 0, A.steps(), nullptr};
  p.nitems = blocks * (128 / BN);
  return tc::run(p, BN, A.plain, A.eight, st);
}

// Products with K by parity classes: of the dense K (columns m in the natural order) only the K blocks that
// hold a class's columns are stored and multiplied, with chunks and sums as in the dense product.
// Order n = 24: 288 of 864 blocks per row, a third of the MMAs of G = F_u K and of the bytes of K in a
// J-build (all zeros left out would be an eighth, but a 16-deep block mixes degrees: bit-equal sums want
// whole blocks).
lrtei_status tc_gemm_K(const SplitMatrix& X, int64_t x_row0, const SplitMatrix& K, const ParityClasses& pc, int64_t rows,
                       bool k_is_a, double* d_C, int splits, double* d_part, int* d_status, cudaStream_t st) {
  const SplitMatrix &A = k_is_a ? K : X, &B = k_is_a ? X : K;
  const int m_lo = k_is_a ? 0 : (int)(x_row0 % 128);
  int BN = tc::tile_n(rows, A.plain);
  if (k_is_a) {
    if (A.eight) BN = tc::tile_of_rows(BN, pc.rows, rows, splits);
  } else {
    int64_t nmax = 0, t128 = 0, t64 = 0;
    for (int c = 0; c < pc.nclass; ++c) {
      nmax = std::max<int64_t>(nmax, pc.size[c]);
      t128 += (pc.size[c] + 127) / 128;
      t64 += (pc.size[c] + 63) / 64;
    }
    const int64_t tiles_m = (rows + m_lo + 127) / 128;
    BN = tc::tile_of_waves(tc::tile_n(nmax, A.plain), tiles_m * t128, tiles_m * t64);
  }
  if ((k_is_a && x_row0 != 0) || X.kpad / 128 != pc.units) {
    set_error("tc_gemm_K: operand does not match the plan's K");
    return LRTEI_ERR_ARG;
  }
  tcg::Params p{};
  lrtei_status s = tc::fill(p, A, B, BN, pc.units, 1.0, d_C, pc.cols, k_is_a, splits, rows, pc.cols, d_part, d_status);
  if (s != LRTEI_OK) return s;
  p.list_is_a = k_is_a ? 0 : 1;
  for (int c = 0; c < pc.nclass; ++c) {
    const int64_t w = (pc.size[c] + 63) / 64 * 64;  // the padding columns come out as zeros
    if (w == 0) continue;
    tcg::Seg& o = p.seg[p.nseg++];
    const int* tab = pc.tab ? pc.tab + pc.tab_off[c] : nullptr;
    if (k_is_a)
      o = {pc.row0[c], 0, w, rows, pc.off[c], p.nitems, 0, 0, pc.units, (int)((w + 127) / 128), (int)((rows + BN - 1) / BN),
           0, X.steps(), tab};
    else
      o = {x_row0 - m_lo, pc.row0[c], rows + m_lo, w, pc.off[c] - m_lo * p.ldc, p.nitems, 0, 0, pc.units,
           (int)((rows + m_lo + 127) / 128), (int)((w + BN - 1) / BN), m_lo, X.steps(), tab};
    p.nitems += (int64_t)o.tiles_m * o.tiles_n;
  }
  s = tc::run(p, BN, A.plain, A.eight, st);
  if (s != LRTEI_OK || splits == 1) return s;
  return tc::reduce(d_part, splits, rows, pc.cols, d_C, pc.cols, st);
}

}  // namespace lrtei
