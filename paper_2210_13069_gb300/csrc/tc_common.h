// tc_common.h -- pieces shared by the tensor-core kernels (k_tcgen05.cu, k_tc_hadamard.cu,
// k_slices.cu): inline PTX for mbarriers, TMA, tcgen05 MMAs and TMEM loads, the shared-memory
// operand descriptor, the tensor-map encoder, and the integer slicing of an FP64 element into the
// three FP16 slices of the split-precision operands.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include "lrtei_internal.h"

namespace lrtei {
namespace tc {

constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz: every mbarrier wait gives up after this

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait_at(uint32_t addr, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(addr), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same without suspending the thread.
__device__ __forceinline__ bool mbar_test_wait_at(uint32_t addr, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(addr), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  return mbar_try_wait_at(smem_u32(bar), parity);
}

// Bounded wait: false if the CTA is aborting or the wait gave up (which raises the abort).
// sleep_ns > 0 parks the waiting warp between polls, leaving issue slots to the MMA thread.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          unsigned sleep_ns = 0, long long limit = kWaitCycles) {
  long long t0 = clock64();
  uint32_t spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    if (sleep_ns) __nanosleep(sleep_ns);
    if ((++spins & 255u) == 0) {
      if (*abort_flag) return false;
      if (clock64() - t0 > limit) {
        *abort_flag = 1;
        atomicExch(status, (int)kDevTimeout);
        return false;
      }
    }
  }
  return true;
}

// Waits, bounded, for a row's bulk copy into shared memory (phase 0 of `bar`); expiry raises the status word.  stall > 0
// (tests only): then waits that many cycles for the next phase, which nothing completes.
__device__ __forceinline__ void wait_staged(uint64_t* bar, int* status, long long stall = 0) {
  for (uint32_t phase = 0; phase < (stall > 0 ? 2u : 1u); ++phase) {
    const long long limit = phase ? stall : kWaitCycles;
    for (long long t0 = clock64(); !mbar_try_wait(bar, phase);)
      if (clock64() - t0 > limit) {
        latch_status(status, (int)kDevTimeout);
        break;
      }
  }
}

// True on one lane of the (converged) warp.  The MMA warps branch on it rather than on the lane number:
// the compiler then knows that one thread runs the branch and issues MMAs without a per-thread loop.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}

__device__ __forceinline__ void tma_load_2d(const CUtensorMap* map, void* dst, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// A contiguous copy into shared memory (16-byte aligned, a multiple of 16 bytes), completing on `bar`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// K-major operand tile with BK*2-byte rows and the matching swizzle: 8-row atoms of 8*BK*2
// bytes stacked along M/N (128-byte swizzle for BK = 64, 64-byte swizzle for BK = 32).
template <int BK>
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  static_assert(BK == 64 || BK == 32, "BK");
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);          // start address
  d |= (uint64_t)1 << 16;                           // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)((8 * BK * 2) >> 4) << 32;         // stride byte offset: next 8-row atom
  d |= (uint64_t)1 << 46;                           // descriptor version
  d |= (uint64_t)(BK == 64 ? 2 : 4) << 61;          // 128-byte or 64-byte swizzle
  return d;
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
          d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// The same with a collector-buffer hint for A: fill (read A and keep it), use (A from the
// buffer), lastuse (from the buffer, then release it).  Consecutive MMAs on one A slice read
// it from shared memory once.
enum class ACol { fill, use, lastuse };
template <ACol C>
__device__ __forceinline__ void mma_bf16_a(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate) {
  if constexpr (C == ACol::fill)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  else if constexpr (C == ACol::use)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------------ operand slices
__device__ __forceinline__ uint16_t f16_bits(float f) {
  __half h = __float2half_rn(f);
  return *reinterpret_cast<uint16_t*>(&h);
}

// Magnitude of x to 20 mantissa bits, ordered as unsigned integers: all that a row's exponent needs.
__device__ __forceinline__ uint32_t magnitude(double x) { return (uint32_t)__double2hiint(x) & 0x7FFFFFFFu; }

// e with max|x| 256/255 < 2^e from the row's largest magnitude: one more than the exponent's where the mantissa reaches
// 255/128.  kZeroRowExpo for rows below ~1e-301 and for NaN: treated as zero (a product with a zero row is 0
// whatever its exponent).  Integers, as two FP64 operations a clock and SM are a visible part of slicing short rows.
constexpr int kZeroRowExpo = -30000;
__device__ __forceinline__ int slice_exponent(uint32_t mag) {
  const int e = (int)(mag >> 20) - 1022 + ((mag & 0xFFFFFu) >= 0xFE000u ? 1 : 0);
  return mag <= 0x7FF00000u && e >= -1000 ? e : kZeroRowExpo;
}

// Slices of one element: q = round(x 2^(32-e)), s0 = round(q / 2^24), r = q - s0 2^24,
// t1 = round(r / 2^12), t2 = r - t1 2^12; x ~ 2^e (s0 2^-8 + t1 2^-20 + t2 2^-32), |s0| <= 255,
// |t1|, |t2| <= 2048: integers that FP16 holds exactly, also over 2^12 and 2^24.
// In 32-bit integers: |q| < 255 2^24 is the top of the mantissa, leading one at bit 31, shifted right by
// s = e + 1022 - E and rounded half up by the bit below (s > 32 leaves nothing; zeros and subnormals give 0).  By
// 64-bit shifts an element took ~2.5 times the instructions, which bound the slicing kernels: 16290 rows of 13824
// 0.96 -> 0.84 ms; the exchange's MT of 180 functions 1.89 -> 1.67 ms.
__device__ __forceinline__ void slice_ints(double x, int e, bool live, int& s0, int& t1, int& t2) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int E = (int)((hi >> 20) & 0x7FF), s = e + 1022 - E;
  const uint32_t top = __funnelshift_l(lo, hi, 11) | 0x80000000u;
  const uint32_t half = __funnelshift_rc(lo << 11, top, s) >> 31;
  const uint32_t a = live && E != 0 && (uint32_t)s <= 32 ? __funnelshift_rc(top, 0, s) + half : 0;  // |q|
  const int neg = (int)(hi >> 31);
  const int m = (int)((a + 0x800000u - (uint32_t)neg) >> 24);  // |s0|: halves round up, for -q down
  int r = (int)(a - ((uint32_t)m << 24));                      // |r| <= 2^23
  s0 = neg ? -m : m;
  r = neg ? -r : r;
  t1 = (r + (1 << 11)) >> 12;
  t2 = r - (t1 << 12);
}

// Integers of magnitude up to 2^22 as FP32 by the exponent trick, times a power of two: no pass through the
// conversion unit (16 a clock and SM; slicing took three of them and three more to FP16 per element).
__device__ __forceinline__ float small_float(int i, float scale) {
  return __fmaf_rn(__int_as_float(0x4B400000 + i), scale, -12582912.f * scale);
}
__device__ __forceinline__ uint32_t f16x2_bits(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// The planes of the GEMM operands, s0, t1 / 2^12 and t2 / 2^24, of two neighbouring elements as FP16 pairs.
__device__ __forceinline__ void slice_pair(double x, double y, int e, bool lx, bool ly, uint32_t& p0, uint32_t& p1,
                                           uint32_t& p2) {
  int a0, a1, a2, b0, b1, b2;
  slice_ints(x, e, lx, a0, a1, a2);
  slice_ints(y, e, ly, b0, b1, b2);
  p0 = f16x2_bits(small_float(a0, 1.f), small_float(b0, 1.f));
  p1 = f16x2_bits(small_float(a1, 0x1p-12f), small_float(b1, 0x1p-12f));
  p2 = f16x2_bits(small_float(a2, 0x1p-24f), small_float(b2, 0x1p-24f));
}

// The planes of the Hadamard form's operands: s0, t1, t2 / 2^12 and, where s1h is given, t1 / 2^12.
__device__ __forceinline__ void slice_store(double x, int e, bool live, int64_t o, uint16_t* s0, uint16_t* s1,
                                            uint16_t* s2, uint16_t* s1h) {
  int a, b, c;
  slice_ints(x, e, live, a, b, c);
  s0[o] = f16_bits((float)a);
  s1[o] = f16_bits((float)b);
  s2[o] = f16_bits((float)c * 0x1p-12f);
  if (s1h) s1h[o] = f16_bits((float)b * 0x1p-12f);
}

// ------------------------------------------------------------------ packed FP32
// Two FP32 numbers in a register pair, each operation rounded as the scalar one, one instruction for both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ f32x2 pack2(uint32_t x, uint32_t y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(x), "r"(y));
  return r;
}
__device__ __forceinline__ float half_of(f32x2 v, int odd) {
  float x, y;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
  return (odd & 1) ? y : x;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ULL; }

// ------------------------------------------------------------------ FP32 pairs to FP64
// An FP32 number as m 2^e, |m| < 2^24.
__device__ __forceinline__ int64_t f32_int(float f, int& e) {
  const uint32_t b = __float_as_uint(f);
  const int E = (int)((b >> 23) & 0xFFu);
  int64_t m = (int64_t)(b & 0x7FFFFFu);
  if (E) m |= 0x800000;
  e = (E ? E : 1) - 150;
  return (b >> 31) ? -m : m;
}

// (hi + lo) 2^k in FP64 from integer arithmetic (this device's FP64 rate would make FP64
// conversions a visible share of the kernels that store pairs): hi + lo = X 2^q with |X| < 2^63,
// exact when the two exponents lie within 38 bits, else the smaller part rounded at 2^-62 of the
// larger; then X 2^(q+k) rounded to 53 bits (half up on the magnitude).  Results below the normal
// range flush to 0.
__device__ __forceinline__ double fpair_ldexp(float hi, float lo, int k) {
  int eb, es;
  int64_t mb = f32_int(hi, eb), ms = f32_int(lo, es);
  if (mb == 0 || (ms != 0 && es > eb)) {  // (mb, eb): the part with the larger exponent
    const int64_t tm = mb;
    mb = ms;
    ms = tm;
    const int te = eb;
    eb = es;
    es = te;
  }
  if (mb == 0) return 0.0;
  int64_t X;
  int q;
  if (ms == 0) {
    X = mb;
    q = eb;
  } else if (eb - es <= 38) {
    X = (mb << (eb - es)) + ms;
    q = es;
  } else {
    const int sh = eb - es - 38;
    X = mb << 38;
    if (sh < 62) {
      const int64_t half = 1LL << (sh - 1);
      X += ms >= 0 ? ((ms + half) >> sh) : -((-ms + half) >> sh);
    }
    q = es + sh;
  }
  if (X == 0) return 0.0;
  const uint64_t a = (uint64_t)(X < 0 ? -X : X);
  const int top = 63 - __clzll((long long)a);  // leading bit
  uint64_t mant;
  int E = top + q + k + 1023;
  if (top > 52) {
    const int sh = top - 52;
    mant = (a + (1ULL << (sh - 1))) >> sh;
    if (mant >> 53) {
      mant >>= 1;
      ++E;
    }
  } else {
    mant = a << (52 - top);
  }
  if (E <= 0) return 0.0;
  if (E > 2046) E = 2046;
  const uint64_t bits = ((uint64_t)(X < 0) << 63) | ((uint64_t)E << 52) | (mant & ((1ULL << 52) - 1));
  return __longlong_as_double((long long)bits);
}

// ------------------------------------------------------------------ stores
// Four consecutive columns of one row of C: 32-byte accesses where ldc and C allow them.
__device__ __forceinline__ void load4(const double* c, int al, int live, double (&v)[4]) {
  if (al == 4 && live == 4) {
    const double4_32a x = *reinterpret_cast<const double4_32a*>(c);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  } else if (al >= 2 && live == 4) {
    const double2 x = *reinterpret_cast<const double2*>(c), y = *reinterpret_cast<const double2*>(c + 2);
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = j < live ? c[j] : 0.0;
  }
}
__device__ __forceinline__ void store4(double* c, int al, int lo, int live, const double (&v)[4]) {
  if (al == 4 && live == 4 && lo <= 0) {
    double4_32a x;
    x.x = v[0]; x.y = v[1]; x.z = v[2]; x.w = v[3];
    *reinterpret_cast<double4_32a*>(c) = x;
  } else if (al >= 2 && live == 4 && lo <= 0) {
    *reinterpret_cast<double2*>(c) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(c + 2) = make_double2(v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j >= lo && j < live) c[j] = v[j];
  }
}

// Doubles per access that every row of C allows (tiles and segments start at multiples of four columns).
inline int store_align(const double* C, int64_t ldc) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(C);
  return (ldc % 4 == 0 && (a & 31) == 0) ? 4 : (ldc % 2 == 0 && (a & 15) == 0) ? 2 : 1;
}

// ------------------------------------------------------------------ host: tensor maps
inline PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    else
      cudaGetLastError();
  }
  return fn;
}

// 2D tensor map of one 16-bit operand plane (rows x kpad, K contiguous): boxes of bk x box_rows,
// 128-byte swizzle for bk = 64, 64-byte swizzle for bk = 32.
inline bool encode_plane(CUtensorMap* m, const uint16_t* base, int64_t rows, int64_t kpad, int box_rows, bool bf16,
                         int bk) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(kpad * 2)};
  cuuint32_t box[2] = {(cuuint32_t)bk, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (void*)base, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, bk == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace tc
}  // namespace lrtei
