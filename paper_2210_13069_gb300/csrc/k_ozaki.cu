// k_ozaki.cu -- FP64 products of the factored form on the tensor cores, by error-free slicing
// (Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication", 2012).
//
// C = A B^T for FP64 matrices (rows x K, K contiguous).  Every row is scaled by a power of two and cut
// into six balanced base-512 digits held exactly in FP16:
//   x = 2^e sum_i d_i 2^(-9 (i + 1)),  |d_i| <= 256, |x| < 2^(e - 1),
// 53 bits below the binade of the row's largest element, which is FP64's own resolution there.  The 21
// digit products d_i d_j with level i + j <= 5 are formed on the tensor cores (the dropped ones are
// about 2^-50 of the row maxima over K = 13 824, below the rounding of an FP64 dot product of that
// length).  The FP32 sum of one level over a chunk of K is exact: at most (level + 1) 64 2^16 <= 2^24
// for levels 0..3 and 64-deep chunks (levels 0 and 1: 128-deep ones too); levels 4 and 5 weigh 2^-36
// and less.  Chunks are added in int32 (K is split before 128 of them), and two levels make one integer
// X = 512 L_even + L_odd, so a result carries one rounding per pair of levels.  Rows holding a NaN or an infinity are marked in
// their exponent and give NaN.
//
// Why: this device runs 1.2 TFLOP/s in FP64 and 1 900 in FP16; 21 products leave ~90.
//
// Wide products (B_u = G F_u^T and G = F_u K) run as three launches (levels 4-5, 2-3, 0-1; smallest
// first, the later ones adding to C): 128 x 128 tiles, two FP32 accumulators double-buffered in the
// 512 TMEM columns, and an epilogue register budget of one 64-bit sum per element allow two levels at
// a time.  Skinny products (J-builds, N <= 32 columns a tile) keep all six levels in TMEM (2 x 6 x 32
// columns) and read their operand once.
// Measured: FP64 B of 60 functions (n = 24, P = 32) 187 -> 3.0 ms; J-build of 16 densities, 120
// functions, 32.7 -> 0.50 ms (6.2 ms with the FP64 kernels of k_jfp64.cu; its products read their
// operand at 6.3 TB/s); the error against 64-bit
// references is the same (1.8e-14) and slightly smaller (1.2e-14 -> 1.1e-14).
#include <math.h>
#include <stdlib.h>

#include <algorithm>
#include <type_traits>

#include "lrtei_internal.h"
#include "tc_common.h"

namespace lrtei {
namespace oz {

using namespace tc;

constexpr int BM = 128;
constexpr int KB = 16;       // K of one operand block (32-byte rows, 32-byte swizzle): one MMA step
constexpr int EPI = 16;      // epilogue warps: four per TMEM lane quadrant
constexpr int THREADS = 64 + 32 * EPI;
constexpr int kGroupM = 16;  // M tiles walked together (operand slabs shared in L2)
constexpr int kGroupRows = 8;

// One block of the product: rows [a_row0, a_row0 + M) of A, rows [b_row0, b_row0 + N) of B, nch chunks of
// 64 K from a_k0 and b_k0, written at C + c_off.
struct Seg {
  int64_t a_row0, b_row0, M, N, c_off, item0;
  int a_k0, b_k0, nch, tiles_m, tiles_n;
  int m_lo;  // rows of the first tile below the wanted ones (a_row0 is a multiple of 128)
};
struct Params {
  Seg seg[8];
  int nseg, splits, symmetric, transpose_out, accumulate, mirror, align;
  int64_t nitems;  // per split
  const uint8_t* a;  // digit tiles of both operands and their tiles' K steps
  const uint8_t* b;
  int64_t a_steps, b_steps;
  const int* ea;
  const int* eb;
  double* C;
  int64_t ldc, split_stride;
  int* status;
  long long test_stall;
};

// X 2^k for |X| < 2^53 from integer arithmetic: an FP64 operation on a 128 x 128 tile takes 8 192 clocks
// of an SM here.  Results below the normal range flush to zero.
__device__ __forceinline__ double int_ldexp(long long X, int k) {
  if (X == 0) return 0.0;
  const unsigned long long a = (unsigned long long)(X < 0 ? -X : X);
  const int lz = __clzll((long long)a);
  const int E = 1023 + 63 - lz + k;
  if (E <= 0) return 0.0;
  const unsigned long long m = E > 2046 ? 0ULL : (a << (lz - 11)) & ((1ULL << 52) - 1);
  return __longlong_as_double((long long)(((unsigned long long)(X < 0) << 63) |
                                          ((unsigned long long)min(E, 2047) << 52) | m));
}

struct Work {
  int seg, m0, n0, c0, nch, split;  // m0, n0: first row and column of the tile inside the segment
  bool mirror;
};

__device__ __forceinline__ Work work_item(const Params& p, int64_t item, int BN) {
  Work w;
  w.split = (int)(item / p.nitems);
  int64_t t = item % p.nitems;
  w.seg = 0;
  while (w.seg + 1 < p.nseg && t >= p.seg[w.seg + 1].item0) ++w.seg;
  const Seg& s = p.seg[w.seg];
  t -= s.item0;
  w.mirror = false;
  if (p.symmetric) {  // upper triangle of 128 x 128 blocks in groups of block rows, column by column
    const int64_t nb = s.tiles_n;
    int64_t r = 0, c = 0;
    for (int64_t R0 = 0; R0 < nb; R0 += kGroupRows) {
      const int64_t R1 = min(nb, R0 + kGroupRows), g = R1 - R0;
      const int64_t tri = g * (g + 1) / 2, in_group = tri + (nb - R1) * g;
      if (t >= in_group) { t -= in_group; continue; }
      if (t >= tri) {
        c = R1 + (t - tri) / g;
        r = R0 + (t - tri) % g;
      } else {
        c = R0;
        while (t >= c - R0 + 1) { t -= c - R0 + 1; ++c; }
        r = R0 + t;
      }
      break;
    }
    w.m0 = (int)(r * BM);
    w.n0 = (int)(c * BN);
    w.mirror = c != r;
  } else {
    const int64_t per_group = (int64_t)kGroupM * s.tiles_n;
    const int64_t first = (t / per_group) * kGroupM, in_g = t % per_group;
    const int64_t gsize = min((int64_t)kGroupM, s.tiles_m - first);
    w.m0 = (int)((first + in_g % gsize) * BM);
    w.n0 = (int)(in_g / gsize * BN);
  }
  const int per = (s.nch + p.splits - 1) / p.splits;
  w.c0 = w.split * per;
  w.nch = max(0, min(s.nch, w.c0 + per) - w.c0);
  return w;
}

// A contiguous copy into shared memory (16-byte aligned, a multiple of 16 bytes), completing on `bar`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

template <int BN, int LV0, int NLV>
struct Cfg {
  static constexpr int NP = LV0 + NLV;  // digit planes of each operand: levels below NP need digits below NP
  static constexpr uint32_t A_BYTES = BM * KB * 2, B_BYTES = BN * KB * 2;
  static constexpr uint32_t STEP = NP * (A_BYTES + B_BYTES);
  // K blocks per stage: one barrier round per 32 KB or more (48 KB with six planes)
  static constexpr int KS = STEP >= 30 * 1024 ? 1 : STEP >= 16 * 1024 ? 2 : 4;
  static constexpr uint32_t STAGE = KS * STEP;
  static constexpr int STAGES = 220 * 1024 / STAGE;
  // 64-deep K pieces per chunk: exactness (top of the file); levels 4 and 5 need none
  static constexpr int CH = NLV == 6 ? 1 : LV0 == 0 ? 2 : LV0 == 4 ? 4 : 1;
  static constexpr int SPP = 64 / KB / KS;  // stages per 64-deep piece
  static constexpr bool FLT = LV0 >= 4;     // FP32 running sums (level 4 weighs 2^-36)
  static constexpr size_t SMEM = STAGES * STAGE + 1024 + 256;
  static_assert(2 * NLV * BN <= 512, "two buffers of the accumulators must fit in TMEM");
};

// K-major operand block of 32-byte rows in the 32-byte swizzle: 8-row atoms of 256 bytes.
__device__ __forceinline__ uint64_t block_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (uint64_t)1 << 16 | (uint64_t)(256 >> 4) << 32 | (uint64_t)1 << 46 |
         (uint64_t)6 << 61;
}

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

// Three roles: warp 0 copies, warp 1 issues the MMAs, warps 2-17 drain and store.  The MMA warp keeps
// warp-uniform control flow and issues from the lane elect.sync names: under `if (lane == 0)` every MMA
// took about 100 clocks to issue, whatever its size (skinny J-build product 330 -> 213 us).  The epilogue
// stores from registers while the next tile's MMAs run.
template <int BN, int LV0, int NLV>
__global__ void __launch_bounds__(THREADS, 1) k_oz_gemm(const __grid_constant__ Params p) {
  using F = Cfg<BN, LV0, NLV>;
  constexpr int NP = F::NP, STAGES = F::STAGES, QC = BN / (EPI / 4);
  constexpr int SPC = F::CH * F::SPP;  // stages of a full chunk
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * F::STAGE);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;
  uint64_t* acce = accf + 2;
  uint64_t* done = acce + 2;
  uint64_t* never = done + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(never + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int64_t nitems = p.nitems * p.splits;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], EPI);
    }
    mbar_init(done, 1);
    mbar_init(never, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {  // producer: the digit planes of one K block are contiguous per operand
      uint32_t it = 0;
      bool stop = false;
      for (int64_t item = blockIdx.x; item < nitems && !stop; item += gridDim.x) {
        const Work w = work_item(p, item, BN);
        const Seg& sg = p.seg[w.seg];
        const uint8_t* a = p.a + (((sg.a_row0 + w.m0) / BM) * p.a_steps + (sg.a_k0 + w.c0 * 64) / KB) * (kOzSlices * F::A_BYTES);
        const uint8_t* b = p.b + (((sg.b_row0 + w.n0) / BN) * p.b_steps + (sg.b_k0 + w.c0 * 64) / KB) * (kOzSlices * F::B_BYTES);
        for (int kk = 0; kk < w.nch * F::SPP; ++kk, ++it) {
          const int s = (int)(it % STAGES);
          if (!mbar_wait(&empty[s], ((it / STAGES) & 1u) ^ 1u, abort_flag, p.status, 32)) { stop = true; break; }
          mbar_arrive_expect_tx(&full[s], F::STAGE);
          uint8_t* st = smem + (size_t)s * F::STAGE;
#pragma unroll
          for (int q = 0; q < F::KS; ++q) {
            bulk_load(st + q * F::STEP, a, NP * F::A_BYTES, &full[s]);
            bulk_load(st + q * F::STEP + NP * F::A_BYTES, b, NP * F::B_BYTES, &full[s]);
            a += kOzSlices * F::A_BYTES;
            b += kOzSlices * F::B_BYTES;
          }
        }
      }
      if (*abort_flag) {  // bounded wait for the loads in flight before the CTA can exit
        for (uint32_t j = (it > (uint32_t)STAGES ? it - STAGES : 0u); j < it; ++j) {
          long long t0 = clock64();
          while (!mbar_try_wait(&full[j % STAGES], (j / STAGES) & 1u) && clock64() - t0 < kWaitCycles) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    const uint32_t idesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    const bool elected = elect_one();
    uint32_t it = 0, cg = 0;
    bool ok = true;
    if (p.test_stall > 0)
      ok = __all_sync(0xffffffffu, mbar_wait(never, 0u, abort_flag, p.status, 0, p.test_stall));
    for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const Work w = work_item(p, item, BN);
      int left = w.nch * F::SPP;
      for (; left > 0 && ok; ++cg) {
        const int buf = (int)(cg & 1u), ns = min(left, SPC);
        left -= ns;
        ok = __all_sync(0xffffffffu, mbar_wait(&acce[buf], ((cg >> 1) & 1u) ^ 1u, abort_flag, p.status));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d0 = tmem_base + (uint32_t)(buf * NLV * BN);
        for (int step = 0; step < ns; ++step, ++it) {
          const int s = (int)(it % STAGES);
          ok = __all_sync(0xffffffffu, mbar_wait(&full[s], (it / STAGES) & 1u, abort_flag, p.status));
          if (!ok) break;
          tc_fence_after();
          const uint32_t base = smem_u32(smem + (size_t)s * F::STAGE);
          const uint64_t a0 = block_desc(base), b0 = block_desc(base + NP * F::A_BYTES);
          if (elected) {
#pragma unroll
            for (int k = 0; k < F::KS; ++k) {
              const uint64_t a = a0 + (uint64_t)((k * F::STEP) >> 4), b = b0 + (uint64_t)((k * F::STEP) >> 4);
              const uint32_t first = (step == 0 && k == 0) ? 0u : 1u;
#pragma unroll
              for (int i = 0; i < NP; ++i) {
                // A digit i meets the B digits j with LV0 <= i + j < LV0 + NLV (consecutive, so that the
                // A slice is read from shared memory once)
                const int j0 = LV0 > i ? LV0 - i : 0, j1 = NP - i;
#pragma unroll
                for (int j = j0; j < j1; ++j) {
                  const uint32_t d = d0 + (uint32_t)((i + j - LV0) * BN);
                  const uint64_t ad = a + (uint64_t)((i * F::A_BYTES) >> 4), bd = b + (uint64_t)((j * F::B_BYTES) >> 4);
                  const uint32_t acc = i == 0 ? first : 1u;
                  if (j1 - j0 == 1) mma_bf16(d, ad, bd, idesc, acc);
                  else if (j == j0) mma_bf16_a<ACol::fill>(d, ad, bd, idesc, acc);
                  else if (j == j1 - 1) mma_bf16_a<ACol::lastuse>(d, ad, bd, idesc, acc);
                  else mma_bf16_a<ACol::use>(d, ad, bd, idesc, acc);
                }
              }
            }
            mma_commit(&empty[s]);
            if (step == ns - 1) mma_commit(&accf[buf]);
          }
          __syncwarp();
        }
      }
    }
    if (elected) {  // retire every MMA issued before TMEM is released
      mma_commit(done);
      long long t0 = clock64();
      while (!mbar_try_wait(done, 0u) && clock64() - t0 < kWaitCycles) {
      }
    }
    __syncwarp();
  } else {
    using Sum = typename std::conditional<F::FLT, float, int>::type;
    const int ew = warp - 2, quad = warp & 3, col0 = (ew >> 2) * QC, row = quad * 32 + lane;
    uint32_t cg = 0;
    bool ok = true;
    for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const Work w = work_item(p, item, BN);
      const Seg& sg = p.seg[w.seg];
      Sum T[NLV][QC];
#pragma unroll
      for (int x = 0; x < NLV; ++x)
#pragma unroll
        for (int j = 0; j < QC; ++j) T[x][j] = 0;
      for (int left = w.nch * F::SPP; left > 0; left -= SPC, ++cg) {
        const int buf = (int)(cg & 1u);
        int got = 1;
        if (lane == 0) got = mbar_wait(&accf[buf], (cg >> 1) & 1u, abort_flag, p.status, 32) ? 1 : 0;
        got = __shfl_sync(0xffffffffu, got, 0);
        if (!got) { ok = false; break; }
        tc_fence_after();
        const uint32_t tbase = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * NLV * BN + col0);
#pragma unroll
        for (int x = 0; x < NLV; x += 2)
#pragma unroll
          for (int j0 = 0; j0 < QC; j0 += 8) {
            uint32_t r[8], q[8];
            tmem_ld8(tbase + x * BN + j0, r);
            tmem_ld8(tbase + (x + 1) * BN + j0, q);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if constexpr (F::FLT) {
                T[x][j0 + j] += __uint_as_float(r[j]);
                T[x + 1][j0 + j] += __uint_as_float(q[j]);
              } else {
                T[x][j0 + j] += __float2int_rn(__uint_as_float(r[j]));
                T[x + 1][j0 + j] += __float2int_rn(__uint_as_float(q[j]));
              }
            }
          }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[buf]);
      }
      if (!ok || *abort_flag) break;
      // Element (gm, gn0 + j): sum over the pairs of levels of (512 T_even + T_odd) 2^(ea + eb - 9 (level + 3)).
      const int m = w.m0 + row, n = w.n0 + col0, M = (int)sg.M, N = (int)sg.N;
      const bool mlive = m < M && m >= sg.m_lo;
      const int ea = mlive ? p.ea[sg.a_row0 + m] - 9 * (LV0 + 3) : 0;
      const int* eb = p.eb + sg.b_row0;
      double* C = p.C + sg.c_off + (int64_t)w.split * p.split_stride;
      const bool diag = p.symmetric && !w.mirror;  // the upper triangle only, mirrored below
#pragma unroll
      for (int j0 = 0; j0 < QC; j0 += 4) {
        // one group of columns at a time (the sums fill the registers): nothing of it is computed earlier
        if constexpr (!F::FLT)
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int x = 0; x < NLV; ++x) asm volatile("" : "+r"(T[x][j0 + j]) : : "memory");
        const int live = mlive ? max(0, min(4, N - n - j0)) : 0;
        double v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int k = ea + (j < live ? __ldg(eb + n + j0 + j) : 0);
          double sum = 0.0;
#pragma unroll
          for (int x = NLV - 2; x >= 0; x -= 2) {
            long long X;
            if constexpr (F::FLT) X = __float2ll_rn(T[x][j0 + j]) * 512 + __float2ll_rn(T[x + 1][j0 + j]);
            else X = (long long)T[x][j0 + j] * 512 + T[x + 1][j0 + j];
            const double t = int_ldexp(X, k - 9 * x);
            sum = x == NLV - 2 ? t : sum + t;
          }
          v[j] = k >= kOzBad / 2 ? __longlong_as_double(0x7FF8000000000000LL) : sum;
        }
        if (p.transpose_out) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < live) {
              double* c = C + (int64_t)(n + j0 + j) * p.ldc + m;
              *c = p.accumulate ? *c + v[j] : v[j];
            }
        } else {
          double* c = C + (int64_t)m * p.ldc + n + j0;
          if (p.accumulate) {
            double old[4];
            load4(c, p.align, live, old);
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] += old[j];
          }
          store4(c, p.align, diag ? max(0, m - n - j0) : 0, live, v);
        }
        if (p.mirror) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < live && (!diag || m < n + j0 + j)) C[(int64_t)(n + j0 + j) * p.ldc + m] = v[j];
        }
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

// ---------------------------------------------------------------- slicing
// Digit tiles: `tile` rows x 16 columns x 6 planes are contiguous (each plane's 32-byte rows in the 32-byte
// swizzle of shared memory), K block after K block, so that a stage is one contiguous copy per operand
// and block, and as shallow as the pipeline wants it.
// Destination row i holds source row rowinv[i] (NULL: i), destination column j source column colinv[j]
// (NULL: j for j < k); -1 gives zeros.  One block per row: the largest magnitude, then the digits.
__global__ void k_oz_split(const double* __restrict__ src, int64_t k, int64_t ld, int64_t kpad, int tile,
                           const int* __restrict__ rowinv, const int* __restrict__ colinv, uint16_t* __restrict__ d,
                           int* __restrict__ expo) {
  __shared__ unsigned long long red[32];
  const int64_t i = blockIdx.x;
  const int64_t r = rowinv ? rowinv[i] : i;
  const double* x = src + r * ld;
  unsigned long long mx = 0;
  if (r >= 0)
    for (int64_t j = threadIdx.x; j < k; j += blockDim.x) {
      const unsigned long long a = (unsigned long long)__double_as_longlong(x[j]) & 0x7FFFFFFFFFFFFFFFULL;
      mx = a > mx ? a : mx;
    }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = red[w] > mx ? red[w] : mx;
  const int E = (int)(mx >> 52);  // biased exponent of the largest magnitude; 0: zero row, 0x7FF: not finite
  const bool live = E > 0 && E < 0x7FF;
  if (threadIdx.x == 0) expo[i] = E == 0x7FF ? kOzBad : live ? E - 1021 : 0;
  for (int64_t j = 4 * (int64_t)threadIdx.x; j < kpad; j += 4 * (int64_t)blockDim.x) {
    uint16_t h[4][kOzSlices];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t c = colinv ? colinv[j + e] : (j + e < k ? j + e : -1);
      const unsigned long long b = (live && c >= 0) ? (unsigned long long)__double_as_longlong(x[c]) : 0ULL;
      const int Ex = (int)((b >> 52) & 0x7FF), sh = E - Ex;
      const unsigned long long m = (b & ((1ULL << 52) - 1)) | (1ULL << 52);
      // q = round(x 2^(54 - e)), |q| <= 2^53
      long long q = (Ex == 0 || sh > 54) ? 0 : sh == 0 ? (long long)m : (long long)((m + (1ULL << (sh - 1))) >> sh);
      if (b >> 63) q = -q;
#pragma unroll
      for (int s = kOzSlices - 1; s > 0; --s) {
        const int dg = (int)((q + 256) & 511) - 256;
        q = (q - dg) >> 9;
        h[e][s] = f16_bits((float)dg);
      }
      h[e][0] = f16_bits((float)(int)q);
    }
    const int rr = (int)(i % tile), kk = (int)(j % KB) * 2;  // byte inside the 32-byte row; 16-byte pieces swizzled
    uint8_t* o = reinterpret_cast<uint8_t*>(d) + ((i / tile) * (kpad / KB) + j / KB) * (int64_t)(kOzSlices * tile * 32) +
                 rr * 32 + (kk ^ (((rr >> 2) & 1) << 4));
#pragma unroll
    for (int s = 0; s < kOzSlices; ++s)
      *reinterpret_cast<ushort4*>(o + s * tile * 32) = make_ushort4(h[0][s], h[1][s], h[2][s], h[3][s]);
  }
}

// Sum of split partials of a symmetric product (upper blocks only) into both triangles.
__global__ void k_oz_reduce_sym(const double* __restrict__ part, int splits, int64_t n, double* __restrict__ C,
                                int64_t ldc) {
  __shared__ double t[32][33];
  const int64_t i0 = (int64_t)blockIdx.y * 32, j0 = (int64_t)blockIdx.x * 32;
  if (j0 < i0) return;
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int64_t i = i0 + y, j = j0 + threadIdx.x;
    if (i < n && j < n && i <= j) {
      double s = 0.0;
      for (int q = 0; q < splits; ++q) s += part[((int64_t)q * n + i) * n + j];
      C[i * ldc + j] = s;
      t[y][threadIdx.x] = s;
    }
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int64_t j = j0 + y, i = i0 + threadIdx.x;
    if (i < n && j < n && i < j) C[j * ldc + i] = t[threadIdx.x][y];
  }
}

// K of the factored form by parity class (lrtei_internal.h, ParityClasses): row krow(a1, a2, a3), column
// index of (b1, b2, b3) inside the class.  One CTA per (a1, b1, a2, b2) of matching parities: the P
// node factors scale w_p A_x A_y once, then one FMA per node and (a3, b3).
__global__ void __launch_bounds__(256) k_oz_build_K(int n, int P, int par, ParityClasses pc, const double* __restrict__ C,
                                                   const double* __restrict__ w, double scale, double* __restrict__ K,
                                                   int64_t ldK) {
  __shared__ double r[kMaxP];
  const int nn = n * n, ab1 = blockIdx.x, ab2 = blockIdx.y;
  const int a1 = ab1 / n, b1 = ab1 % n, a2 = ab2 / n, b2 = ab2 % n;
  if (par && (((a1 + b1) | (a2 + b2)) & 1)) return;
  for (int p = threadIdx.x; p < P; p += blockDim.x)
    r[p] = scale * w[p] * C[(size_t)p * nn + ab1] * C[((size_t)P + p) * nn + ab2];
  __syncthreads();
  const int step = par ? 2 : 1;
  for (int e = threadIdx.x; e < nn; e += blockDim.x) {
    const int a3 = e / n, b3 = e % n;
    if ((a3 + b3) % step) continue;
    double acc = 0.0;
    for (int p = 0; p < P; ++p) acc = fma(r[p], C[((size_t)2 * P + p) * nn + e], acc);
    K[pc.row(a1, a2, a3) * ldK + pc.index(b1, b2, b3)] = acc;
  }
}

// Unique-pair densities, one row per density: u[q][r] = D_q(mu, nu) (2 - [mu == nu]).
__global__ void k_oz_pack(int nbf, int R, int64_t npair, const int* __restrict__ pair_mu,
                          const int* __restrict__ pair_nu, const double* __restrict__ D, double* __restrict__ u) {
  const int64_t total = npair * R;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t % npair, q = t / npair;
    const int mu = pair_mu[r], nu = pair_nu[r];
    const double v = D[q * nbf * nbf + (int64_t)mu * nbf + nu];
    u[t] = mu == nu ? v : 2.0 * v;
  }
}

// ---------------------------------------------------------------- host side
template <int BN, int LV0, int NLV>
static lrtei_status launch(const Params& p, cudaStream_t st) {
  using F = Cfg<BN, LV0, NLV>;
  static bool attr_set = false;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_oz_gemm<BN, LV0, NLV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "oz_gemm smem attribute");
    attr_set = true;
  }
  static int nsm = 0;
  if (nsm <= 0) {
    int dev = 0;
    LRTEI_CUDA(cudaGetDevice(&dev));
    LRTEI_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  }
  const int64_t items = p.nitems * p.splits;
  if (items <= 0) return LRTEI_OK;
  count_launch();
  k_oz_gemm<BN, LV0, NLV><<<(unsigned)std::min<int64_t>(items, nsm), THREADS, F::SMEM, st>>>(p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "oz_gemm launch");
  return LRTEI_OK;
}

// Splits of K that shorten the last wave of `items` tiles on 152 SMs, each at least 8 pieces of 64; a
// split more costs about `store` pieces (its tile's store and its share of the reduction).  At most 120
// pieces each: the int32 sums of a chunk's at most 2^24 hold 127.
static int pick_splits(int64_t items, int chunks, double store) {
  int best = 1;
  double cost = 1e30;
  const int least = (chunks + 119) / 120;
  for (int s = least; s <= std::max(16, least) && (s == least || chunks / s >= 8); ++s) {
    const double c = (double)((items * s + 151) / 152) * ((double)chunks / s + store) * (1.0 + 0.01 * s);
    if (c < cost) { cost = c; best = s; }
  }
  return best;
}

}  // namespace oz

void launch_oz_split(const double* d_src, int64_t k, int64_t ld, const int* d_rowinv, const int* d_colinv, OzMatrix& m,
                     cudaStream_t st) {
  if (m.rows <= 0) return;
  count_launch();
  oz::k_oz_split<<<(unsigned)m.rows, m.rows < 2 * 152 ? 1024 : 256, 0, st>>>(d_src, k, ld, m.kpad, m.tile, d_rowinv, d_colinv,
                                                                          m.d, m.expo);
}

void launch_oz_build_K(int n, int P, bool parity, const ParityClasses& pc, const double* d_C, const double* d_w,
                       double scale, double* d_K, int64_t ldK, cudaStream_t st) {
  count_launch();
  oz::k_oz_build_K<<<dim3((unsigned)(n * n), (unsigned)(n * n)), 256, 0, st>>>(n, P, parity ? 1 : 0, pc, d_C, d_w, scale,
                                                                             d_K, ldK);
}

void launch_oz_pack(const PairTable& t, int nbf, int R, const double* d_D, double* d_u, cudaStream_t st) {
  count_launch();
  oz::k_oz_pack<<<(unsigned)std::min<int64_t>((t.npair * R + 255) / 256, 152 * 16), 256, 0, st>>>(
      nbf, R, t.npair, t.pair_mu, t.pair_nu, d_D, d_u);
}

// C = A B^T over the segments; C rows are A rows (transpose_out: C^T).  symmetric: one segment, C square,
// both triangles written from the upper one.  Split partials hold c_rows x c_cols elements each.
lrtei_status oz_gemm(const OzMatrix& A, const OzMatrix& B, const std::vector<OzSegment>& segs, double* d_C, int64_t ldc,
                     bool transpose_out, bool symmetric, int64_t c_rows, int64_t c_cols, int* d_status, cudaStream_t st) {
  oz::Params p{};
  const int BN = B.tile;
  p.nseg = (int)segs.size();
  if (A.tile != 128 || (BN != 32 && BN != 128) || (BN == 32 && symmetric)) { set_error("oz_gemm: operand tiles of %d and %d rows", A.tile, B.tile); return LRTEI_ERR_ARG; }
  if (p.nseg < 1 || p.nseg > 8) { set_error("oz_gemm: 1 to 8 segments"); return LRTEI_ERR_ARG; }
  int max_ch = 1;
  for (int i = 0; i < p.nseg; ++i) {
    const OzSegment& s = segs[i];
    oz::Seg& o = p.seg[i];
    // the tiles start at a multiple of 128 rows of A; rows below a_row0 are computed and not stored
    const int m_lo = (int)(s.a_row0 % 128);
    if (m_lo && symmetric) { set_error("oz_gemm: symmetric products start at row 0"); return LRTEI_ERR_ARG; }
    o = {s.a_row0 - m_lo, s.b_row0, s.M + m_lo, s.N, s.c_off, p.nitems, s.a_k0,
         s.b_k0, s.k / 64, (int)((s.M + m_lo + 127) / 128), (int)((s.N + BN - 1) / BN), m_lo};
    max_ch = std::max(max_ch, o.nch);
    p.nitems += symmetric ? (int64_t)o.tiles_n * (o.tiles_n + 1) / 2 : (int64_t)o.tiles_m * o.tiles_n;
  }
  if (p.nitems == 0) return LRTEI_OK;
  p.splits = oz::pick_splits(p.nitems, max_ch, BN == 32 ? 1.5 : 6.0);
  double* part = nullptr;
  if (p.splits > 1) {
    cudaError_t e = scratch_alloc((void**)&part, sizeof(double) * (size_t)p.splits * c_rows * c_cols, st);
    if (e != cudaSuccess) {
      cudaGetLastError();
      set_error("oz_gemm: partial sums: %s", cudaGetErrorString(e));
      return LRTEI_ERR_ALLOC;
    }
  }
  p.symmetric = symmetric ? 1 : 0;
  p.transpose_out = transpose_out ? 1 : 0;
  p.a = reinterpret_cast<const uint8_t*>(A.d);
  p.b = reinterpret_cast<const uint8_t*>(B.d);
  p.a_steps = A.kpad / oz::KB;
  p.b_steps = B.kpad / oz::KB;
  p.ea = A.expo;
  p.eb = B.expo;
  p.C = part ? part : d_C;
  p.ldc = part ? c_cols : ldc;
  p.split_stride = part ? c_rows * c_cols : 0;
  for (int i = 0; i < p.nseg; ++i) p.seg[i].c_off -= transpose_out ? p.seg[i].m_lo : p.seg[i].m_lo * p.ldc;
  p.status = d_status;
  // doubles per access that every row of C allows (segments start at multiples of 64 columns)
  p.align = (p.ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(p.C) & 31) == 0) ? 4
            : (p.ldc % 2 == 0 && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0) ? 2 : 1;
  {
    const char* v = getenv("LRTEI_TEST_STALL_CYCLES");
    p.test_stall = (v && *v) ? std::max(0LL, atoll(v)) : 0;
  }
  lrtei_status s;
  {
    ProfScope ps("gemm_fp64", st);
    if (BN == 32) {
      s = oz::launch<32, 0, 6>(p, st);
    } else {
      s = oz::launch<128, 4, 2>(p, st);
      p.accumulate = 1;
      if (s == LRTEI_OK) s = oz::launch<128, 2, 2>(p, st);
      p.mirror = (symmetric && !part) ? 1 : 0;
      if (s == LRTEI_OK) s = oz::launch<128, 0, 2>(p, st);
    }
  }
  if (part) {
    if (s == LRTEI_OK) {
      if (symmetric) {
        const unsigned g = (unsigned)((c_cols + 31) / 32);
        count_launch();
        oz::k_oz_reduce_sym<<<dim3(g, g), dim3(32, 8), 0, st>>>(part, p.splits, c_cols, d_C, ldc);
      } else {
        launch_reduce_splits(part, p.splits, c_rows * c_cols, c_rows, c_cols, c_cols, d_C, ldc, st);
      }
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) s = cuda_fail(e, "oz_gemm reduction");
    }
    cudaFreeAsync(part, st);
  }
  return s;
}

}  // namespace lrtei
