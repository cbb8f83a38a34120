// k_ozaki.cu -- FP64 products of the factored form on the tensor cores, by error-free slicing
// (Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication", 2012).
//
// C = A B^T for FP64 matrices (rows x K, K contiguous).  Every row is scaled by a power of two and cut
// into eight balanced base-512 digits held exactly in FP16:
//   x = 2^e sum_i d_i 2^(-9 (i + 1)),  |d_i| <= 256, |x| < 2^(e - 1),
// 71 bits below the binade of the row's largest element: an element down to 2^-18 of it is held as FP64 holds it.
// The 36 digit products d_i d_j with level i + j <= 7 are formed on the tensor cores; the dropped ones are below
// 2^-66 of the row maxima.  With six digits and 21 products the error had the size of FP64's in the norm only: small
// elements of B, contractions of the small elements of two rows (the high multipoles of one charge distribution with
// those of another), were off by up to 1e-9 where FP64 is by 1e-12.  Element by element, two atoms of s, p and d
// functions, elements above 1e-10 of the largest, 99.9 % quantile / maximum of the relative error of B against 80-bit
// sums from the same factors: FP64 8.9e-15 / 1.1e-13, six digits 1.6e-11 / 9.4e-10, seven 3.3e-14 / 8.3e-13, eight
// 3.1e-15 / 7.3e-14; on a wider molecule FP64 8.8e-13 / 1.6e-11, seven 1.2e-12 / 9.3e-12, eight 4.1e-13 / 6.7e-12.
//
// The FP32 sum of one level over a chunk of K is exact, at most (level + 1) columns 2^16 <= 2^24: chunks of 128 columns
// for levels 0 and 1, 64 for 2 and 3, 32 for 4 and 5 and for all eight of the skinny product.  In the wide products
// levels 6 and 7, which weigh 2^-54 and less, stay FP32 sums.  Chunks are added in int32 (K is split before they could
// overflow, oz_splits.h), and two levels make one integer X = 512 L_even + L_odd, so a result carries one rounding per
// pair of levels.  Rows holding a NaN or an infinity are marked in their exponent and give NaN.
//
// Why: this device runs 1.2 TFLOP/s in FP64 and 1 900 in FP16; 36 products leave ~53.
//
// Wide products (B_u = G F_u^T and G = F_u K) run as four launches (levels 6-7, 4-5, 2-3, 0-1; smallest
// first, the later ones adding to C): 128 x 128 tiles, two FP32 accumulators double-buffered in the
// 512 TMEM columns, and registers for one 64-bit sum per element allow two levels at a time.  Skinny products
// (J-builds, N <= 32 columns a tile) keep all eight levels in TMEM (2 x 8 x 32 columns) and read their operand once.
// Measured: FP64 B of 60 functions (n = 24, P = 32) 187 ms on the CUDA cores, 2.55 with six digits, 4.23 with eight;
// J-build of 16 densities, 120 functions, 32.7 (6.2 with the kernels of k_jfp64.cu), 0.47 and 0.61 ms, the products
// reading their operand at 6.5 TB/s.
#include <cuda_fp16.h>

#include "oz_splits.h"
#include "tc_gemm.h"

namespace lrtei {
namespace oz {

using tcg::KB;

// Levels [LV0, LV0 + NLV) of the digit products, digits below NP of each operand.
template <int BN_, int LV0, int NLV>
struct Levels {
  static constexpr int BN = BN_, NP = LV0 + NLV, PT = kOzSlices, NACC = NLV;
  static constexpr bool BF16 = false, ACCUM = NLV == 2, LIST = false;
  static constexpr bool FLT = LV0 >= 6;  // FP32 running sums (level 6 weighs 2^-54)
  // K blocks per stage: one barrier round per 30 KB or more
  static constexpr int STEP = NP * (128 + BN) * 32, KS = STEP >= 30 * 1024 ? 1 : STEP >= 16 * 1024 ? 2 : 4;
  static constexpr int UNIT = 4;  // 64-deep split units
  // chunk, in 16-deep steps: exactness (top of the file), which levels 6 and 7 of the wide products do without
  static constexpr int CHUNK = NLV == 8 || LV0 == 4 ? 2 : LV0 == 2 ? 4 : LV0 == 0 ? 8 : 16;
  static_assert(FLT || (LV0 + NLV) * CHUNK * 16 * 65536 <= 1 << 24, "a chunk's sums are exact in FP32");

  static __device__ __forceinline__ void mma(uint32_t d0, uint64_t a, uint64_t b, uint32_t idesc, uint32_t first) {
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      // A digit i meets the B digits j with LV0 <= i + j < LV0 + NLV (consecutive, so that the A slice is read
      // from shared memory once)
      const int j0 = LV0 > i ? LV0 - i : 0, j1 = NP - i;
#pragma unroll
      for (int j = j0; j < j1; ++j) {
        const uint32_t d = d0 + (uint32_t)((i + j - LV0) * BN);
        const uint64_t ad = a + (uint64_t)((i * 128 * 32) >> 4), bd = b + (uint64_t)((j * BN * 32) >> 4);
        const uint32_t acc = i == 0 ? first : 1u;
        if (j1 - j0 == 1) tc::mma_bf16(d, ad, bd, idesc, acc);
        else if (j == j0) tc::mma_bf16_a<tc::ACol::fill>(d, ad, bd, idesc, acc);
        else if (j == j1 - 1) tc::mma_bf16_a<tc::ACol::lastuse>(d, ad, bd, idesc, acc);
        else tc::mma_bf16_a<tc::ACol::use>(d, ad, bd, idesc, acc);
      }
    }
  }

  template <int QC>
  struct Sums {
    using Sum = typename std::conditional<FLT, float, int>::type;
    Sum T[NLV][QC];
    __device__ __forceinline__ void clear() {
#pragma unroll
      for (int x = 0; x < NLV; ++x)
#pragma unroll
        for (int j = 0; j < QC; ++j) T[x][j] = 0;
    }
    __device__ __forceinline__ void drain(uint32_t tbase) {
#pragma unroll
      for (int x = 0; x < NLV; x += 2)
#pragma unroll
        for (int j0 = 0; j0 < QC; j0 += 8) {
          uint32_t r[8], q[8];
          tc::tmem_ld8(tbase + x * BN + j0, r);
          tc::tmem_ld8(tbase + (x + 1) * BN + j0, q);
          tc::tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if constexpr (FLT) {
              T[x][j0 + j] += __uint_as_float(r[j]);
              T[x + 1][j0 + j] += __uint_as_float(q[j]);
            } else {
              T[x][j0 + j] += __float2int_rn(__uint_as_float(r[j]));
              T[x + 1][j0 + j] += __float2int_rn(__uint_as_float(q[j]));
            }
          }
        }
    }
    template <int C>
    __device__ __forceinline__ void hold(int j0) {
      if constexpr (!FLT) {
#pragma unroll
        for (int j = 0; j < C; ++j)
#pragma unroll
          for (int x = 0; x < NLV; ++x) asm volatile("" : "+r"(T[x][j0 + j]) : : "memory");
      }
    }
    // Sum over the pairs of levels of (512 T_even + T_odd) 2^(ea + eb - 9 (level + 3)).
    __device__ __forceinline__ double value(int j, int k, double) const {
      double sum = 0.0;
#pragma unroll
      for (int x = NLV - 2; x >= 0; x -= 2) {
        long long X;
        if constexpr (FLT) X = __float2ll_rn(T[x][j]) * 512 + __float2ll_rn(T[x + 1][j]);
        else X = (long long)T[x][j] * 512 + T[x + 1][j];
        const double t = tcg::int_ldexp(X, k - 9 * (LV0 + x + 3));
        sum = x == NLV - 2 ? t : sum + t;
      }
      return k >= kOzBad / 2 ? __longlong_as_double(0x7FF8000000000000LL) : sum;
    }
  };
};

// ---------------------------------------------------------------- slicing
// Digit tiles: `tile` rows x 16 columns x 8 planes are contiguous (each plane's 32-byte rows in the 32-byte
// swizzle of shared memory), K block after K block, so that a stage is one contiguous copy per operand
// and block, and as shallow as the pipeline wants it.
// Destination row i holds source row rowinv[i] (NULL: i), destination column j source column colinv[j]
// (NULL: j for j < k); -1 gives zeros.  colexp (NULL: none): source column j comes times 2^-colexp[j].  One block per
// row: the largest magnitude, then the digits.
// Bound by instructions, and by the conversion unit (16 a clock and SM) where the digits pass through it twice: six
// planes of 1830 rows of 13824 took 134 us so, 118 with FP16 integers made by an addition to 1536 and the row staged in
// shared memory (`staged`; longer rows are read twice), and eight planes take 144 (0.6 GB); the three operands of 16
// densities of 120 functions 35, 27 and, in eight planes, 34 us.
// The digits of q = round(x 2^(72 - e)), |q| <= 2^71, as two words of four: q = hi 2^36 + lo with lo between -256 and
// 255 times 1 + 512 + 512^2 + 512^3; a word plus 256 times its digits' weights (without the first digit's) has the
// digits plus 256 as its 9-bit fields, the first one as it is.
struct Digits {
  long long hi, lo;
};
constexpr long long kBias3 = 256LL * (1 + (1LL << 9) + (1LL << 18)), kBias4 = kBias3 + (256LL << 27);

// The digits of an element of a row whose largest biased exponent is E.
__device__ __forceinline__ Digits biased_digits(unsigned long long b, int E) {
  const int Ex = (int)((b >> 52) & 0x7FF), sh = E - Ex;  // |q| = m 2^(18 - sh)
  unsigned long long m = (b & ((1ULL << 52) - 1)) | (1ULL << 52);
  if (sh > 18) m = sh > 72 ? 0 : (m + (1ULL << (sh - 19))) >> (sh - 18);
  if (Ex == 0) m = 0;
  const int up = max(18 - sh, 0);
  const long long neg = (long long)b >> 63;  // 0 or -1
  const long long h = (long long)(m >> (36 - up)), l = (long long)((m << up) & ((1ULL << 36) - 1));
  const long long lo = ((l ^ neg) - neg) + kBias4;
  return {((h ^ neg) - neg) + (lo >> 36) + kBias3, lo};
}

// Plane s of two neighbouring elements: small integers as FP16, through 1536 + i (whose last place is 1).
template <int S>
__device__ __forceinline__ uint32_t digit_pair(const Digits& u, const Digits& v) {
  constexpr int SH = 9 * (3 - S % 4);
  const long long x = S < 4 ? u.hi : u.lo, y = S < 4 ? v.hi : v.lo;
  uint32_t w;
  if constexpr (S == 0) w = 0x66006600u + (uint32_t)(int)(x >> SH) + ((uint32_t)(int)(y >> SH) << 16);
  else w = 0x65006500u + ((uint32_t)(x >> SH) & 511u) + (((uint32_t)(y >> SH) & 511u) << 16);
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __half2half2(__ushort_as_half(0x6600)));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// x 2^-s for |x| < 2^s, zero below the normal range.
__device__ __forceinline__ double scaled_down(double x, int s) {
  const long long b = __double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF) - s;
  if (((b >> 52) & 0x7FF) == 0 || E <= 0) return 0.0;
  return __longlong_as_double(b - s * (1LL << 52));
}

__global__ void __launch_bounds__(512) k_oz_split(const double* __restrict__ src, int64_t k, int64_t ld, int64_t kpad,
                                                  int tile, int staged, const int* __restrict__ rowinv,
                                                  const int* __restrict__ colinv, const int* __restrict__ colexp,
                                                  uint16_t* __restrict__ d, int* __restrict__ expo) {
  extern __shared__ double row[];
  __shared__ uint32_t red[32];
  const int64_t i = blockIdx.x;
  const int64_t r = rowinv ? rowinv[i] : i;
  const double* x = src + r * ld;
  uint32_t mx = 0;  // the exponent's word is enough
  if (r >= 0) {
#pragma unroll 4
    for (int64_t j = threadIdx.x; j < k; j += blockDim.x) {
      const double v = colexp ? scaled_down(x[j], colexp[j]) : x[j];
      if (staged) row[j] = v;
      mx = max(mx, tc::magnitude(v));
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  const unsigned lane = threadIdx.x & 31;
  mx = __reduce_max_sync(0xffffffffu, lane < (blockDim.x >> 5) ? red[lane] : 0u);
  const int E = (int)(mx >> 20);  // biased exponent of the largest magnitude; 0: zero row, 0x7FF: not finite
  const bool live = E > 0 && E < 0x7FF;
  if (threadIdx.x == 0) expo[i] = E == 0x7FF ? kOzBad : live ? E - 1021 : 0;
  if (staged) x = row;
  for (int64_t j = 4 * (int64_t)threadIdx.x; j < kpad; j += 4 * (int64_t)blockDim.x) {
    Digits q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t c = colinv ? colinv[j + e] : (j + e < k ? j + e : -1);
      double v = live && c >= 0 ? x[c] : 0.0;
      if (colexp && !staged && c >= 0) v = scaled_down(v, colexp[c]);
      q[e] = biased_digits((unsigned long long)__double_as_longlong(v), E);
    }
    const int rr = (int)(i % tile), kk = (int)(j % KB) * 2;  // byte inside the 32-byte row; 16-byte pieces swizzled
    uint8_t* o = reinterpret_cast<uint8_t*>(d) + ((i / tile) * (kpad / KB) + j / KB) * (int64_t)(kOzSlices * tile * 32) +
                 rr * 32 + (kk ^ (((rr >> 2) & 1) << 4));
    const int step = tile * 32;
    *reinterpret_cast<uint2*>(o) = make_uint2(digit_pair<0>(q[0], q[1]), digit_pair<0>(q[2], q[3]));
    *reinterpret_cast<uint2*>(o + step) = make_uint2(digit_pair<1>(q[0], q[1]), digit_pair<1>(q[2], q[3]));
    *reinterpret_cast<uint2*>(o + 2 * step) = make_uint2(digit_pair<2>(q[0], q[1]), digit_pair<2>(q[2], q[3]));
    *reinterpret_cast<uint2*>(o + 3 * step) = make_uint2(digit_pair<3>(q[0], q[1]), digit_pair<3>(q[2], q[3]));
    *reinterpret_cast<uint2*>(o + 4 * step) = make_uint2(digit_pair<4>(q[0], q[1]), digit_pair<4>(q[2], q[3]));
    *reinterpret_cast<uint2*>(o + 5 * step) = make_uint2(digit_pair<5>(q[0], q[1]), digit_pair<5>(q[2], q[3]));
    *reinterpret_cast<uint2*>(o + 6 * step) = make_uint2(digit_pair<6>(q[0], q[1]), digit_pair<6>(q[2], q[3]));
    *reinterpret_cast<uint2*>(o + 7 * step) = make_uint2(digit_pair<7>(q[0], q[1]), digit_pair<7>(q[2], q[3]));
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

// Unique-pair densities, one row per density, in the units of the pairs' rows of F_u: u[q][r] =
// D_q(mu, nu) (2 - [mu == nu]) 2^expo[r], to meet F_u^T with its columns scaled by 2^-expo.  Unscaled, a row of F_u^T
// holds a pair of small overlap far below its largest one: a density on such pairs alone gave J off by 1e-12 of its terms.
__global__ void k_oz_pack(int nbf, int R, int64_t npair, const int* __restrict__ pair_mu,
                          const int* __restrict__ pair_nu, const int* __restrict__ expo, const double* __restrict__ D,
                          double* __restrict__ u) {
  const int64_t total = npair * R;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t % npair, q = t / npair;
    const int mu = pair_mu[r], nu = pair_nu[r];
    const double v = D[q * nbf * nbf + (int64_t)mu * nbf + nu];
    u[t] = scalbn(v, expo[r] + (mu == nu ? 0 : 1));
  }
}
}  // namespace oz

// ---------------------------------------------------------------- host side
void launch_oz_split(const double* d_src, int64_t k, int64_t ld, const int* d_rowinv, const int* d_colinv,
                     const int* d_colexp, OzMatrix& m, cudaStream_t st) {
  if (m.rows <= 0) return;
  constexpr int64_t most = 28000;  // columns that fit shared memory
  shared_opt_in<&oz::k_oz_split>(sizeof(double) * most);  // a refusal shows at the launch
  const int staged = k <= most ? 1 : 0;
  count_launch();
  oz::k_oz_split<<<(unsigned)m.rows, m.rows < 2 * 152 || k > 4096 ? 512 : 256, staged ? sizeof(double) * (size_t)k : 0, st>>>(
      d_src, k, ld, m.kpad, m.tile, staged, d_rowinv, d_colinv, d_colexp, m.d, m.expo);
}

void launch_oz_build_K(int n, int P, bool parity, const ParityClasses& pc, const double* d_C, const double* d_w,
                       double scale, double* d_K, int64_t ldK, cudaStream_t st) {
  count_launch();
  oz::k_oz_build_K<<<dim3((unsigned)(n * n), (unsigned)(n * n)), 256, 0, st>>>(n, P, parity ? 1 : 0, pc, d_C, d_w, scale,
                                                                             d_K, ldK);
}

void launch_oz_pack(const PairTable& t, int nbf, int R, const double* d_D, const int* d_expo, double* d_u, cudaStream_t st) {
  count_launch();
  oz::k_oz_pack<<<(unsigned)std::min<int64_t>((t.npair * R + 255) / 256, 152 * 16), 256, 0, st>>>(
      nbf, R, t.npair, t.pair_mu, t.pair_nu, d_expo, d_D, d_u);
}

// C = A B^T over the segments; C rows are A rows (transpose_out: C^T).  symmetric: one segment, C square,
// both triangles written from the upper one.  Split partials hold c_rows x c_cols elements each.
lrtei_status oz_gemm(const OzMatrix& A, const OzMatrix& B, const std::vector<OzSegment>& segs, double* d_C, int64_t ldc,
                     bool transpose_out, bool symmetric, int64_t c_rows, int64_t c_cols, int* d_status, cudaStream_t st) {
  tcg::Params p{};
  const int BN = B.tile;
  p.nseg = (int)segs.size();
  if (A.tile != 128 || (BN != 32 && BN != 128) || (BN == 32 && symmetric)) {
    set_error("oz_gemm: operand tiles of %d and %d rows", A.tile, B.tile);
    return LRTEI_ERR_ARG;
  }
  if (p.nseg < 1 || p.nseg > 8) { set_error("oz_gemm: 1 to 8 segments"); return LRTEI_ERR_ARG; }
  int max_units = 1;
  for (int i = 0; i < p.nseg; ++i) {
    const OzSegment& s = segs[i];
    tcg::Seg& o = p.seg[i];
    // the tiles start at a multiple of 128 rows of A; rows below a_row0 are computed and not stored
    const int m_lo = (int)(s.a_row0 % 128);
    if (m_lo && symmetric) { set_error("oz_gemm: symmetric products start at row 0"); return LRTEI_ERR_ARG; }
    o = {s.a_row0 - m_lo, s.b_row0, s.M + m_lo, s.N, s.c_off, p.nitems, s.a_k0 / tcg::KB, s.b_k0 / tcg::KB, s.k / 64,
         (int)((s.M + m_lo + 127) / 128), (int)((s.N + BN - 1) / BN), m_lo, s.k / tcg::KB, nullptr};
    max_units = std::max(max_units, o.units);
    p.nitems += symmetric ? (int64_t)o.tiles_n * (o.tiles_n + 1) / 2 : (int64_t)o.tiles_m * o.tiles_n;
  }
  if (p.nitems == 0) return LRTEI_OK;
  p.blk0 = 0;
  p.blk1 = p.nb = p.seg[0].tiles_n;
  p.splits = oz::product_splits(p.nitems, max_units, BN == 32);
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
  p.a_steps = A.kpad / tcg::KB;
  p.b_steps = B.kpad / tcg::KB;
  p.b_tile = BN;
  p.ea = A.expo;
  p.eb = B.expo;
  p.C = part ? part : d_C;
  p.ldc = part ? c_cols : ldc;
  p.split_stride = part ? c_rows * c_cols : 0;
  for (int i = 0; i < p.nseg; ++i) p.seg[i].c_off -= transpose_out ? p.seg[i].m_lo : p.seg[i].m_lo * p.ldc;
  p.status = d_status;
  p.align = tc::store_align(p.C, p.ldc);
  p.test_stall = tcg::test_stall_cycles();
  lrtei_status s;
  {
    ProfScope ps("gemm_fp64", st);
    if (BN == 32) {
      s = tcg::launch<oz::Levels<32, 0, 8>>(p, st);
    } else {
      s = tcg::launch<oz::Levels<128, 6, 2>>(p, st);
      p.accumulate = 1;
      if (s == LRTEI_OK) s = tcg::launch<oz::Levels<128, 4, 2>>(p, st);
      if (s == LRTEI_OK) s = tcg::launch<oz::Levels<128, 2, 2>>(p, st);
      p.mirror = (symmetric && !part) ? 1 : 0;
      if (s == LRTEI_OK) s = tcg::launch<oz::Levels<128, 0, 2>>(p, st);
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
