// k_slices.cu -- FP64 rows to the operand planes of the tensor-core GEMM (three integer slices
// held exactly in FP16 and one exponent per row, or one BF16 plane), plus the transpose and
// split-K reduction kernels around the skinny GEMMs of the J-build.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdlib.h>

#include <algorithm>

#include "lrtei_internal.h"
#include "tc_common.h"

namespace cg = cooperative_groups;

namespace lrtei {
namespace tc {

// The block's largest magnitude, on all its threads (red: a word per warp).
__device__ __forceinline__ uint32_t block_max(uint32_t mx, uint32_t* red) {
  mx = __reduce_max_sync(0xffffffffu, mx);
  const unsigned lane = threadIdx.x & 31;
  if (lane == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  return __reduce_max_sync(0xffffffffu, lane < (blockDim.x >> 5) ? red[lane] : 0u);
}

// Where the eight consecutive columns j .. j + 7 (j a multiple of 8) of row i go: tiles of `tile` rows x 16
// columns x `planes` planes, 32-byte rows whose two 16-byte pieces are swapped in every other group of
// four rows (the 32-byte swizzle of shared memory, tc_gemm.h).  In units of 16-bit elements.
__device__ __forceinline__ int64_t piece(int64_t i, int64_t j, int tile, int64_t kpad, int planes) {
  const int rr = (int)(i % tile);
  return ((i / tile) * (kpad / 16) + j / 16) * (int64_t)(planes * tile * 16) + rr * 16 +
         ((int)((j >> 3) & 1) ^ ((rr >> 2) & 1)) * 8;
}

__device__ __forceinline__ uint4 pack8(const uint16_t (&h)[8]) {
  return make_uint4(h[0] | (uint32_t)h[1] << 16, h[2] | (uint32_t)h[3] << 16, h[4] | (uint32_t)h[5] << 16,
                    h[6] | (uint32_t)h[7] << 16);
}

// The three slice planes of eight elements (k: live columns of the row, nz: the row is not zero).
__device__ __forceinline__ void store_slices(const double (&v)[8], int e, bool nz, int64_t i, int64_t j, int64_t k,
                                             int tile, int64_t kpad, uint16_t* __restrict__ d) {
  uint32_t p0[4], p1[4], p2[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    slice_pair(v[2 * u], v[2 * u + 1], e, j + 2 * u < k && nz, j + 2 * u + 1 < k && nz, p0[u], p1[u], p2[u]);
  uint16_t* o = d + piece(i, j, tile, kpad, 3);
  *reinterpret_cast<uint4*>(o) = make_uint4(p0[0], p0[1], p0[2], p0[3]);
  *reinterpret_cast<uint4*>(o + tile * 16) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
  *reinterpret_cast<uint4*>(o + 2 * tile * 16) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
}

// Columns j .. j + 7 of a row: 16-byte loads where the row allows them, zeros beyond k; map (may be NULL):
// the source column of each column.
__device__ __forceinline__ void load8(const double* __restrict__ x, int64_t j, int64_t k, bool vec,
                                      const int* __restrict__ map, double (&v)[8]) {
  if (map) {
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = j + u < k ? x[map[j + u]] : 0.0;
  } else if (vec && j + 7 < k) {
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      const double2 a = *reinterpret_cast<const double2*>(x + j + u);
      v[u] = a.x;
      v[u + 1] = a.y;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = j + u < k ? x[j + u] : 0.0;
  }
}

__device__ __forceinline__ uint32_t max_mag(const double (&v)[8], uint32_t mx) {
#pragma unroll
  for (int u = 0; u < 8; ++u) mx = max(mx, magnitude(v[u]));
  return mx;
}

// A row staged in shared memory (16-byte aligned) into columns j0 .. j0 + n of operand row i, j0 a multiple of 8 and n
// of 2; zeros from its column k on.  A thread takes two neighbouring columns: the reads have no bank conflicts
// (eight columns of one thread are 16-way ones) and a warp's stores fill whole sectors.  16290 rows of 13824 (3.15 GB):
// 0.84 ms by eight columns, 0.61 by two; 1035 rows of 2197 12.8 us, 9.3.
__device__ __forceinline__ void store_row(const double* __restrict__ row, const int* __restrict__ map, int64_t k, int e,
                                          int64_t i, int64_t j0, int64_t n, int tile, int64_t kpad,
                                          uint16_t* __restrict__ d) {
  const bool nz = e != kZeroRowExpo;
  const int rr = (int)(i % tile), sw = (rr >> 2) & 1;
  uint16_t* base = d + (i / tile) * (kpad / 16) * (int64_t)(3 * tile * 16) + rr * 16;
  for (int j = 2 * (int)threadIdx.x; j < n; j += 2 * (int)blockDim.x) {
    const bool l0 = nz && j < k, l1 = nz && j + 1 < k;
    double x = 0.0, y = 0.0;
    if (map) {
      if (l0) x = row[map[j]];
      if (l1) y = row[map[j + 1]];
    } else if (l1) {
      const double2 t = *reinterpret_cast<const double2*>(row + j);
      x = t.x;
      y = t.y;
    } else if (l0) {
      x = row[j];
    }
    uint32_t p0, p1, p2;
    slice_pair(x, y, e, l0, l1, p0, p1, p2);
    const int64_t c = j0 + j;
    uint16_t* o = base + (c >> 4) * (int64_t)(3 * tile * 16) + ((int)((c >> 3) & 1) ^ sw) * 8 + (int)(c & 7);
    *reinterpret_cast<uint32_t*>(o) = p0;
    *reinterpret_cast<uint32_t*>(o + tile * 16) = p1;
    *reinterpret_cast<uint32_t*>(o + 2 * tile * 16) = p2;
  }
}

// Short rows (padded length at most 256): one warp per row, eight consecutive elements per lane.
__global__ void __launch_bounds__(256) k_split_rows_warp(const double* __restrict__ src, int64_t rows, int64_t k,
                                                         int64_t ld, int64_t kpad, int tile,
                                                         const int* __restrict__ map, uint16_t* __restrict__ d,
                                                         int* __restrict__ expo) {
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= rows) return;  // the whole warp: r is the same on its lanes
  const double* x = src + r * ld;
  const bool vec = (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  const int64_t i0 = 8 * (int64_t)lane;
  double v[8];
  load8(x, i0, k, vec, map, v);
  const int e = slice_exponent(__reduce_max_sync(0xffffffffu, max_mag(v, 0)));
  if (lane == 0) expo[r] = e;
  if (i0 < kpad) store_slices(v, e, e != kZeroRowExpo, r, i0, k, tile, kpad, d);
}

// One block per row, the row staged in shared memory (rows of up to kSplitCols columns): read once, by one
// bulk copy where its address allows, and gathered through the map from there (a class order's eight
// neighbours are two runs of four, one element per sector and lane from global memory).
constexpr int64_t kSplitCols = 28000;
__global__ void __launch_bounds__(512) k_split_rows(const double* __restrict__ src, int64_t cols, int64_t k, int64_t ld,
                                                    int64_t kpad, int tile, int bulk, const int* __restrict__ map,
                                                    uint16_t* __restrict__ d, int* __restrict__ expo, int* status,
                                                    long long stall) {
  extern __shared__ __align__(16) double row[];  // cols: the source row's columns (k without a map)
  __shared__ uint32_t red[32];
  __shared__ uint64_t bar;
  const int64_t r = blockIdx.x;
  const double* x = src + r * ld;
  const int nc = (int)cols;
  uint32_t mx = 0;
  if (bulk) {
    if (threadIdx.x == 0) {
      mbar_init(&bar, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      mbar_arrive_expect_tx(&bar, (uint32_t)(nc * 8));
      bulk_load(row, x, (uint32_t)(nc * 8), &bar);
    }
    __syncthreads();
    wait_staged(&bar, status, stall);
#pragma unroll 4
    for (int i = threadIdx.x; i < nc; i += blockDim.x) mx = max(mx, magnitude(row[i]));
  } else {
#pragma unroll 4
    for (int i = threadIdx.x; i < nc; i += blockDim.x) {
      const double v = x[i];
      row[i] = v;
      mx = max(mx, magnitude(v));
    }
  }
  const int e = slice_exponent(block_max(mx, red));  // (synchronises: the whole row is staged)
  if (threadIdx.x == 0) expo[r] = e;
  store_row(row, map, k, e, r, 0, kpad, tile, kpad, d);
}

// Longer rows: two passes, the second from L2.
__global__ void __launch_bounds__(256) k_split_rows_long(const double* __restrict__ src, int64_t k, int64_t ld,
                                                         int64_t kpad, int tile, const int* __restrict__ map,
                                                         uint16_t* __restrict__ d, int* __restrict__ expo) {
  __shared__ uint32_t red[32];
  const int64_t r = blockIdx.x;
  const double* x = src + r * ld;
  const bool vec = (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
  uint32_t mx = 0;
  double v[8];
  for (int64_t j = 8 * (int64_t)threadIdx.x; j < k; j += 2048) {
    load8(x, j, k, vec, map, v);
    mx = max_mag(v, mx);
  }
  const int e = slice_exponent(block_max(mx, red));
  const bool nz = e != kZeroRowExpo;
  if (threadIdx.x == 0) expo[r] = e;
  for (int64_t j = 8 * (int64_t)threadIdx.x; j < kpad; j += 2048) {
    load8(x, j, k, vec, map, v);
    store_slices(v, e, nz, r, j, k, tile, kpad, d);
  }
}

// Columns j .. j + 7 of row r: of FP64 rows, or of packed densities D_r(mu, nu) (mu == nu ? 1 : 2).
struct RowSource {
  const double* src;
  int64_t ld;
  const int* map;
  __device__ __forceinline__ void load(int64_t r, int64_t j, int64_t k, double (&v)[8]) const {
    const bool vec = (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0;
    load8(src + r * ld, j, k, vec, map, v);
  }
};
struct DensitySource {
  const double* D;
  int nbf;
  const int *mu, *nu;
  __device__ __forceinline__ void load(int64_t r, int64_t j, int64_t k, double (&v)[8]) const {
    const double* x = D + r * nbf * nbf;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = 0.0;
      if (j + u < k) {
        const int a = mu[j + u], b = nu[j + u];
        v[u] = x[a * nbf + b] * (a == b ? 1.0 : 2.0);
      }
    }
  }
};

// Few long rows (fewer rows than SMs, e.g. the R density rows of a J-build): a cluster of
// kSplitCluster CTAs per row, each taking an eighth of the padded row.  Every CTA reduces the
// magnitude bits over its share, the cluster combines the eight maxima through distributed shared
// memory, and each CTA slices its share with the row's exponent: the exponent and the slices are
// those of the one-block-per-row kernels.  A share of one step stays in registers between the two.
// 32 densities of 180 functions: 15.5 us packed, transposed and sliced by three kernels, 8.8 from the densities.
constexpr int kSplitCluster = 8;
template <class Source>
__global__ void __cluster_dims__(kSplitCluster, 1, 1) __launch_bounds__(256)
    k_split_rows_cluster(Source src, int64_t k, int64_t kpad, int tile, uint16_t* __restrict__ d,
                         int* __restrict__ expo) {
  __shared__ uint32_t red[32];
  __shared__ uint32_t share;
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned rank = cluster.block_rank();
  const int64_t r = blockIdx.y;
  const int64_t per = (kpad / 8 + kSplitCluster - 1) / kSplitCluster * 8;
  const int64_t c0 = (int64_t)rank * per, c1 = min(kpad, c0 + per);
  uint32_t mx = 0;
  double v[8];
  for (int64_t j = c0 + 8 * (int64_t)threadIdx.x; j < c1; j += 8 * (int64_t)blockDim.x) {
    src.load(r, j, k, v);
    mx = max_mag(v, mx);
  }
  mx = block_max(mx, red);
  if (threadIdx.x == 0) share = mx;
  cluster.sync();  // every CTA's share is written
  uint32_t all = 0;
  for (int q = 0; q < kSplitCluster; ++q) all = max(all, *cluster.map_shared_rank(&share, q));
  cluster.sync();  // every CTA has read the shares before any of them exits
  const int e = slice_exponent(all);
  const bool nz = e != kZeroRowExpo;
  if (rank == 0 && threadIdx.x == 0) expo[r] = e;
  const bool once = per <= 8 * (int64_t)blockDim.x;
  for (int64_t j = c0 + 8 * (int64_t)threadIdx.x; j < c1; j += 8 * (int64_t)blockDim.x) {
    if (!once) src.load(r, j, k, v);
    store_slices(v, e, nz, r, j, k, tile, kpad, d);
  }
}

// ---- operands of the long-range exchange, sliced where they lie (no transposed or permuted FP64 copies)
// Rows (mu, m) of MT, columns la: F_u(pair(mu, la), m), N_b <= 256 columns.  One CTA per mu and 32 columns m of
// F_u: the rows of F_u are read along m into shared memory, a column per lane, which also takes its maximum; then the
// slices are stored.  Blocks beyond the last column but one are not read by the products and stay unwritten.
// 2.5 M rows of 180: 3.3 ms through a gathered 3.6 GB copy, 1.67 with a warp per row maximum, 1.23 now (6.5 GB).
__global__ void __launch_bounds__(256) k_split_MT(int nbf, int64_t n3, const double* __restrict__ F, int64_t ldF,
                                                  int64_t kpad, int kuse, int tile, uint16_t* __restrict__ d,
                                                  int* __restrict__ expo) {
  extern __shared__ double t[];  // [nbf][33]
  __shared__ uint32_t top[8][32];
  __shared__ int re[32];  // row exponents
  const int mu = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t m0 = (int64_t)blockIdx.x * 32;
  const double* src = F + m0 + lane;
  const bool in = m0 + lane < n3;
  uint32_t mx = 0;
  for (int l0 = warp; l0 < nbf; l0 += 64) {  // eight rows' loads in flight per warp
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int la = l0 + 8 * u, lo = min(mu, la), hi = max(mu, la);
      const int r = lo * nbf - lo * (lo - 1) / 2 + (hi - lo);
      v[u] = la < nbf && in ? src[r * ldF] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      mx = max(mx, magnitude(v[u]));
      if (l0 + 8 * u < nbf) t[(l0 + 8 * u) * 33 + lane] = v[u];
    }
  }
  top[warp][lane] = mx;
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) mx = max(mx, top[w][lane]);
    re[lane] = slice_exponent(mx);
    if (in) expo[(int64_t)mu * n3 + m0 + lane] = re[lane];
  }
  __syncthreads();
  // a warp takes 16 rows of one 16-column block, a lane half a row of it: 512 contiguous bytes per plane and store
  const int nitem = kuse / 16 * 2;
  for (int it = warp; it < nitem; it += 8) {
    const int q = (it & 1) * 16 + (lane >> 1), c0 = (it >> 1) * 16 + (lane & 1) * 8;
    if (m0 + q >= n3) continue;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = c0 + u < nbf ? t[(c0 + u) * 33 + q] : 0.0;
    const int e = re[q];
    store_slices(v, e, e != kZeroRowExpo, (int64_t)mu * n3 + m0 + q, c0, nbf, tile, kpad, d);
  }
}

// Largest magnitude over the rows (j, mu), j < nj, of Z for each mu: the row maxima of Zp[mu][(j, m)].
__global__ void __launch_bounds__(256) k_orbital_max(int nbf, int64_t cols, int64_t ld, const double* __restrict__ Z,
                                                     uint32_t* __restrict__ mx) {
  __shared__ uint32_t red[32];
  const int64_t row = blockIdx.x;  // j nbf + mu
  const double* x = Z + row * ld;
  uint32_t v = 0;
#pragma unroll 8
  for (int64_t m = threadIdx.x; m < cols; m += 256) v = max(v, magnitude(x[m]));
  v = block_max(v, red);
  if (threadIdx.x == 0) atomicMax(mx + row % nbf, v);
}

// Zp[mu][(j, m)] = Z[(j, mu)][map[m]] into slices (n3 a multiple of 8): one CTA per row (j, mu), staged by one
// bulk copy, with the exponent of row mu: of its largest magnitude, or the largest of Z's row exponents (an exponent
// grows with the magnitude; saves the pass for the maxima where Z's rows are sliced anyway).
__global__ void __launch_bounds__(512) k_split_orbital_rows(int nbf, int64_t n3, int nj, int64_t cols, int64_t ld,
                                                            const double* __restrict__ Z, const int* __restrict__ map,
                                                            const uint32_t* __restrict__ mx,
                                                            const int* __restrict__ row_expo, int64_t k, int64_t kpad,
                                                            int tile, uint16_t* __restrict__ d, int* __restrict__ expo,
                                                            int* status, long long stall) {
  extern __shared__ __align__(16) double row[];
  __shared__ uint64_t bar;
  const int64_t i = blockIdx.x;
  const int j = (int)(i / nbf), mu = (int)(i % nbf);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_arrive_expect_tx(&bar, (uint32_t)(cols * 8));
    bulk_load(row, Z + i * ld, (uint32_t)(cols * 8), &bar);
  }
  int e = kZeroRowExpo;
  if (row_expo) {
    for (int q = threadIdx.x & 31; q < nj; q += 32) e = max(e, row_expo[(int64_t)q * nbf + mu]);
    e = __reduce_max_sync(0xffffffffu, e);
  } else {
    e = slice_exponent(mx[mu]);
  }
  if (j == 0 && threadIdx.x == 0) expo[mu] = e;
  __syncthreads();
  wait_staged(&bar, status, stall);
  store_row(row, map, n3, e, mu, (int64_t)j * n3, n3, tile, kpad, d);
  if ((int64_t)(j + 1) * n3 == k)  // the padding after the last orbital
    store_row(row, nullptr, 0, e, mu, k, kpad - k, tile, kpad, d);
}

// Plain BF16 operands: one rounded copy per element, exponent 8 so that the epilogue scale
// 2^(ea + eb - 16) is 1.
__global__ void k_plain_rows(const double* __restrict__ src, int64_t k, int64_t ld, int64_t kpad, int tile,
                             const int* __restrict__ map, uint16_t* __restrict__ d, int* __restrict__ expo) {
  const int64_t r = blockIdx.x;
  const double* x = src + r * ld;
  if (threadIdx.x == 0) expo[r] = 8;
  for (int64_t j = 8 * (int64_t)threadIdx.x; j < kpad; j += 8 * (int64_t)blockDim.x) {
    double v[8];
    uint16_t h[8];
    load8(x, j, k, false, map, v);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      __nv_bfloat16 b = __float2bfloat16_rn((float)v[u]);
      h[u] = *reinterpret_cast<uint16_t*>(&b);
    }
    *reinterpret_cast<uint4*>(d + piece(r, j, tile, kpad, 1)) = pack8(h);
  }
}

// 32 x 32 tiled transpose of an FP64 matrix: out (cols x rows) = in (rows x cols)^T.
__global__ void k_transpose(const double* __restrict__ in, int64_t rows, int64_t cols, int64_t ldi,
                            double* __restrict__ out, int64_t ldo) {
  __shared__ double t[32][33];
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int64_t r = r0 + i, c = c0 + threadIdx.x;
    if (r < rows && c < cols) t[i][threadIdx.x] = in[r * ldi + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int64_t c = c0 + i, r = r0 + threadIdx.x;
    if (r < rows && c < cols) out[c * ldo + r] = t[threadIdx.x][i];
  }
}

// Sum of split-K partials: out[i] = sum_s part[s * stride + i] (row-major rows x cols, ld).
__global__ void k_reduce_splits(const double* __restrict__ part, int splits, int64_t stride, int64_t rows,
                                int64_t cols, int64_t ld, double* __restrict__ out, int64_t ldo) {
  const int64_t total = rows * cols;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / cols, j = t % cols;
    double s = 0.0;
    for (int q = 0; q < splits; ++q) s += part[q * stride + i * ld + j];
    out[i * ldo + j] = s;
  }
}

// Few outputs of many parts (the exchange's N_b x N_b): a block per 32 outputs, eight threads to each.  75 x 75
// outputs of 128 parts: 30 us by a thread each, 5.3 here.
__global__ void __launch_bounds__(256) k_reduce_many(const double* __restrict__ part, int splits, int64_t stride,
                                                     int64_t rows, int64_t cols, int64_t ld, double* __restrict__ out,
                                                     int64_t ldo) {
  __shared__ double sum[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t t = blockIdx.x * (int64_t)32 + lane, i = t / cols, j = t % cols;
  double s = 0.0;
  if (i < rows) {
    const double* x = part + i * ld + j;
#pragma unroll 8
    for (int q = w; q < splits; q += 8) s += x[q * stride];
  }
  sum[w][lane] = s;
  __syncthreads();
  if (w == 0 && i < rows) {
#pragma unroll
    for (int q = 1; q < 8; ++q) s += sum[q][lane];
    out[i * ldo + j] = s;
  }
}

// LRTEI_TEST_STALL_STAGED_CYCLES (tests only): the kernels that stage rows also wait that long for what never comes.
static long long staged_stall_cycles() {
  const char* v = getenv("LRTEI_TEST_STALL_STAGED_CYCLES");
  return (v && *v) ? std::max(0LL, atoll(v)) : 0;
}

}  // namespace tc

bool launch_split_density(const PairTable& t, int nbf, int64_t R, const double* d_D, const SplitMatrix& m,
                          cudaStream_t st) {
  if (R <= 0 || R >= 4 * 152 || m.plain) return false;
  count_launch();
  tc::k_split_rows_cluster<<<dim3(tc::kSplitCluster, (unsigned)R), 256, 0, st>>>(
      tc::DensitySource{d_D, nbf, t.pair_mu, t.pair_nu}, t.npair, m.kpad, m.tile, m.d, m.expo);
  return true;
}

void launch_split_rows(const double* d_src, int64_t rows, int64_t k, int64_t ld, const SplitMatrix& m, const int* d_map,
                       int* d_status, cudaStream_t st) {
  if (rows <= 0) return;
  count_launch();
  if (m.plain) {
    tc::k_plain_rows<<<(unsigned)rows, 256, 0, st>>>(d_src, k, ld, m.kpad, m.tile, d_map, m.d, m.expo);
    return;
  }
  if (m.kpad <= 256) {  // short rows (e.g. the N_b-long rows of the exchange's MT): a warp per row
    tc::k_split_rows_warp<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(d_src, rows, k, ld, m.kpad, m.tile, d_map, m.d,
                                                                    m.expo);
    return;
  }
  // few long rows (fewer than four per SM, e.g. the R density rows of a J-build or the N_b rows of
  // the exchange's last product): eight CTAs per row
  if ((rows < 4 * 152 && k >= 8192) || (rows < 152 && k >= 2048)) {
    tc::k_split_rows_cluster<<<dim3(tc::kSplitCluster, (unsigned)rows), 256, 0, st>>>(
        tc::RowSource{d_src, ld, d_map}, k, m.kpad, m.tile, m.d, m.expo);
    return;
  }
  const int64_t cols = d_map ? ld : k;  // a mapped row's columns lie anywhere in it
  if (cols > tc::kSplitCols) {
    tc::k_split_rows_long<<<(unsigned)rows, 256, 0, st>>>(d_src, k, ld, m.kpad, m.tile, d_map, m.d, m.expo);
    return;
  }
  shared_opt_in<&tc::k_split_rows>(sizeof(double) * tc::kSplitCols);  // a refusal shows at the launch
  const int bulk = (cols % 2 == 0 && ld % 2 == 0 && (reinterpret_cast<uintptr_t>(d_src) & 15) == 0) ? 1 : 0;
  tc::k_split_rows<<<(unsigned)rows, cols > 8192 ? 512 : 256, sizeof(double) * (size_t)cols, st>>>(
      d_src, cols, k, ld, m.kpad, m.tile, bulk, d_map, m.d, m.expo, d_status, tc::staged_stall_cycles());
}

bool launch_split_MT(int nbf, int64_t n3, const double* d_F, int64_t ldF, const SplitMatrix& m, cudaStream_t st) {
  const size_t smem = sizeof(double) * 33 * (size_t)nbf;
  if (m.plain || nbf > 256 || m.kpad > 256) return false;
  shared_opt_in<&tc::k_split_MT>(sizeof(double) * 33 * 256);
  count_launch();
  tc::k_split_MT<<<dim3((unsigned)((n3 + 31) / 32), (unsigned)nbf), 256, smem, st>>>(
      nbf, n3, d_F, ldF, m.kpad, (m.steps() + 1) / 2 * 32, m.tile, m.d, m.expo);
  return true;
}

bool launch_split_orbitals(int nbf, int64_t n3, int nj, const double* d_Z, int64_t cols, const int* d_map,
                           uint32_t* d_max, const int* d_row_expo, const SplitMatrix& m, int* d_status, cudaStream_t st) {
  if (m.plain || n3 % 8 != 0 || cols % 2 != 0 || cols > tc::kSplitCols || (reinterpret_cast<uintptr_t>(d_Z) & 15)) return false;
  shared_opt_in<&tc::k_split_orbital_rows>(sizeof(double) * tc::kSplitCols);
  if (!d_row_expo) {
    cudaMemsetAsync(d_max, 0, sizeof(uint32_t) * (size_t)nbf, st);
    count_launch();
    tc::k_orbital_max<<<(unsigned)((int64_t)nj * nbf), 256, 0, st>>>(nbf, cols, cols, d_Z, d_max);
  }
  count_launch();
  tc::k_split_orbital_rows<<<(unsigned)((int64_t)nj * nbf), cols > 8192 ? 512 : 256, sizeof(double) * (size_t)cols, st>>>(
      nbf, n3, nj, cols, cols, d_Z, d_map, d_max, d_row_expo, m.k, m.kpad, m.tile, m.d, m.expo, d_status,
      tc::staged_stall_cycles());
  return true;
}

void launch_transpose(const double* in, int64_t rows, int64_t cols, int64_t ldi, double* out, int64_t ldo,
                      cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return;
  dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((rows + 31) / 32)), block(32, 8);
  count_launch();
  tc::k_transpose<<<grid, block, 0, st>>>(in, rows, cols, ldi, out, ldo);
}

void launch_reduce_splits(const double* part, int splits, int64_t stride, int64_t rows, int64_t cols, int64_t ld,
                          double* out, int64_t ldo, cudaStream_t st) {
  const int64_t total = rows * cols;
  if (total <= 0) return;
  int64_t b = (total + 255) / 256;
  if (b > 152 * 32) b = 152 * 32;
  count_launch();
  if (splits > 32 && total <= 152 * 256) {  // one output per thread would leave SMs without work
    tc::k_reduce_many<<<(unsigned)((total + 31) / 32), 256, 0, st>>>(part, splits, stride, rows, cols, ld, out, ldo);
    return;
  }
  tc::k_reduce_splits<<<(unsigned)b, 256, 0, st>>>(part, splits, stride, rows, cols, ld, out, ldo);
}

}  // namespace lrtei
