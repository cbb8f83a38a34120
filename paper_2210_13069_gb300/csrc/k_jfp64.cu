// k_jfp64.cu -- the FP64 CUDA-core J-build and node sum.
//   X = F_u^T u, Y = sum_p w_p (A_x^p (x) A_y^p (x) A_z^p) X (eq. ig1), J_u = F_u Y (eq. coulapprox)
// This device runs about two FP64 FMAs per clock and SM, so every kernel here is bound by its FMA
// count once the chip is full; below that, by launches.  Hence as few of them as there are products, whatever n and
// P (k_jx and k_jy once per eight densities, two kernels of the node sum per 128 MB of its intermediate, a reduction
// where X comes in more than eight parts: five for the molecule below), and the node sum skips the zeros of the Chebyshev coefficients: A^(p)(a, b) = 0 for odd
// a + b, because the kernel exp(-s^2 (x - y)^2) on two boxes about one centre is unchanged by
// (x, y) -> (-x, -y).
// One density of the 20-function molecule (n = 16, P = 20), a CUDA graph replay: 4 810 us with the
// 64 x 64-tile GEMM and 4 P mode-product launches before, 30 here.
#include <algorithm>

#include "lrtei_internal.h"

namespace lrtei {

// ---------------------------------------------------------------- node sum (eq. ig1)
// Z[q][p][m1][b2][b3] = w_p sum_{m2, m3} A_y(b2, m2) A_z(b3, m3) X[q][m1][m2][m3]: one CTA per
// (m1, row q) and group of nodes; the n x n slab, both matrices and the intermediate stay in shared
// memory (131 KB at n = 64).  X may come as `nsplit` partial sums.
__global__ void __launch_bounds__(256) k_node_modes(int n, int P, int pb, int par, const double* __restrict__ C,
                                                    const double* __restrict__ w, const double* __restrict__ X,
                                                    int nsplit, int64_t split_stride, double* __restrict__ Z) {
  extern __shared__ double sm[];
  const int nn = n * n, ld = n + 1;
  double* Xs = sm;            // [n][n]
  double* T = Xs + nn;        // [n][n]
  double* Ay = T + nn;        // [n][ld]
  double* Az = Ay + n * ld;   // [n][ld]
  const int m1 = blockIdx.x;
  const int64_t q = blockIdx.z, n3 = (int64_t)nn * n;
  const double* x = X + q * n3 + (int64_t)m1 * nn;
  for (int i = threadIdx.x; i < nn; i += blockDim.x) {
    double v = x[i];
    for (int s = 1; s < nsplit; ++s) v += x[s * split_stride + i];
    Xs[i] = v;
  }
  const int step = par ? 2 : 1;
  const int p1 = min(P, (int)(blockIdx.y + 1) * pb);
  for (int p = blockIdx.y * pb; p < p1; ++p) {
    const double* cy = C + ((size_t)P + p) * nn;
    const double* cz = C + ((size_t)2 * P + p) * nn;
    for (int i = threadIdx.x; i < nn; i += blockDim.x) {
      Ay[i / n * ld + i % n] = cy[i];
      Az[i / n * ld + i % n] = cz[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nn; i += blockDim.x) {
      const int m2 = i / n, b3 = i % n;
      double acc = 0.0;
#pragma unroll 4
      for (int m3 = par ? (b3 & 1) : 0; m3 < n; m3 += step) acc = fma(Az[b3 * ld + m3], Xs[m2 * n + m3], acc);
      T[i] = acc;
    }
    __syncthreads();
    double* z = Z + ((q * P + p) * n + m1) * nn;
    const double wp = w[p];
    for (int i = threadIdx.x; i < nn; i += blockDim.x) {
      const int b2 = i / n, b3 = i % n;
      double acc = 0.0;
#pragma unroll 4
      for (int m2 = par ? (b2 & 1) : 0; m2 < n; m2 += step) acc = fma(Ay[b2 * ld + m2], T[m2 * n + b3], acc);
      z[i] = wp * acc;
    }
    __syncthreads();  // T and the matrices are overwritten by the next node
  }
}

// Y[q][b1][c] = sum_p sum_{m1} A_x(b1, m1) Z[q][p][m1][c], c = (b2, b3): a thread owns a column c and
// NB1 values of b1 of one parity (Z read once for them); PG groups of threads share the nodes and
// meet in shared memory (few rows: the chain of P n / 2 FMAs would otherwise be the time).
template <int NB1, int PG>
__global__ void __launch_bounds__(256) k_node_sum(int n, int P, int par, const double* __restrict__ C,
                                                  const double* __restrict__ Z, double* __restrict__ Y) {
  constexpr int CX = 256 / PG;
  __shared__ double red[PG > 1 ? 256 * NB1 : 1];
  const int nn = n * n, g = threadIdx.x / CX, cx = threadIdx.x % CX;
  const int c = blockIdx.x * CX + cx;
  // b1 values of this block: with parity, first + 2 i (even ones, then odd ones), else first + i
  const int step = par ? 2 : 1;
  const int per_par = par ? ((n + 1) / 2 + NB1 - 1) / NB1 : (n + NB1 - 1) / NB1;
  const int odd = (int)blockIdx.y / per_par, b10 = (par ? odd : 0) + step * NB1 * ((int)blockIdx.y % per_par);
  const int64_t q = blockIdx.z;
  double acc[NB1];
#pragma unroll
  for (int i = 0; i < NB1; ++i) acc[i] = 0.0;
  if (c < nn)
    for (int p = g; p < P; p += PG) {
      const double* cp = C + (size_t)p * nn;
      const double* z = Z + (q * P + p) * (int64_t)nn * n + c;
#pragma unroll 4
      for (int m1 = par ? odd : 0; m1 < n; m1 += step) {
        const double v = z[(int64_t)m1 * nn];
#pragma unroll
        for (int i = 0; i < NB1; ++i) {
          const int b1 = min(b10 + step * i, n - 1);
          acc[i] = fma(cp[b1 * n + m1], v, acc[i]);
        }
      }
    }
  if constexpr (PG > 1) {
#pragma unroll
    for (int i = 0; i < NB1; ++i) red[i * 256 + threadIdx.x] = acc[i];
    __syncthreads();
    if (g != 0) return;
#pragma unroll
    for (int i = 0; i < NB1; ++i)
      for (int k = 1; k < PG; ++k) acc[i] += red[i * 256 + k * CX + cx];
  }
  if (c >= nn) return;
#pragma unroll
  for (int i = 0; i < NB1; ++i) {
    const int b1 = b10 + step * i;
    if (b1 < n) Y[(q * n + b1) * nn + c] = acc[i];
  }
}

// Rows of Z (P n^3 doubles each) are formed in chunks within 128 MB.  Few rows take one b1 per thread
// and four node groups; from 8 rows on the chip is full and four b1 per thread read Z a quarter as often.
cudaError_t launch_kron_apply(int n, int P, const double* d_C, const double* d_w, const double* d_X, int nsplit,
                              int64_t split_stride, double* d_Y, int64_t ncol, bool parity, cudaStream_t st) {
  if (ncol <= 0) return cudaSuccess;
  const int64_t n3 = (int64_t)n * n * n;
  const int64_t rows = std::min<int64_t>(
      {ncol, 65535, std::max<int64_t>(1, (int64_t)((128ULL << 20) / (sizeof(double) * (size_t)P * n3)))});
  double* Z = nullptr;
  cudaError_t e = scratch_alloc((void**)&Z, sizeof(double) * (size_t)rows * P * n3, st);
  if (e != cudaSuccess) return e;
  const size_t smem = sizeof(double) * 2 * ((size_t)n * n + (size_t)n * (n + 1));
  shared_opt_in<&k_node_modes>(sizeof(double) * 2 * (kMaxN * kMaxN + kMaxN * (kMaxN + 1)));  // a refusal shows below
  const int par = parity ? 1 : 0;
  for (int64_t r0 = 0; r0 < ncol; r0 += rows) {
    const int64_t nr = std::min(rows, ncol - r0);
    // nodes per CTA: enough CTAs for eight per SM, then as many nodes as possible on one loaded slab
    const int pb = (int)std::max<int64_t>(1, std::min<int64_t>(P, (int64_t)P * n * nr / (8 * 152)));
    count_launch();
    k_node_modes<<<dim3((unsigned)n, (unsigned)((P + pb - 1) / pb), (unsigned)nr), 256, smem, st>>>(
        n, P, pb, par, d_C, d_w, d_X + r0 * n3, nsplit, split_stride, Z);
    count_launch();
    if (nr < 8) {
      const unsigned gy = (unsigned)(par ? 2 * ((n + 1) / 2) : n);
      k_node_sum<1, 4><<<dim3((unsigned)((n * n + 63) / 64), gy, (unsigned)nr), 256, 0, st>>>(n, P, par, d_C, Z,
                                                                                            d_Y + r0 * n3);
    } else {
      const unsigned gy = (unsigned)(par ? 2 * (((n + 1) / 2 + 3) / 4) : (n + 3) / 4);
      k_node_sum<4, 1><<<dim3((unsigned)((n * n + 255) / 256), gy, (unsigned)nr), 256, 0, st>>>(n, P, par, d_C, Z,
                                                                                              d_Y + r0 * n3);
    }
  }
  e = cudaGetLastError();
  cudaFreeAsync(Z, st);
  return e;
}

// ---------------------------------------------------------------- the two F_u products
constexpr int kJRows = 128;  // pairs whose densities k_jx stages in shared memory at a time

// part[s][q][m] = sum over the pairs r of split s of u_q(r) F(r, m), u_q(r) = D_q(mu, nu) (2 - [mu == nu]):
// one thread per column m, F read once for Q densities.
template <int Q>
__global__ void __launch_bounds__(128) k_jx(int nbf, int64_t npair, int64_t n3, int R, int q0, int64_t per,
                                            const double* __restrict__ D, const int* __restrict__ pair_mu,
                                            const int* __restrict__ pair_nu, const double* __restrict__ F,
                                            double* __restrict__ part) {
  __shared__ double u[kJRows * Q];
  const int64_t rend = min(npair, (int64_t)(blockIdx.y + 1) * per);
  const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double acc[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) acc[i] = 0.0;
  for (int64_t r0 = (int64_t)blockIdx.y * per; r0 < rend; r0 += kJRows) {
    const int nr = (int)min((int64_t)kJRows, rend - r0);
    __syncthreads();  // the previous rows' densities have been read
    for (int i = threadIdx.x; i < nr * Q; i += blockDim.x) {
      const int64_t r = r0 + i / Q;
      const int q = q0 + i % Q, mu = pair_mu[r], nu = pair_nu[r];
      const double v = q < R ? D[(size_t)q * nbf * nbf + (size_t)mu * nbf + nu] : 0.0;
      u[i] = mu == nu ? v : 2.0 * v;
    }
    __syncthreads();
    if (m >= n3) continue;
    const double* f = F + r0 * n3 + m;
#pragma unroll 8
    for (int j = 0; j < nr; ++j) {
      const double v = f[(int64_t)j * n3];
#pragma unroll
      for (int i = 0; i < Q; ++i) acc[i] = fma(u[j * Q + i], v, acc[i]);
    }
  }
  if (m >= n3) return;
#pragma unroll
  for (int i = 0; i < Q; ++i)
    if (q0 + i < R) part[((int64_t)blockIdx.y * R + q0 + i) * n3 + m] = acc[i];
}

// J_q(mu, nu) = J_q(nu, mu) = scale sum_m F(r, m) Y_q(m): one CTA per unique pair r.
template <int Q>
__global__ void __launch_bounds__(256) k_jy(int nbf, int64_t n3, int R, int q0, const int* __restrict__ pair_mu,
                                            const int* __restrict__ pair_nu, const double* __restrict__ F,
                                            const double* __restrict__ Y, double scale, double* __restrict__ J,
                                            int* status) {
  __shared__ double red[8 * Q];
  const int64_t r = blockIdx.x;
  const double* f = F + r * n3;
  const double* y[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) y[i] = Y + (int64_t)min(q0 + i, R - 1) * n3;
  double acc[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) acc[i] = 0.0;
#pragma unroll 4
  for (int64_t m = threadIdx.x; m < n3; m += 256) {
    const double v = f[m];
#pragma unroll
    for (int i = 0; i < Q; ++i) acc[i] = fma(v, y[i][m], acc[i]);
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
    if ((threadIdx.x & 31) == 0) red[(threadIdx.x >> 5) * Q + i] = acc[i];
  }
  __syncthreads();
  if (threadIdx.x >= Q || q0 + (int)threadIdx.x >= R) return;
  double s = 0.0;
  for (int k = 0; k < 8; ++k) s += red[k * Q + threadIdx.x];
  s *= scale;
  if (!isfinite(s)) latch_status(status, (int)kDevNonFinite);
  const int mu = pair_mu[r], nu = pair_nu[r];
  double* j = J + (size_t)(q0 + threadIdx.x) * nbf * nbf;
  j[(size_t)mu * nbf + nu] = s;
  j[(size_t)nu * nbf + mu] = s;
}

// Splits of the pairs: about eight CTAs per SM, at least 16 pairs each (below that the partial sums
// cost more than they hide).
int jx_splits(int64_t npair, int64_t n3) {
  const int64_t blocks = (n3 + 127) / 128;
  return (int)std::max<int64_t>(1, std::min<int64_t>(npair / 16, 8 * 152 / blocks));
}

template <int Q>
static void jx_q(const PairTable& t, int nbf, int64_t n3, int R, int q0, int nsplit, const double* D, const double* F,
                 double* part, cudaStream_t st) {
  const int64_t per = (t.npair + nsplit - 1) / nsplit;
  const unsigned gy = (unsigned)((t.npair + per - 1) / per);
  count_launch();
  k_jx<Q><<<dim3((unsigned)((n3 + 127) / 128), gy), 128, 0, st>>>(nbf, t.npair, n3, R, q0, per, D, t.pair_mu, t.pair_nu,
                                                                F, part);
}

int launch_jx(const PairTable& t, int nbf, int64_t n3, int R, int nsplit, const double* d_D, const double* d_F,
              double* d_part, cudaStream_t st) {
  for (int q = 0; q < R;) {
    const int left = R - q;
    if (left >= 5) { jx_q<8>(t, nbf, n3, R, q, nsplit, d_D, d_F, d_part, st); q += 8; }
    else if (left >= 3) { jx_q<4>(t, nbf, n3, R, q, nsplit, d_D, d_F, d_part, st); q += 4; }
    else if (left == 2) { jx_q<2>(t, nbf, n3, R, q, nsplit, d_D, d_F, d_part, st); q += 2; }
    else { jx_q<1>(t, nbf, n3, R, q, nsplit, d_D, d_F, d_part, st); q += 1; }
  }
  const int64_t per = (t.npair + nsplit - 1) / nsplit;
  return (int)((t.npair + per - 1) / per);
}

void launch_jy(const PairTable& t, int nbf, int64_t n3, int R, const double* d_F, const double* d_Y, double scale,
               double* d_J, int* d_status, cudaStream_t st) {
  const unsigned g = (unsigned)t.npair;
  for (int q = 0; q < R;) {
    const int left = R - q;
    count_launch();
    if (left >= 5) { k_jy<8><<<g, 256, 0, st>>>(nbf, n3, R, q, t.pair_mu, t.pair_nu, d_F, d_Y, scale, d_J, d_status); q += 8; }
    else if (left >= 3) { k_jy<4><<<g, 256, 0, st>>>(nbf, n3, R, q, t.pair_mu, t.pair_nu, d_F, d_Y, scale, d_J, d_status); q += 4; }
    else if (left == 2) { k_jy<2><<<g, 256, 0, st>>>(nbf, n3, R, q, t.pair_mu, t.pair_nu, d_F, d_Y, scale, d_J, d_status); q += 2; }
    else { k_jy<1><<<g, 256, 0, st>>>(nbf, n3, R, q, t.pair_mu, t.pair_nu, d_F, d_Y, scale, d_J, d_status); q += 1; }
  }
}

}  // namespace lrtei
