// tc_gemm.h -- the tensor-core GEMM kernel (tcgen05 + TMEM, sm_103a) shared by the split-precision products
// (k_tcgen05.cu) and the FP64 digit products (k_ozaki.cu).
//
// C = A B^T for two operands cut into planes of FP16 (or BF16) slices.  A scheme S says which slice
// products are formed, into which FP32 accumulators, how deep a chunk of K is accumulated before it is
// drained into registers, and what an output element is made of.
//
// Operand layout: tiles of 128 rows (or of the N of a skinny product) x 16 columns x S::PT planes are
// contiguous, K block after K block, each plane's 32-byte rows in the 32-byte swizzle of shared memory, so
// that the operands of one 16-deep MMA step are one contiguous copy each.  With 64-deep stages of
// row-major planes (two of 112 KB) every refill exposed its latency; nine 24 KB steps hide it, and the
// planes carry the powers of two of their weights, so that A and B need the same three (four for B before).
//
// Roles (18 warps, one persistent CTA per SM): warp 0 copies, the elected thread of warp 1 issues the MMAs,
// warps 2-17 drain and store.  Finished tiles are stored from registers while the next tile's MMAs run;
// staged through the ring they stalled it for ~15 us a tile.
// Every mbarrier wait is bounded: on expiry the CTA raises the device status word, stops issuing work,
// waits (bounded) for what it issued, frees TMEM and exits.
#pragma once
#include <stdlib.h>

#include <algorithm>
#include <type_traits>

#include "lrtei_internal.h"
#include "tc_common.h"

namespace lrtei {
namespace tcg {

using namespace tc;

constexpr int BM = 128;      // rows of A per tile (M of the MMA)
constexpr int KB = 16;       // K of one operand block
constexpr int EPI = 16;      // epilogue warps: four per TMEM lane quadrant
constexpr int THREADS = 64 + 32 * EPI;
constexpr int kGroupM = 16;  // M tiles walked together (operand slabs shared in L2)
constexpr int kGroupRows = 8;
// Flags of a step table's entries (K block numbers below 2^26): the entry opens a stage that ends its chunk; how many
// entries share a stage that it opens, less one.
constexpr int kLast = 1 << 30, kCountBit = 26, kBlock = (1 << kCountBit) - 1;
__host__ __device__ constexpr int stage_entries(int e) { return ((e >> kCountBit) & 7) + 1; }

// One block of the product: rows a_row0 + [0, M) of A, b_row0 + [0, N) of B, `units` split units of K from
// block a_blk and b_blk, written at C + c_off.  Rows below m_lo belong to the first tile only (a_row0 is a
// multiple of 128) and are not stored.
// tab: the step table (ParityClasses) of a scheme with LIST: the K blocks of the operand that holds them all;
// the other operand holds only the listed ones, one after the other.
constexpr int kMaxSeg = 36;  // the pairs of eight partitions (adaptive boxes)
struct Seg {
  int64_t a_row0, b_row0, M, N, c_off, item0;
  int a_blk, b_blk, units, tiles_m, tiles_n, m_lo;
  int steps;       // K blocks that hold columns (the rest of the last unit is zeros); without a table
  const int* tab;
};
struct Params {
  Seg seg[kMaxSeg];
  int nseg, splits, symmetric, transpose_out, accumulate, mirror, align;
  int list_is_a;    // step tables list blocks of A (B is the compact operand), else of B
  int64_t nitems;   // per split
  int64_t blk0, blk1, nb;  // symmetric: block rows [blk0, blk1) of the nb x nb triangle of 128 x 128 blocks
  const uint8_t* a;
  const uint8_t* b;
  int64_t a_steps, b_steps;  // K blocks of a row tile
  int b_tile;                // rows of B's tiles: BN, or 128 with BN a divisor
  const int* ea;
  const int* eb;
  double scale;
  double* C;
  int64_t ldc, split_stride;
  int* status;
  long long test_stall;  // > 0 (tests only): the MMA warp first waits that many cycles on a barrier that
                         // nothing completes, so that the bounded-wait failure path runs
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

// K-major operand block of 32-byte rows in the 32-byte swizzle: 8-row atoms of 256 bytes.
__device__ __forceinline__ uint64_t block_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (uint64_t)1 << 16 | (uint64_t)(256 >> 4) << 32 | (uint64_t)1 << 46 |
         (uint64_t)6 << 61;
}

// A work item: a tile (m0, n0: its first row and column inside the segment) and the K steps [t0, t1).
struct Work {
  int seg, m0, n0, split, t0, t1, nch;
  bool mirror;
};

// Items are split-major, so that the items running at once share operand slabs in L2.
template <class S>
__device__ __forceinline__ Work work_item(const Params& p, int64_t item) {
  Work w;
  w.split = (int)(item / p.nitems);
  int64_t t = item % p.nitems;
  w.seg = 0;
  while (w.seg + 1 < p.nseg && t >= p.seg[w.seg + 1].item0) ++w.seg;
  const Seg& s = p.seg[w.seg];
  t -= s.item0;
  w.mirror = false;
  if (p.symmetric) {  // upper triangle of 128 x 128 blocks in groups of block rows, column by column
    constexpr int SUB = BM / S::BN;
    const int sub = (int)(t % SUB);
    t /= SUB;
    int64_t r = 0, c = 0;
    for (int64_t R0 = p.blk0; R0 < p.blk1; R0 += kGroupRows) {
      const int64_t R1 = min(p.blk1, R0 + kGroupRows), g = R1 - R0;
      const int64_t tri = g * (g + 1) / 2, in_group = tri + (p.nb - R1) * g;
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
    w.n0 = (int)(c * BM + sub * S::BN);
    w.mirror = c != r;
  } else {
    const int64_t per_group = (int64_t)kGroupM * s.tiles_n;
    const int64_t first = (t / per_group) * kGroupM, in_g = t % per_group;
    const int64_t gsize = min((int64_t)kGroupM, s.tiles_m - first);
    w.m0 = (int)((first + in_g % gsize) * BM);
    w.n0 = (int)(in_g / gsize * S::BN);
  }
  const int per = (s.units + p.splits - 1) / p.splits;
  const int u0 = min(s.units, w.split * per), u1 = min(s.units, u0 + per);
  if constexpr (S::LIST) {  // [units + 1] first list entry of each unit, [units + 1] chunks with entries before it, the list
    w.t0 = s.tab[u0];
    w.t1 = s.tab[u1];
    w.nch = s.tab[s.units + 1 + u1] - s.tab[s.units + 1 + u0];
  } else {
    w.t1 = min((s.steps + S::KS - 1) / S::KS * S::KS, u1 * S::UNIT);  // whole stages (the padding is zeros)
    w.t0 = min(w.t1, u0 * S::UNIT);
    w.nch = (w.t1 - w.t0 + S::CHUNK - 1) / S::CHUNK;
  }
  return w;
}

template <class S>
struct Geo {
  static constexpr uint32_t A_BYTES = BM * KB * 2, B_BYTES = S::BN * KB * 2;  // one plane of a block
  static constexpr uint32_t STEP = S::NP * (A_BYTES + B_BYTES);
  static constexpr uint32_t STAGE = S::KS * STEP;
  static constexpr int STAGES = 220 * 1024 / STAGE < 16 ? 220 * 1024 / STAGE : 16;
  static constexpr size_t SMEM = STAGES * STAGE + 1024 + 512;
  static_assert(2 * S::NACC * S::BN <= 512, "two buffers of the accumulators must fit in TMEM");
};

template <class S>
__global__ void __launch_bounds__(THREADS, 1) k_tc_gemm(const __grid_constant__ Params p) {
  using G = Geo<S>;
  constexpr int NP = S::NP, STAGES = G::STAGES, BN = S::BN, QC = BN / (EPI / 4), KS = S::KS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * G::STAGE);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;  // [2] accumulator buffer ready
  uint64_t* acce = accf + 2;        // [2] accumulator buffer drained
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
    if (lane == 0) {  // producer
      uint32_t it = 0;
      bool stop = false;
      for (int64_t item = blockIdx.x; item < nitems && !stop; item += gridDim.x) {
        const Work w = work_item<S>(p, item);
        const Seg& sg = p.seg[w.seg];
        const int* list = S::LIST ? sg.tab + 2 * (sg.units + 1) : nullptr;
        const uint8_t* a = p.a + (((sg.a_row0 + w.m0) / BM) * p.a_steps + sg.a_blk) * (S::PT * G::A_BYTES);
        const int64_t br = sg.b_row0 + w.n0, b_blk = (int64_t)S::PT * p.b_tile * KB * 2;
        const uint8_t* b = p.b + ((br / p.b_tile) * p.b_steps + sg.b_blk) * b_blk + (br % p.b_tile) * (KB * 2);
        for (int t = w.t0; t < w.t1; ++it) {
          const int s = (int)(it % STAGES);
          const int e = S::LIST ? list[t] : 0;
          const int cnt = S::LIST ? stage_entries(e) : KS;  // steps of this stage
          if (!mbar_wait(&empty[s], ((it / STAGES) & 1u) ^ 1u, abort_flag, p.status, 32)) { stop = true; break; }
          mbar_arrive_expect_tx(&full[s], (uint32_t)cnt * G::STEP);
          uint8_t* st = smem + (size_t)s * G::STAGE;
#pragma unroll
          for (int q = 0; q < KS; ++q) {
            if (q >= cnt) break;
            const int pos = t + q, nat = S::LIST ? (q == 0 ? e : list[pos]) & kBlock : pos;
            const int ka = S::LIST && p.list_is_a ? nat : pos, kb = S::LIST && !p.list_is_a ? nat : pos;
            bulk_load(st + q * G::STEP, a + (int64_t)ka * (S::PT * G::A_BYTES), NP * G::A_BYTES, &full[s]);
            uint8_t* sb = st + q * G::STEP + NP * G::A_BYTES;
            const uint8_t* bs = b + kb * b_blk;
            if (p.b_tile == BN) {
              bulk_load(sb, bs, NP * G::B_BYTES, &full[s]);
            } else {
#pragma unroll
              for (int i = 0; i < NP; ++i)
                bulk_load(sb + i * G::B_BYTES, bs + (int64_t)i * p.b_tile * KB * 2, G::B_BYTES, &full[s]);
            }
          }
          t += cnt;
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
    // kind::f16, D FP32, both operands K-major; FP16 (format 0) or BF16 (format 1)
    constexpr uint32_t f = S::BF16 ? 1u : 0u;
    const uint32_t idesc = (1u << 4) | (f << 7) | (f << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
    if (elect_one()) {
      // One thread runs the whole loop.  The tensor pipe queues little beyond the MMA it runs, so what lies
      // between two stages is kept short: the next stage's barrier is tested and the next list entry loaded
      // before the MMAs issue, offsets run along.  (Behind `if (lane == 0)`, with the bounded-wait helper at
      // every stage, an MMA took up to 100 clocks to issue and a stage ~900 more.)
      const uint32_t full0 = smem_u32(full);
      const uint64_t a_desc = block_desc(smem_u32(smem)), b_desc = block_desc(smem_u32(smem) + NP * G::A_BYTES);
      uint32_t s = 0, ph = 0, cg = 0;
      bool ok = true, ready = false;
      if (p.test_stall > 0) ok = mbar_wait(never, 0u, abort_flag, p.status, 0, p.test_stall);
      for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
        const Work w = work_item<S>(p, item);
        const Seg& sg = p.seg[w.seg];
        const int* list = S::LIST ? sg.tab + 2 * (sg.units + 1) : nullptr;
        int in_chunk = 0;  // steps of the current chunk so far
        int next = S::LIST && w.t0 < w.t1 ? list[w.t0] : 0;
        for (int t = w.t0; t < w.t1;) {
          const int e = next, cnt = S::LIST ? stage_entries(e) : KS;
          t += cnt;
          // the chunk ends with a flagged stage, after CHUNK steps, or with the item
          const bool last = (S::LIST ? (e & kLast) != 0 : in_chunk + cnt >= S::CHUNK) || t >= w.t1;
          if (S::LIST) next = list[min(t, w.t1 - 1)];
          if (in_chunk == 0 && !mbar_wait(&acce[cg & 1u], ((cg >> 1) & 1u) ^ 1u, abort_flag, p.status)) { ok = false; break; }
          if (!ready && !mbar_wait(&full[s], ph, abort_flag, p.status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t cur = s;
          if (++s == STAGES) {
            s = 0;
            ph ^= 1u;
          }
          ready = mbar_test_wait_at(full0 + s * 8, ph);
          const uint32_t d0 = tmem_base + (cg & 1u) * (uint32_t)(S::NACC * BN);
          const uint64_t so = (uint64_t)(cur * (G::STAGE >> 4));
#pragma unroll
          for (int k = 0; k < KS; ++k)
            if (k < cnt)
              S::mma(d0, a_desc + so + (uint64_t)((k * G::STEP) >> 4), b_desc + so + (uint64_t)((k * G::STEP) >> 4), idesc,
                     (in_chunk == 0 && k == 0) ? 0u : 1u);
          mma_commit(&empty[cur]);
          if (last) mma_commit(&accf[cg & 1u]);
          in_chunk = last ? 0 : in_chunk + cnt;
          cg += last ? 1u : 0u;
        }
      }
      // retire every MMA issued before TMEM is released
      mma_commit(done);
      long long t0 = clock64();
      while (!mbar_try_wait(done, 0u) && clock64() - t0 < kWaitCycles) {
      }
    }
    __syncwarp();
  } else {
    const int ew = warp - 2, quad = warp & 3, col0 = (ew >> 2) * QC, row = quad * 32 + lane;
    uint32_t cg = 0;
    bool ok = true;
    for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const Work w = work_item<S>(p, item);
      const Seg& sg = p.seg[w.seg];
      typename S::template Sums<QC> T;
      T.clear();
      for (int c = 0; c < w.nch; ++c, ++cg) {
        const int buf = (int)(cg & 1u);
        ok = __all_sync(0xffffffffu, mbar_wait(&accf[buf], (cg >> 1) & 1u, abort_flag, p.status));
        if (!ok) break;
        tc_fence_after();
        T.drain(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * S::NACC * BN + col0));
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acce[buf]);
      }
      if (!ok || *abort_flag) break;
      const int m = w.m0 + row, n = w.n0 + col0, M = (int)sg.M, N = (int)sg.N;
      const bool mlive = m < M && m >= sg.m_lo;
      const int ea = mlive ? p.ea[sg.a_row0 + m] : 0;
      const int* eb = p.eb + sg.b_row0;
      double* C = p.C + sg.c_off + (int64_t)w.split * p.split_stride;
      const bool diag = p.symmetric && !w.mirror;  // the upper triangle only, mirrored below
      if (n >= N || !__any_sync(0xffffffffu, mlive)) continue;  // a warp without rows to store
#pragma unroll
      for (int j0 = 0; j0 < QC; j0 += 4) {
        T.template hold<4>(j0);  // one group of columns at a time (the sums fill the registers)
        const int live = mlive ? max(0, min(4, N - n - j0)) : 0;
        double v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = T.value(j0 + j, ea + (j < live ? __ldg(eb + n + j0 + j) : 0), p.scale);
        if (p.transpose_out) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < live) {
              double* c = C + (int64_t)(n + j0 + j) * p.ldc + m;
              if constexpr (S::ACCUM) *c = p.accumulate ? *c + v[j] : v[j];
              else *c = v[j];
            }
        } else {
          double* c = C + (int64_t)m * p.ldc + n + j0;
          if constexpr (S::ACCUM) {
            if (p.accumulate) {
              double old[4];
              load4(c, p.align, live, old);
#pragma unroll
              for (int j = 0; j < 4; ++j) v[j] += old[j];
            }
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

// ------------------------------------------------------------------ host side
template <class S>
lrtei_status launch(const Params& p, cudaStream_t st) {
  LRTEI_CUDA(shared_opt_in<&k_tc_gemm<S>>(Geo<S>::SMEM));
  int nsm = 0;  // persistent grid: one CTA per SM (shared memory and TMEM allow one)
  LRTEI_CUDA(sm_count(&nsm));
  const int64_t items = p.nitems * p.splits;
  if (items <= 0) return LRTEI_OK;
  count_launch();
  k_tc_gemm<S><<<(unsigned)std::min<int64_t>(items, nsm), THREADS, Geo<S>::SMEM, st>>>(p);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "tensor-core GEMM launch");
  return LRTEI_OK;
}

inline long long test_stall_cycles() {
  const char* v = getenv("LRTEI_TEST_STALL_CYCLES");
  return (v && *v) ? std::max(0LL, atoll(v)) : 0;
}
}  // namespace tcg
}  // namespace lrtei
