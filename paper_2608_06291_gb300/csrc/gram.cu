// bakron_gram: G <- beta G + alpha X^T diag(w) X on the tensor cores (Sec. 4,
// "Choosing the Factorization"), and the sample norms of one-step Shampoo.
//
// One persistent kernel, k_gram, walks work items (a block of G's lower
// triangle times a range of the samples).  Block and operand kinds:
//   OP_BF16_MN  bf16 samples without weights, read straight from X: features
//               are contiguous, so a slot (64 samples) holds MN-major operands,
//               64-feature boxes of 64 rows; kind::f16, products exact in fp32.
//               128 x 256 blocks.
//   OP_BF16_K   the same from a transposed, padded copy (K-major boxes), for an
//               X that TMA cannot read as it is (d not a multiple of 64, rows
//               or base not 16-byte aligned).
//   OP_TF32     fp32 or weighted samples: K-major tf32 hi/lo planes (k_gram_split)
//               and 3xTF32 products, 32 samples per slot, 128 x 128 blocks.
// A block's sum over at most 256 samples (bf16) or 32 (tf32) accumulates in
// place in TMEM, which does not round to nearest; those partial sums are added
// in fp32 registers by the epilogue warps.
//
// What bounds it: with 128 x 128 bf16 blocks an SM's shared memory takes 128 B
// per cycle from TMA and gives 128 B per cycle to the MMAs, twice its bandwidth;
// 128 x 256 blocks need 96 + 96.  The finished block leaves through shared
// memory, 64 columns at a time, so that both its rows and (mirrored) its
// columns are written 128 bytes per warp; written one row per lane it took as
// long as 10 000 samples' products.  The ring is not used for that, so the next
// block's loads and MMAs run meanwhile; old values (beta) are prefetched to L2 at
// the block's start.  On GB300: 2048 bf16 samples of 11008 features added to a
// running sum 1.61 -> 0.49 ms (reading and writing G alone takes 0.14), 16384
// samples of 4096 features 0.54 -> 0.24 ms (1.13 PFLOP/s), of which 0.07 was the
// transposed copy that MN-major operands need no more.  Blocks too few for the SMs
// are split along the samples (gram_splits), the parts summed in order by
// k_gram_reduce (5000 weighted fp32 samples of 1531 features: 120 -> 75 us).  The bf16
// forms' epilogue threads hold 128 sums each and spill 58 bytes.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>

#include <algorithm>

#include "common.cuh"
#include "tc_gemm.cuh"
#include "tcgen05.cuh"

namespace bakron {

namespace {

enum OpKind { OP_BF16_MN = 0, OP_BF16_K = 1, OP_TF32 = 2 };

constexpr int GR_M = 128;                      // rows of a block
constexpr int GR_EPI_WARPS = 8;                // two per TMEM lane quarter
constexpr int GR_THREADS = 32 * (2 + GR_EPI_WARPS);
constexpr int GR_STAGE_COLS = 64;              // columns staged at a time
constexpr int GR_STAGE_LD = GR_STAGE_COLS + 1; // odd: rows and columns both conflict-free
constexpr uint32_t PLANE = 16384;              // 128 rows (or 64 rows x 2 boxes) of 128 bytes

template <int OP>
struct GramShape {
  static constexpr bool tf32 = OP == OP_TF32;
  static constexpr int BN = tf32 ? 128 : 256;            // columns of a block
  static constexpr int KS = tf32 ? 32 : 64;              // samples of a slot
  static constexpr int group = tf32 ? 1 : 4;             // slots summed in place in TMEM
  static constexpr uint32_t a_bytes = tf32 ? 2 * PLANE : PLANE;
  static constexpr uint32_t b_bytes = 2 * PLANE;         // tf32: hi, lo; bf16: 256 features
  static constexpr uint32_t slot = a_bytes + b_bytes;
  static constexpr int slots = tf32 ? 3 : 4;
  static constexpr int nacc = 512 / BN;                  // TMEM accumulators
  static constexpr int cols = BN / 2;                    // columns an epilogue warp sums
  static constexpr uint32_t smem =
      slots * slot + GR_M * GR_STAGE_LD * 4 + 1024 /*align*/ + 256 /*barriers*/;
};
static_assert(GramShape<OP_TF32>::smem <= 232448 && GramShape<OP_BF16_K>::smem <= 232448, "smem");

struct GramParams {
  int tiles;             // blocks of the lower triangle
  int splits;            // ranges of the samples per block
  int nslots;            // slots of all samples
  int per_split;         // slots of one range (the last may be shorter)
  int d;
  float alpha, beta;
  float* G;
  int64_t ldg;
  float* part;           // splits > 1: [split][tile][128][BN]
  int a_exact, b_exact;  // tf32: that operand's lo plane is zero
  int* status;
  long long spin_cycles;
};

// Block t of the lower triangle, row by row: row block rb (128 rows) has the
// column blocks (BN wide) that reach the diagonal.
template <int BN>
__host__ __device__ inline void gram_block(int t, int& rb, int& cb) {
  constexpr int R = BN / 128;   // row blocks per column block: 1 or 2
  // row blocks R i .. R i + R - 1 have i + 1 blocks each; R i (i + 1) / 2 precede R i
  int i = (int)((sqrtf(8.f * (float)t / R + 1.f) - 1.f) * 0.5f);
  while (R * (i + 1) * (i + 2) / 2 <= t) ++i;
  while (R * i * (i + 1) / 2 > t) --i;
  const int in = t - R * i * (i + 1) / 2;
  rb = R * i + in / (i + 1);
  cb = in % (i + 1);
}

// mbar_wait that also gives up once another role has.
__device__ __forceinline__ bool gr_wait(uint64_t* bar, uint32_t parity, long long limit,
                                        volatile int* abort_flag) {
  if (mbar_test(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_test(bar, parity)) return true;
    if (*abort_flag || clock64() - t0 > limit) return false;
  }
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// Descriptor of an MN-major operand: 64-element (128-byte, swizzled) rows of
// one sample each, 8-sample groups 1024 bytes apart (stride offset), the next
// 64 features 8 KiB on (leading offset).
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)(8192 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

template <int OP>
__global__ void __launch_bounds__(GR_THREADS, 1)
    k_gram(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
           const GramParams P) {
  using S = GramShape<OP>;
  constexpr int NST = S::slots, NACC = S::nacc, BN = S::BN;
  extern __shared__ __align__(1024) unsigned char gr_smem[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)gr_smem + 1023) & ~(uintptr_t)1023);
  float* stage = (float*)(smem + NST * S::slot);            // [128][GR_STAGE_LD]
  uint64_t* bars = (uint64_t*)(smem + NST * S::slot + GR_M * GR_STAGE_LD * 4);
  uint64_t* full = bars;               // [NST] slot loaded
  uint64_t* empty = bars + NST;        // [NST] slot read by its MMAs
  uint64_t* accF = bars + 2 * NST;     // [NACC] accumulator holds a finished group
  uint64_t* accE = accF + NACC;        // [NACC] accumulator read out
  uint64_t* done = accE + NACC;        // every MMA complete
  uint32_t* tmem_slot = (uint32_t*)(done + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < NACC; ++a) {
      mbar_init(&accF[a], 1);
      mbar_init(&accE[a], GR_EPI_WARPS);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  const int items = P.tiles * P.splits;
  const long long drain = 4000000000LL;   // ~2 s: wind-down bound
  auto range = [&](int item, int& s0, int& n) {
    s0 = (item / P.tiles) * P.per_split;
    n = min(P.per_split, P.nslots - s0);
  };
  auto timed_out = [&]() {
    raise_status(P.status, BAKRON_ERR_TIMEOUT);
    *abort_flag = 1;
  };

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      const uint32_t bytes = (S::tf32 && P.a_exact ? PLANE : S::a_bytes) +
                             (S::tf32 && P.b_exact ? PLANE : S::b_bytes);
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        int rb, cb, s0, n;
        gram_block<BN>(item % P.tiles, rb, cb);
        range(item, s0, n);
        for (int i = 0; i < n; ++i, ++it) {
          const int s = it % NST;
          if (it >= NST &&
              !gr_wait(&empty[s], (uint32_t)(it / NST - 1) & 1u, P.spin_cycles, abort_flag)) {
            if (!*abort_flag) timed_out();
            ok = false;
            break;
          }
          unsigned char* a = smem + s * S::slot;
          unsigned char* b = a + S::a_bytes;
          const int k = (s0 + i) * S::KS;
          mbar_expect_tx(&full[s], bytes);
          if constexpr (OP == OP_BF16_MN) {
            tma_load_3d(a, &mapA, &full[s], 0, k, 2 * rb);
            tma_load_3d(b, &mapB, &full[s], 0, k, 4 * cb);
          } else if constexpr (OP == OP_BF16_K) {
            tma_load_2d(a, &mapA, &full[s], k, rb * GR_M);
            tma_load_2d(b, &mapB, &full[s], k, cb * BN);
          } else {
            tma_load_3d(a, &mapA, &full[s], k, rb * GR_M, 0);
            tma_load_3d(b, &mapB, &full[s], k, cb * BN, 0);
          }
        }
      }
      // every copy issued has landed before the CTA (and its shared memory) goes
      for (int j = it > NST ? it - NST : 0; j < it; ++j)
        if (!mbar_wait(&full[j % NST], (uint32_t)(j / NST) & 1u, drain)) timed_out();
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int it = 0, g = 0;
      bool ok = true;
      const uint32_t idesc =
          S::tf32 ? idesc_tf32(GR_M, BN)
                  : (idesc_bf16(GR_M, BN) | (OP == OP_BF16_MN ? (1u << 15) | (1u << 16) : 0u));
      const uint64_t desc0 =
          OP == OP_BF16_MN ? smem_desc_mn(smem_u32(smem)) : smem_desc(smem_u32(smem));
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        int s0, n;
        range(item, s0, n);
        for (int i = 0; i < n; ++i, ++it) {
          const int s = it % NST, a = g % NACC, in = i % S::group;
          if (!gr_wait(&full[s], (uint32_t)(it / NST) & 1u, P.spin_cycles, abort_flag) ||
              (in == 0 && g >= NACC &&
               !gr_wait(&accE[a], (uint32_t)(g / NACC - 1) & 1u, P.spin_cycles, abort_flag))) {
            if (!*abort_flag) timed_out();
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = desc0 + (uint64_t)((s * S::slot) >> 4);
          const uint64_t db = da + (S::a_bytes >> 4);
          const uint32_t d = tmem + (uint32_t)(a * BN);
          if constexpr (S::tf32) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              const uint64_t o = (uint64_t)(2 * kk);
              mma_tf32(d, da + o, db + o, idesc, (kk > 0 || in > 0) ? 1u : 0u);
              if (!P.b_exact) mma_tf32(d, da + o, db + (PLANE >> 4) + o, idesc, 1u);
              if (!P.a_exact) mma_tf32(d, da + (PLANE >> 4) + o, db + o, idesc, 1u);
            }
          } else {
            // 16 samples per MMA: 32 bytes along a K-major row, or two 8-sample groups
            constexpr uint64_t step = OP == OP_BF16_MN ? (2048 >> 4) : 2;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              mma_bf16(d, da + kk * step, db + kk * step, idesc, (kk > 0 || in > 0) ? 1u : 0u);
          }
          mma_commit(&empty[s]);
          if (in == S::group - 1 || i == n - 1) {
            mma_commit(&accF[a]);
            ++g;
          }
        }
      }
      mma_commit(done);
      if (!mbar_wait(done, 0, drain)) timed_out();   // before anyone frees TMEM
    }
    __syncwarp();
  } else {
    const int q = warp & 3;                          // TMEM lane quarter
    const int half = (warp - 2) >> 2;                // half of the columns
    const int ew = warp - 2;
    const int row = q * 32 + lane;
    int g = 0;
    bool dead = false;
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
      int rb, cb, s0, n;
      gram_block<BN>(item % P.tiles, rb, cb);
      range(item, s0, n);
      if (P.beta != 0.f && P.splits == 1) {
        // the old values of the block and of its mirror on their way to L2
        // while the samples are multiplied
        const int64_t gi0 = (int64_t)rb * GR_M, gj0 = (int64_t)cb * BN;
        for (int e = threadIdx.x - 64; e < GR_M * (BN / 32); e += 32 * GR_EPI_WARPS) {
          const int64_t gi = gi0 + e / (BN / 32), gj = gj0 + 32 * (e % (BN / 32));
          if (gi < P.d && gj <= gi)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(P.G + gi * P.ldg + gj));
          const int64_t mj = gj0 + e / (GR_M / 32), mi = gi0 + 32 * (e % (GR_M / 32));
          if (mi < P.d && mj < mi + 31 && mj < P.d)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(P.G + mj * P.ldg + mi));
        }
      }
      const int ng = (n + S::group - 1) / S::group;
      float acc[S::cols];
#pragma unroll
      for (int u = 0; u < S::cols; ++u) acc[u] = 0.f;
      for (int i = 0; i < ng && !dead; ++i, ++g) {
        const int a = g % NACC;
        int ok = 1;
        if (lane == 0) {   // one lane waits; tcgen05.ld is warp-collective
          ok = gr_wait(&accF[a], (uint32_t)(g / NACC) & 1u, P.spin_cycles, abort_flag) ? 1 : 0;
          if (!ok && !*abort_flag) timed_out();
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) {
          dead = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * BN + half * S::cols);
#pragma unroll
        for (int c = 0; c < S::cols / 32; ++c) {
          uint32_t r[32];
          tmem_ld32(ta + 32 * c, r);
          tmem_wait_ld();
#pragma unroll
          for (int u = 0; u < 32; ++u) acc[32 * c + u] += __uint_as_float(r[u]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&accE[a]);
      }
      // out, 64 columns at a time; every epilogue warp passes every barrier,
      // also after a time-out (then nothing is written)
#pragma unroll
      for (int p = 0; p < BN / GR_STAGE_COLS; ++p) {
        constexpr int PH = S::cols / GR_STAGE_COLS;    // passes per column half
        if (p / PH == half) {
#pragma unroll
          for (int u = 0; u < GR_STAGE_COLS; ++u)
            stage[row * GR_STAGE_LD + u] = acc[(p % PH) * GR_STAGE_COLS + u];
        }
        asm volatile("bar.sync 2, %0;" ::"n"(GR_EPI_WARPS * 32) : "memory");
        if (!*abort_flag) {
          const int64_t gi0 = (int64_t)rb * GR_M, gj0 = (int64_t)cb * BN + p * GR_STAGE_COLS;
          if (P.splits > 1) {
            float* o = P.part + (int64_t)item * GR_M * BN + p * GR_STAGE_COLS;
#pragma unroll 4
            for (int r = ew; r < GR_M; r += GR_EPI_WARPS) {
              o[(int64_t)r * BN + lane] = stage[r * GR_STAGE_LD + lane];
              o[(int64_t)r * BN + 32 + lane] = stage[r * GR_STAGE_LD + 32 + lane];
            }
          } else {
            // entries (gi, gj <= gi) along rows, then their mirrors along
            // columns, 16 loads of a lane in flight
            auto put = [&](int64_t gi, int64_t gj, bool in, float v, float old) {
              if (in) P.G[gi * P.ldg + gj] = P.beta == 0.f ? v : fmaf(P.beta, old, v);
            };
#pragma unroll 1
            for (int r0 = 0; r0 < GR_M; r0 += 8 * GR_EPI_WARPS) {
              float old[8][2];
#pragma unroll
              for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  const int64_t gi = gi0 + r0 + GR_EPI_WARPS * j + ew, gj = gj0 + 32 * h + lane;
                  old[j][h] = (P.beta != 0.f && gi < P.d && gj <= gi) ? P.G[gi * P.ldg + gj] : 0.f;
                }
#pragma unroll
              for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  const int r = r0 + GR_EPI_WARPS * j + ew, c = 32 * h + lane;
                  put(gi0 + r, gj0 + c, gi0 + r < P.d && gj0 + c <= gi0 + r,
                      P.alpha * stage[r * GR_STAGE_LD + c], old[j][h]);
                }
            }
#pragma unroll 1
            for (int c0 = 0; c0 < GR_STAGE_COLS; c0 += 4 * GR_EPI_WARPS) {
              float old[4][4];
#pragma unroll
              for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                  const int64_t gj = gj0 + c0 + GR_EPI_WARPS * j + ew, gi = gi0 + 32 * h + lane;
                  old[j][h] = (P.beta != 0.f && gi < P.d && gj < gi) ? P.G[gj * P.ldg + gi] : 0.f;
                }
#pragma unroll
              for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                  const int c = c0 + GR_EPI_WARPS * j + ew, r = 32 * h + lane;
                  put(gj0 + c, gi0 + r, gi0 + r < P.d && gj0 + c < gi0 + r,
                      P.alpha * stage[r * GR_STAGE_LD + c], old[j][h]);
                }
            }
          }
        }
        asm volatile("bar.sync 2, %0;" ::"n"(GR_EPI_WARPS * 32) : "memory");
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
}

// G's lower triangle and its mirror from the parts of k_gram (splits > 1),
// added in the order of the splits: 32 x 32 entries per block.  After a time-out
// parts are missing, and G is left as it is.
template <int BN>
__global__ void __launch_bounds__(256) k_gram_reduce(const GramParams P) {
  __shared__ float t[32][33];
  if (*P.status != BAKRON_OK) return;         // uniform: k_gram is done
  int rb, cb;
  gram_block<BN>(blockIdx.x, rb, cb);
  const int r0 = 32 * (blockIdx.y / (BN / 32)), c0 = 32 * (blockIdx.y % (BN / 32));
  const int64_t gi0 = (int64_t)rb * GR_M + r0, gj0 = (int64_t)cb * BN + c0;
  if (gi0 >= P.d || gj0 > gi0 + 31) return;   // uniform over the block
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = y + 8 * j;
    const float* p = P.part + ((int64_t)blockIdx.x * GR_M + r0 + r) * BN + c0 + x;
    float v = 0.f;
    for (int s = 0; s < P.splits; ++s) v += p[(int64_t)s * P.tiles * GR_M * BN];
    v *= P.alpha;
    t[r][x] = v;
    const int64_t gi = gi0 + r, gj = gj0 + x;
    if (gi < P.d && gj <= gi) {
      float* o = P.G + gi * P.ldg + gj;
      *o = P.beta == 0.f ? v : fmaf(P.beta, *o, v);
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = y + 8 * j;
    const int64_t gj = gj0 + c, gi = gi0 + x;
    if (gi < P.d && gj < gi) {
      float* o = P.G + gj * P.ldg + gi;
      const float v = t[x][c];
      *o = P.beta == 0.f ? v : fmaf(P.beta, *o, v);
    }
  }
}

// Gram operands: samples t0 .. t0 + kc of X (k x d, row stride ldx, fp32 or
// bf16) transposed into the K-major planes T = X^T (dp x kc, zeros past k and
// d), split as hi + lo; with weights, also WT = (diag(w) X)^T, the product
// w_t x_ti rounded once to fp32 before the split.  32 x 32 tiles through
// shared memory: coalesced reads along features, writes along samples.
__global__ void k_gram_split(const void* X, int xdt, int k, int d, int64_t ldx, int t0, int kc,
                             const float* w, float* Th, float* Tl, float* Wh, float* Wl) {
  __shared__ float tile[32][33];
  __shared__ float wt[32];
  const int tx = threadIdx.x, ty = threadIdx.y;     // 32 x 8
  const int tb = blockIdx.x * 32, ib = blockIdx.y * 32;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int t = t0 + tb + ty + 8 * r, i = ib + tx;
    float v = 0.f;
    if (t < k && i < d) {
      const int64_t o = (int64_t)t * ldx + i;
      v = xdt == BAKRON_BF16 ? __bfloat162float(((const __nv_bfloat16*)X)[o])
                             : ((const float*)X)[o];
    }
    tile[ty + 8 * r][tx] = v;
  }
  if (w && ty == 0) wt[tx] = (t0 + tb + tx < k) ? w[t0 + tb + tx] : 0.f;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = ib + ty + 8 * r, tc = tb + tx;
    const int64_t o = (int64_t)i * kc + tc;
    const float v = tile[tx][ty + 8 * r], h = tf32_hi(v);
    Th[o] = h;
    Tl[o] = v - h;
    if (w) {
      const float u = wt[tx] * v, uh = tf32_hi(u);
      Wh[o] = uh;
      Wl[o] = u - uh;
    }
  }
}

// bf16 samples t0 .. t0 + kc of X (k x d, row stride ldx) transposed into
// the K-major bf16 plane T = X^T (dp x kc, zeros past k and d): the operand of
// the kind::f16 Gram, exact (no split).  64 x 64 tiles through shared memory,
// 16-byte vectors both ways: a load is 8 features of one sample (when X and
// ldx allow 16-byte alignment and the 8 lie inside d; else element by
// element), a store 8 samples of one feature (always whole: dp and kc are
// multiples of 64).  A warp reads 4 rows of 128 bytes and stores 32 rows'
// 16-byte pieces; its shared-memory gathers read one 64-byte row segment.
constexpr int TR_TILE = 64, TR_LD = 72;   // row stride 144 B: 16-byte aligned rows

__global__ void __launch_bounds__(256)
    k_gram_transpose_bf16(const __nv_bfloat16* X, int k, int d, int64_t ldx, int t0, int kc,
                          int vec_ok, __nv_bfloat16* T) {
  __shared__ __align__(16) __nv_bfloat16 tile[TR_TILE][TR_LD];
  const int tb = blockIdx.x * TR_TILE, ib = blockIdx.y * TR_TILE;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int c = threadIdx.x + 256 * r;          // 512 chunks of 8 features
    const int tr = c >> 3, i0 = ib + 8 * (c & 7);
    const int t = t0 + tb + tr;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (t < k) {
      const __nv_bfloat16* src = X + (int64_t)t * ldx + i0;
      if (vec_ok && i0 + 8 <= d) {
        v = *reinterpret_cast<const uint4*>(src);
      } else {
        __align__(16) __nv_bfloat16 e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = (i0 + j < d) ? src[j] : __float2bfloat16(0.f);
        v = *reinterpret_cast<const uint4*>(e);
      }
    }
    *reinterpret_cast<uint4*>(&tile[tr][8 * (c & 7)]) = v;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int c = threadIdx.x + 256 * r;          // 512 chunks of 8 samples
    const int ir = c & 63, tc = c >> 6;
    __align__(16) __nv_bfloat16 e[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) e[j] = tile[8 * tc + j][ir];
    *reinterpret_cast<uint4*>(T + (int64_t)(ib + ir) * kc + tb + 8 * tc) =
        *reinterpret_cast<const uint4*>(e);
  }
}

// |y_t|^2 per row (warp per row, fp32, lane-strided partial sums then a
// butterfly): the one-step Shampoo weight tr(b_t^T b_t) of a vector sample.
__global__ void k_sqnorms(const void* Y, int ydt, int k, int d, int64_t ldy, float* out) {
  const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= k) return;
  float acc = 0.f;
  for (int j = lane; j < d; j += 32) {
    const int64_t o = row * ldy + j;
    const float v = ydt == BAKRON_BF16 ? __bfloat162float(((const __nv_bfloat16*)Y)[o])
                                       : ((const float*)Y)[o];
    acc = fmaf(v, v, acc);
  }
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) out[row] = acc;
}

}  // namespace
}  // namespace bakron

using namespace bakron;

// ------------------------------------------------------------------ host
namespace {
constexpr int GRAM_MAX_D = 1 << 16;
constexpr int SM_COUNT = 152;

cudaError_t gram_attrs() {
  static OncePerDevice once;
  return once([] {
    cudaError_t e =
        cudaFuncSetAttribute(k_gram<OP_BF16_MN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             GramShape<OP_BF16_MN>::smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_gram<OP_BF16_K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               GramShape<OP_BF16_K>::smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_gram<OP_TF32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               GramShape<OP_TF32>::smem);
    return e;
  });
}

// A tiled tensor map with the 128-byte swizzle and boxes inside 128-byte rows.
bool gram_map(CUtensorMap* map, CUtensorMapDataType type, int rank, const void* base,
              const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box) {
  if (!get_encode()) return false;
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return g_encode(map, type, rank, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// X as 64-feature boxes of 64 samples, `boxes` side by side: (feature in box,
// sample, box).  d is a multiple of 64: every box lies inside the rows.
bool map_bf16_mn(CUtensorMap* map, const void* X, int64_t k, int64_t d, int64_t ldx, int boxes) {
  const cuuint64_t dims[3] = {64u, (cuuint64_t)k, (cuuint64_t)(d / 64)};
  const cuuint64_t strides[2] = {(cuuint64_t)(ldx * 2), 128u};
  const cuuint32_t box[3] = {64u, 64u, (cuuint32_t)boxes};
  return gram_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, X, dims, strides, box);
}

// The transposed bf16 plane (rows x cols, row stride ld), boxes of 64 samples.
bool map_bf16_k(CUtensorMap* map, const void* T, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  return gram_map(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, T, dims, strides, box);
}

// A tf32 plane pair (lo `plane` bytes after hi), boxes of 32 samples x 128 rows;
// an exact operand's lo plane is left out of its boxes.
bool map_tf32(CUtensorMap* map, const float* hi, int64_t rows, int64_t cols, int64_t ld,
              int64_t plane, bool is_exact) {
  const cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, 2u};
  const cuuint64_t strides[2] = {(cuuint64_t)(ld * 4), (cuuint64_t)plane};
  const cuuint32_t box[3] = {32u, 128u, is_exact ? 1u : 2u};
  return gram_map(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, hi, dims, strides, box);
}

// Ranges of the samples per block, for `tiles` blocks over nslots slots: the
// count with the shortest schedule, in slots, of `tiles * S` items over the SMs.
// An item costs its slots and about 8 more (ring start, the way out); split
// blocks cost the reduction, one launch and S reads of a block's parts.
int gram_splits(int tiles, int nslots) {
  int best = 1;
  double cost = 0;
  for (int S = 1; S <= 32 && (S == 1 || nslots / S >= 8); ++S) {
    const int rounds = ceil_div(tiles * S, SM_COUNT);
    const double c = rounds * (ceil_div(nslots, S) + 8.0) +
                     (S > 1 ? 16.0 + 4.0 * S * tiles / SM_COUNT : 0.0);
    if (S == 1 || c < 0.95 * cost) {
      best = S;
      cost = c;
    }
  }
  return best;
}

template <int OP>
int launch_gram(const CUtensorMap& mA, const CUtensorMap& mB, GramParams& P, cudaStream_t s) {
  const int items = P.tiles * P.splits;
  k_gram<OP><<<std::min(items, SM_COUNT), GR_THREADS, GramShape<OP>::smem, s>>>(mA, mB, P);
  BK_CUDA_OK(cudaGetLastError());
  if (P.splits > 1) {
    constexpr int BN = GramShape<OP>::BN;
    k_gram_reduce<BN><<<dim3(P.tiles, 4 * (BN / 32)), 256, 0, s>>>(P);
    BK_CUDA_OK(cudaGetLastError());
  }
  return BAKRON_OK;
}
}  // namespace

extern "C" size_t bakron_gram_workspace_bytes(int d, int k_chunk, int weighted) {
  if (d < 1 || d > GRAM_MAX_D || k_chunk < 1) return 0;
  const int64_t dp = round_up(d, PAD), kc = round_up(k_chunk, 32);
  return 256 + (size_t)(weighted ? 4 : 2) * (size_t)dp * (size_t)kc * 4;
}

extern "C" int bakron_gram(const void* X, int xdtype, int k, int d, int64_t ldx, const float* w,
                           float alpha, float beta, float* G, int64_t ldg, void* workspace,
                           size_t workspace_bytes, int sync, void* stream) {
  if (!X || !G || !workspace || k < 1 || d < 1 || d > GRAM_MAX_D || ldx < d || ldg < d)
    return BAKRON_ERR_INVALID_ARG;
  if (xdtype != BAKRON_F32 && xdtype != BAKRON_BF16) return BAKRON_ERR_INVALID_ARG;
  const int64_t dp = round_up(d, PAD);
  const bool bf16_ops = xdtype == BAKRON_BF16 && !w;
  const int op = !bf16_ops ? OP_TF32
                 : (d % 64 == 0 && ldx % 8 == 0 && (uintptr_t)X % 16 == 0) ? OP_BF16_MN
                                                                           : OP_BF16_K;
  const int64_t kq = bf16_ops ? 64 : 32;                  // samples of a slot
  const size_t per_sample = bf16_ops ? (size_t)dp * 2 : (size_t)(w ? 4 : 2) * dp * 4;
  if (workspace_bytes < 256 + per_sample * kq) return BAKRON_ERR_WORKSPACE;
  const size_t room = workspace_bytes - 256;
  const int BN = bf16_ops ? 256 : 128, R = BN / 128;
  const int nb = (int)(dp / GR_M), nh = nb / R;           // column blocks of the whole row blocks
  const int tiles = R * nh * (nh + 1) / 2 + (nb % R ? nh + 1 : 0);
  const size_t part_one = (size_t)tiles * GR_M * BN * 4;
  const int64_t kall = round_up(k, kq);
  // samples of a chunk: what fits, with the parts' room set aside when at least
  // half the samples (or 4096) still fit beside it; chunks of equal length.  Samples
  // that are read in place need no room; there a chunk bounds how many partial sums
  // are added one after the other: kc / 256 in registers, then k / kc in G.  Their
  // rounding errors' variance goes as kc^2 / (256 k) + k / kc, least at kc = 5 k^(2/3),
  // so a chunk is as long as would fit, or that if it is longer.  (In one pass over
  // 524288 samples the diagonal was off by 4.7e-7, in chunks of 32768 by 0.5e-7.)
  int splits = gram_splits(tiles, (int)(kall / kq));
  const int64_t fit = (int64_t)(room / per_sample) / kq * kq;
  int64_t kc = kall;
  if (op != OP_BF16_MN) {
    const size_t parts = splits > 1 ? splits * part_one : 0;
    const int64_t beside = parts < room ? (int64_t)((room - parts) / per_sample) / kq * kq : 0;
    if (beside >= std::min<int64_t>(kall, std::max<int64_t>(kq, std::min<int64_t>(kall / 2, 4096))))
      kc = std::min(kall, beside);
    else {
      kc = std::min(kall, fit);
      splits = 1;
    }
  } else {
    kc = std::min(kall, std::max(fit, round_up((int64_t)(5.0 * cbrt((double)k * k)), kq)));
    while (splits > 1 && splits * part_one > room) --splits;
  }
  kc = std::min<int64_t>(kc, (int64_t)1 << 30);
  const int64_t chunks = (kall + kc - 1) / kc;
  kc = std::min(kc, round_up((k + chunks - 1) / chunks, kq));
  BK_CUDA_OK(gram_attrs());
  cudaStream_t s = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  int* status = (int*)ws;
  char* planes = ws + 256;
  BK_CUDA_OK(cudaMemsetAsync(status, 0, 256, s));
  GramParams P{};
  P.tiles = tiles;
  P.d = d;
  P.alpha = alpha;
  P.G = G;
  P.ldg = ldg;
  P.status = status;
  P.spin_cycles = spin_cycles_from_env();
  P.part = (float*)(planes + (op == OP_BF16_MN ? 0 : per_sample * kc));
  P.b_exact = xdtype == BAKRON_BF16;              // bf16 is exact in tf32: lo plane zero
  P.a_exact = xdtype == BAKRON_BF16 && !w;
  for (int64_t t0 = 0; t0 < k; t0 += kc) {
    const int64_t kcl = std::min<int64_t>(kc, round_up(k - t0, kq));   // this chunk's samples
    P.beta = t0 == 0 ? beta : 1.f;
    P.nslots = (int)(kcl / kq);
    P.per_split = ceil_div(P.nslots, std::min(splits, gram_splits(tiles, P.nslots)));
    P.splits = ceil_div(P.nslots, P.per_split);
    CUtensorMap mA, mB;
    int rc;
    if (op == OP_BF16_MN) {
      const __nv_bfloat16* Xc = (const __nv_bfloat16*)X + t0 * ldx;
      const int64_t rows = std::min<int64_t>(kcl, k - t0);
      if (!map_bf16_mn(&mA, Xc, rows, d, ldx, 2) || !map_bf16_mn(&mB, Xc, rows, d, ldx, 4))
        return BAKRON_ERR_CUDA;
      rc = launch_gram<OP_BF16_MN>(mA, mB, P, s);
    } else if (op == OP_BF16_K) {
      __nv_bfloat16* Tb = (__nv_bfloat16*)planes;
      const int vec_ok = ((uintptr_t)X % 16 == 0 && ldx % 8 == 0) ? 1 : 0;
      dim3 tg((unsigned)(kcl / TR_TILE), (unsigned)(dp / TR_TILE));
      k_gram_transpose_bf16<<<tg, 256, 0, s>>>((const __nv_bfloat16*)X, k, d, ldx, (int)t0,
                                               (int)kc, vec_ok, Tb);
      BK_CUDA_OK(cudaGetLastError());
      if (!map_bf16_k(&mA, Tb, dp, kcl, kc, 128) || !map_bf16_k(&mB, Tb, dp, kcl, kc, 256))
        return BAKRON_ERR_CUDA;
      rc = launch_gram<OP_BF16_K>(mA, mB, P, s);
    } else {
      float* Th = (float*)planes;
      float* Tl = Th + dp * kc;
      float* Wh = w ? Tl + dp * kc : nullptr;
      float* Wl = w ? Wh + dp * kc : nullptr;
      dim3 sg((unsigned)(kcl / 32), (unsigned)(dp / 32));
      k_gram_split<<<sg, dim3(32, 8), 0, s>>>(X, xdtype, k, d, ldx, (int)t0, (int)kc, w, Th, Tl,
                                              Wh, Wl);
      BK_CUDA_OK(cudaGetLastError());
      if (!map_tf32(&mA, w ? Wh : Th, dp, kcl, kc, dp * kc * 4, P.a_exact) ||
          !map_tf32(&mB, Th, dp, kcl, kc, dp * kc * 4, P.b_exact))
        return BAKRON_ERR_CUDA;
      rc = launch_gram<OP_TF32>(mA, mB, P, s);
    }
    if (rc != BAKRON_OK) return rc;
  }
  if (!sync) return BAKRON_OK;
  return bakron_read_status(workspace, stream);
}

extern "C" int bakron_sample_sqnorms(const void* Y, int ydtype, int k, int d, int64_t ldy,
                                     float* out, void* stream) {
  if (!Y || !out || k < 1 || d < 1 || ldy < d) return BAKRON_ERR_INVALID_ARG;
  if (ydtype != BAKRON_F32 && ydtype != BAKRON_BF16) return BAKRON_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  k_sqnorms<<<(unsigned)(((int64_t)k * 32 + 255) / 256), 256, 0, s>>>(Y, ydtype, k, d, ldy, out);
  BK_CUDA_OK(cudaGetLastError());
  return BAKRON_OK;
}
