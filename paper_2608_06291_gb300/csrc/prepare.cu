// bakron_prepare: damping and unit-lower factors of the Kronecker Grams.
//
// Paper: Alg. 2, first two lines (L = Cholesky(H^-1), columns scaled to a unit
// diagonal), done once at top level (Appendix, equivalence proof, conventions);
// damping H + damp * mean(diag H) * I (Sec. 4, Appendix "Experiments").
//
// Route.  With R = RevCholesky(H_d) (R^T R = H_d, R lower), Cholesky(H_d^-1) =
// R^-1, so the unit-lower factor is R^-1 diag(R).  R comes from the ordinary
// Cholesky of the reversed matrix: J H_d J = C C^T gives R = J C^T J, hence
//     Lhat[i][j] = (C^-1)[d-1-j][d-1-i] * C[d-1-j][d-1-j]     (i >= j).
// So: reverse+damp -> blocked Cholesky of C -> inverse of C by halving -> flip,
// transpose and scale into the fp32 factor buffer.  No explicit H^-1.
//
// Precision and units.  An fp32 factorisation has relative error ~kappa * 2^-24
// (1e-5 at the condition numbers of the power-law Grams); error feedback
// multiplies that into the pre-rounding values, too close to the 1e-4 tie band
// on 4096-wide problems.  So the arithmetic is that of fp64 or better, but the
// GPU's fp64 units do 2 multiply-adds a cycle and SM (1.2 TFLOP/s in all), so
// all products of matrices run on the tensor cores, on exact slices (Ozaki et
// al. 2012, error-free transformations of matrix multiplication):
//   * Row and column i of the matrix are scaled by 2^-e_i (exact) so that the
//     diagonal lies in [1/4, 1): then |H_ij| < 1 and the rows of its Cholesky
//     factor have norm < 1, and both are kept as 64-bit fixed point, unit 2^-62
//     ("Q62"), which loses less than an fp64 of the same matrix would.
//   * An operand is cut into seven balanced base-256 digits, 56 bits (Q62 as it
//     is; fp64 matrices relative to a power of two above each row's norm), each
//     an fp16 integer of [-128, 127].  The 28 products of digit planes (i, j) with
//     i + j <= 6 are exact in the tensor cores' fp32 accumulators over 64 terms
//     (7 * 64 * 2^14 < 2^23); planes of equal i + j share one.  Their sum, shifted
//     8 bits apart, is formed in 64-bit integers modulo 2^64: it cannot be lost,
//     since the result itself is known to fit (Cauchy-Schwarz).  Dropped digit
//     products are below 2^-53 of the product of the norms.
// Diagonal 64 x 64 blocks are factored and inverted in fp64 by one CTA.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "common.cuh"
#include "tc_gemm.cuh"
#include "tcgen05.cuh"

namespace bakron {

namespace {

constexpr int NB = 64;            // Cholesky panel width, contraction chunk
constexpr int OT = 128;           // output tile of the sliced products
constexpr int SLICES = 7;
constexpr int WORKERS = 16;       // warps that cut operands and sum accumulators
constexpr int WT = 32 * WORKERS;
constexpr int OZ_THREADS = WT + 32;             // and one that issues the MMAs
constexpr uint32_t OPLANE = OT * 128;           // 128 rows of 64 fp16
constexpr uint32_t OZ_SMEM = 2 * SLICES * OPLANE + 1024 /*align*/ + 256 /*barriers*/;
constexpr int OUT_LD = OT + 2;                  // staged output row, 8-byte words
static_assert(OT * OUT_LD * 8 <= 2 * SLICES * OPLANE, "the output is staged over the planes");

// One side (A or B) of a prepare call.  C is dp x dp, row-major, 64-bit words:
// lower triangle and diagonal blocks Q62, first the scaled matrix, then its
// Cholesky factor; above the diagonal, during the inverse, intermediate products
// (fp64).  X: the factor's inverse (fp64, lower).
struct PrepSide {
  const float* H;
  int d, dp;
  long long* C;
  double* X;
  double* dinv;      // dp x 64: inverses of the diagonal blocks
  double* ldiag;     // dp: diagonal of the scaled factor
  double* mean;      // damp * mean(diag)
  int* e;            // dp: scale exponents
  int* f;            // dp: exponents of the rows of dinv
  int* xc;           // dp: exponents of columns (first halves) of X
  int* xr;           // dp: exponents of rows (second halves) of X
  int* tr;           // dp: exponents of rows of the intermediate
};
struct PrepArgs {
  PrepSide side[2];
  float damp;
  int* status;
  long long spin_cycles;
};

// ------------------------------------------------------------- exponents
// The least E (for a finite v > 0, up to rounding) with 1.05 v < 2^E.
__device__ __forceinline__ int exp_above(double v) {
  const int ex = (__double2hiint(v * 1.05) >> 20) & 0x7ff;
  return ex - 1022;
}
// The same for sqrt(v).
__device__ __forceinline__ int exp_above_sqrt(double v) {
  const int p = ((__double2hiint(v * 1.05) >> 20) & 0x7ff) - 1023;
  return (p >> 1) + 1;
}

// x * 2^u rounded to an integer, by integer operations (no fp64 unit); the
// caller's bounds keep it below 2^62, larger magnitudes give garbage.
__device__ __forceinline__ long long to_fix(double x, int u) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  const long long m = ex ? ((b & 0xfffffffffffffLL) | 0x10000000000000LL) : 0;
  const int sh = ex - 1075 + u;
  long long w;
  if (sh >= 0) {
    w = m << min(sh, 10);
  } else {
    const int r = min(-sh, 60);
    w = (m + (1LL << (r - 1))) >> r;
  }
  return b < 0 ? -w : w;
}

// x * 2^u for results inside fp64's normal range.
__device__ __forceinline__ double times_pow2(double x, int u) {
  return x == 0.0 ? 0.0 : __longlong_as_double(__double_as_longlong(x) + ((long long)u << 52));
}
// v * 2^u as fp64 (one rounding).
__device__ __forceinline__ double from_fix(long long v, int u) {
  return times_pow2(__ll2double_rn(v), u);
}

// ---------------------------------------------------------------- scaling
// damp * mean(diag) and the scale exponents of one side (blockIdx.x): row i
// of C is row d-1-i of H, rows past d the identity.
__global__ void __launch_bounds__(1024) k_prep_scale(const PrepArgs P) {
  const PrepSide& S = P.side[blockIdx.x];
  __shared__ double red[32];
  const int t = threadIdx.x;
  double acc = 0.0;
  for (int i = t; i < S.d; i += 1024) acc += (double)S.H[(int64_t)i * S.d + i];
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((t & 31) == 0) red[t >> 5] = acc;
  __syncthreads();
  if (t < 32) {
    acc = red[t];
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (t == 0) red[0] = (double)P.damp * (acc / (double)S.d);
  }
  __syncthreads();
  const double add = red[0];
  if (t == 0) *S.mean = add;
  bool bad = false;
  for (int i = t; i < S.dp; i += 1024) {
    double h = 1.0;
    if (i < S.d) h = (double)S.H[(int64_t)(S.d - 1 - i) * S.d + (S.d - 1 - i)] + add;
    if (!(h > 0.0) || !isfinite(h)) {
      bad = true;
      h = 1.0;
    }
    S.e[i] = exp_above_sqrt(h);
  }
  if (bad) raise_status(P.status, BAKRON_ERR_NOT_SPD);
}

// C from H (lower triangle read), zeros above the diagonal inside the diagonal
// 128 x 128 tiles.  32 x 32 per block, transposed through shared memory so that
// both sides are coalesced.  An off-diagonal entry as large as its row's and
// column's diagonal allow none to be (or not finite) is recorded as not SPD.
__global__ void __launch_bounds__(256) k_prep_load(const PrepArgs P) {
  const PrepSide& S = P.side[blockIdx.z];
  const int ti = blockIdx.y, tj = blockIdx.x;
  if (32 * ti >= S.dp || 32 * tj >= S.dp || tj / 4 > ti / 4) return;
  __shared__ float tile[32][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int d = S.d;
  for (int r = y; r < 32; r += 8) {
    const int i = 32 * ti + x, j = 32 * tj + r;
    tile[r][x] = (i < d && j <= i) ? S.H[(int64_t)(d - 1 - j) * d + (d - 1 - i)] : 0.f;
  }
  __syncthreads();
  const double add = *S.mean;
  bool bad = false;
  for (int r = y; r < 32; r += 8) {
    const int i = 32 * ti + r, j = 32 * tj + x;
    double h = (double)tile[x][r];
    if (i == j) h = i < d ? h + add : 1.0;
    // 1 or more (infinities and NaN too): beyond sqrt(H_ii H_jj) < 0.976
    const int u = 62 - S.e[i] - S.e[j], ex = (__double2hiint(h) >> 20) & 0x7ff;
    long long v = ex - 1023 + u >= 62 ? 1LL << 62 : to_fix(h, u);
    const long long lim = (1LL << 62) - (1LL << 56);   // 0.984
    if (v > lim || v < -lim) {
      bad = true;
      v = 0;
    }
    S.C[(int64_t)i * S.dp + j] = v;
  }
  if (bad) raise_status(P.status, BAKRON_ERR_NOT_SPD);
}

// ------------------------------------------------------- diagonal blocks
struct PotrfSmem {
  double s[NB][NB + 1];
  double inv[NB][NB + 1];   // and, above the diagonal, the products of its halving
  double pub[8][8];
  double rinv[NB];
};

__device__ __forceinline__ void workers_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(WT) : "memory");
}

// 1 / sqrt(p) for a normal p: the hardware's approximation and one cubic step.
__device__ __forceinline__ double rsqrt64(double p) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(p));
  const double e = fma(-p * r, r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}

// Factors the block of C at (k0, k0) and inverts the factor, by the first WT
// threads of the CTA.  Writes the factor to C, its inverse to dinv and to X's
// diagonal block, the exponents of the inverse's rows to f.  A pivot that is not
// positive raises NOT_SPD and is replaced by 1.
//
// The fp64 units take a warp's instruction every 64 cycles per scheduler, so
// the count of warp instructions sets the time: eight columns at a time, a
// thread per row with the columns' entries in registers (unscaled pivots and
// the eight rows they share are published once per column, 1 / sqrt is formed
// redundantly), then one update of the rest by all warps; the inverse by halving,
// all warps on each product.
__device__ void potrf_block(const PrepSide& S, int k0, PotrfSmem& M, int* status) {
  const int t = threadIdx.x;
  for (int e = t; e < NB * NB; e += WT) {
    const int r = e / NB, c = e % NB;
    M.s[r][c] = c <= r ? from_fix(S.C[(int64_t)(k0 + r) * S.dp + k0 + c], -62) : 0.0;
  }
  workers_sync();
  for (int c0 = 0; c0 < NB; c0 += 8) {
    if (t < NB && t >= (c0 & 32)) {   // whole warps: rows of finished warps are done
      const int r = t;
      const int live = NB - (c0 & 32);
      double a[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = M.s[r][c0 + j];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (r >= c0 && r < c0 + 8) M.pub[j][r - c0] = a[j];
        asm volatile("bar.sync 2, %0;" ::"r"(live) : "memory");
        double p = M.pub[j][j];
        if (!(p > 0.0)) {
          if (r == c0 + j) raise_status(status, BAKRON_ERR_NOT_SPD);
          p = 1.0;
        }
        const double ri = rsqrt64(p);
        const double l = (r == c0 + j ? p : a[j]) * ri, lr = l * ri;
        a[j] = l;
        if (r == c0 + j) M.rinv[r] = ri;
#pragma unroll
        for (int k = j + 1; k < 8; ++k) a[k] = fma(-lr, M.pub[j][k], a[k]);
      }
      if (r >= c0) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (c0 + j <= r) M.s[r][c0 + j] = a[j];
      }
    }
    workers_sync();
    const int b0 = c0 + 8, rem = NB - b0;
    for (int e = t; e < rem * (rem + 1) / 2; e += WT) {
      int r = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
      while ((r + 1) * (r + 2) / 2 <= e) ++r;
      while (r * (r + 1) / 2 > e) --r;
      const int c = e - r * (r + 1) / 2;
      double v = M.s[b0 + r][b0 + c];
#pragma unroll
      for (int k = 0; k < 8; ++k) v = fma(-M.s[b0 + r][c0 + k], M.s[b0 + c][c0 + k], v);
      M.s[b0 + r][b0 + c] = v;
    }
    workers_sync();
  }
  // the inverse: 8 x 8 diagonal blocks, a thread per column ...
  if (t < NB) {
    const int b = t & ~7, c = t & 7;
    double x[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < r; ++k) v = fma(M.s[b + r][b + k], x[k], v);
      x[r] = r == c ? M.rinv[b + r] : -v * M.rinv[b + r];
      if (r < c) x[r] = 0.0;
      M.inv[b + r][b + c] = x[r];
    }
  }
  workers_sync();
  // ... then [[X11, 0], [-X22 L21 X11, X22]] at 8, 16, 32
  for (int h = 8; h < NB; h *= 2) {
    for (int e = t; e < NB / 2 * h; e += WT) {
      const int i0 = 2 * h * (e / (h * h)), c = (e / h) % h, r = e % h;
      double v = 0.0;
      for (int k = c; k < h; ++k) v = fma(M.s[i0 + h + r][i0 + k], M.inv[i0 + k][i0 + c], v);
      M.inv[i0 + c][i0 + h + r] = v;                   // (L21 X11)[r][c], transposed
    }
    workers_sync();
    for (int e = t; e < NB / 2 * h; e += WT) {
      const int i0 = 2 * h * (e / (h * h)), r = (e / h) % h, c = e % h;
      double v = 0.0;
      for (int k = 0; k <= r; ++k) v = fma(-M.inv[i0 + h + r][i0 + h + k], M.inv[i0 + c][i0 + h + k], v);
      M.inv[i0 + h + r][i0 + c] = v;
    }
    workers_sync();
  }
  for (int e = t; e < NB * NB; e += WT) {
    const int r = e / NB, c = e % NB;
    const double x = c <= r ? M.inv[r][c] : 0.0;
    const int64_t o = (int64_t)(k0 + r) * S.dp + k0 + c;
    S.dinv[(int64_t)(k0 + r) * NB + c] = x;
    S.X[o] = x;
    S.C[o] = c <= r ? to_fix(M.s[r][c], 62) : 0;
    if (r == c) S.ldiag[k0 + r] = M.s[r][c];
  }
  for (int r = t >> 5; r < NB; r += WORKERS) {
    const int l = t & 31;
    unsigned m = l <= r ? __double2hiint(M.inv[r][l]) & 0x7fffffff : 0;
    if (l + 32 <= r) m = max(m, __double2hiint(M.inv[r][l + 32]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if (l == 0) S.f[k0 + r] = min(exp_above(__hiloint2double((int)m, -1)), 300);
  }
}

__global__ void __launch_bounds__(WT) k_prep_first(const PrepArgs P) {
  extern __shared__ __align__(16) unsigned char prep_smem[];
  pdl_wait();
  pdl_trigger();
  potrf_block(P.side[blockIdx.x], 0, *reinterpret_cast<PotrfSmem*>(prep_smem), P.status);
}

// --------------------------------------------------------- sliced products
// out(r, c) = sum_k a(r, k) b(c, k) over 128 x 128 tiles, operands and output by mode:
//   OZ_TRSM  the panel below a diagonal block: L = P Dinv^T, in place
//   OZ_SYRK  the matrix right of the panel: C -= L L^T (lower tiles); the CTA of
//            the first tile then factors the next diagonal block, which overlaps
//            with the other tiles
//   OZ_INV1  node (i0, h) of the inverse: R = X11^T L21^T, above C's diagonal
//   OZ_INV2  X21 = -X22 R^T
enum OzMode { OZ_TRSM, OZ_SYRK, OZ_INV1, OZ_INV2 };

// Seven digits of eight values (56-bit fixed point) to the planes: 16 bytes of
// a row each, in the 128-byte swizzled layout.
__device__ __forceinline__ void put_digits(unsigned char* planes, uint32_t plane, int row, int oct,
                                           const long long (&w)[8]) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const unsigned long long u = (unsigned long long)w[k] + 0x0080808080808080ULL;
    lo[k] = (uint32_t)u;
    hi[k] = (uint32_t)(u >> 32);
  }
  unsigned char* dst = planes + row * 128 + ((oct ^ (row & 7)) << 4);
#pragma unroll
  for (int s = 0; s < SLICES; ++s) {
    const int b = SLICES - 1 - s;                      // byte of the digit, biased by 128
    uint32_t o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t x = b < 4 ? lo[2 * k] : hi[2 * k], y = b < 4 ? lo[2 * k + 1] : hi[2 * k + 1];
      // fp16 1024 + byte, minus 1024 + 128
      uint32_t v = (__byte_perm(x, y, (b & 3) | ((b & 3) << 4) | ((4 + (b & 3)) << 8) |
                                          ((4 + (b & 3)) << 12)) &
                    0x00ff00ffu) |
                   0x64006400u;
      __half2 hv = __hsub2(*reinterpret_cast<__half2*>(&v), __half2half2(__ushort_as_half(0x6480)));
      o[k] = *reinterpret_cast<uint32_t*>(&hv);
    }
    *reinterpret_cast<uint4*>(dst + s * plane) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// kind::f16 with fp16 A and B (K-major), D fp32.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool oz_wait(uint64_t* bar, uint32_t parity, long long limit,
                                        volatile int* abort_flag) {
  if (mbar_test(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_test(bar, parity)) return true;
    if (*abort_flag || clock64() - t0 > limit) return false;
  }
}

// What one CTA computes: operand and output windows, all in units of entries.
struct OzTile {
  int ra, rb;        // first row of the a and of the b operand (in their matrices)
  int na, nb;        // rows of each (multiples of 64, at most 128)
  int k0, kn;        // chunks of 64: first and count, along the contraction
};

template <int MODE>
__device__ __forceinline__ bool oz_tile(const PrepSide& S, int arg, OzTile& T, int& i0) {
  if constexpr (MODE == OZ_TRSM) {
    const int t0 = arg + NB + OT * (int)blockIdx.x;
    i0 = arg;
    T = OzTile{t0, arg, min(OT, S.dp - t0), NB, 0, 1};
    return t0 < S.dp;
  } else if constexpr (MODE == OZ_SYRK) {
    const int t0 = arg + NB;
    i0 = arg;
    int I = (int)((sqrtf(8.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= (int)blockIdx.x) ++I;
    while (I * (I + 1) / 2 > (int)blockIdx.x) --I;
    const int J = (int)blockIdx.x - I * (I + 1) / 2;
    T = OzTile{t0 + OT * I, t0 + OT * J, min(OT, S.dp - t0 - OT * I), min(OT, S.dp - t0 - OT * J), 0, 1};
    return T.ra < S.dp;
  } else {
    const int h = arg;                                // first half; the second may be shorter
    i0 = 2 * h * (int)blockIdx.y;
    const int n2 = min(h, S.dp - i0 - h);
    if (n2 <= 0) return false;
    const int rows = MODE == OZ_INV1 ? h : n2, cols = MODE == OZ_INV1 ? n2 : h;
    const int tc = (h + OT - 1) / OT;                 // tiles across, of the widest node
    const int I = (int)blockIdx.x / tc, J = (int)blockIdx.x % tc;
    if (OT * I >= rows || OT * J >= cols) return false;
    if constexpr (MODE == OZ_INV1) {
      // columns j of X11 (zero above row j) against rows of L21
      const int kb = OT * I / NB;
      T = OzTile{OT * I, OT * J, min(OT, rows - OT * I), min(OT, cols - OT * J), kb, h / NB - kb};
    } else {
      // rows of X22 (zero right of the diagonal) against rows of R
      T = OzTile{OT * I, OT * J, min(OT, rows - OT * I), min(OT, cols - OT * J), 0,
                 min(n2, OT * (I + 1)) / NB};
    }
    return true;
  }
}

template <int MODE>
__global__ void __launch_bounds__(OZ_THREADS, 1) k_oz(const PrepArgs P, int arg) {
  extern __shared__ __align__(1024) unsigned char oz_smem[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)oz_smem + 1023) & ~(uintptr_t)1023);
  unsigned char* pa = smem;
  constexpr int BN = MODE == OZ_TRSM ? NB : OT;        // columns of the MMAs
  constexpr uint32_t b_plane = BN * 128;
  unsigned char* pb = smem + SLICES * OPLANE;
  uint64_t* accF = (uint64_t*)(smem + 2 * SLICES * OPLANE);   // [4] a digit sum is complete
  uint64_t* accE = accF + 4;                                   // [4] it has been read out
  uint64_t* done = accE + 4;
  uint32_t* tmem_slot = (uint32_t*)(done + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const PrepSide& S = P.side[blockIdx.z];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  constexpr int drains = BN / 32 * 4;                  // warps that read accumulators
  pdl_wait();
  pdl_trigger();
  OzTile T;
  int i0;
  if ((MODE == OZ_TRSM || MODE == OZ_SYRK) && arg + NB >= S.dp) return;
  if (!oz_tile<MODE>(S, arg, T, i0)) return;           // uniform over the CTA
  if (t == 0) {
    for (int a = 0; a < 4; ++a) {
      mbar_init(&accF[a], 1);
      mbar_init(&accE[a], drains);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == WORKERS) {
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
  const int64_t ld = S.dp;
  const int q = warp & 3, cg = warp >> 2;              // lane quarter, 32 columns
  const long long drain_limit = 4000000000LL;
  auto timed_out = [&]() {
    raise_status(P.status, BAKRON_ERR_TIMEOUT);
    *abort_flag = 1;
  };
  long long acc[32];
#pragma unroll
  for (int u = 0; u < 32; ++u) acc[u] = 0;
  bool issuing = true, dead = false;
  for (int ch = 0; ch < T.kn; ++ch) {
    const int kk = NB * (T.k0 + ch);
    if (warp < WORKERS) {
      // ---------------------------------------------------- cut the operands
      for (int u = t; u < OT * 8; u += WT) {
        int row, oct;
        if constexpr (MODE == OZ_INV1) {
          row = u & (OT - 1);
          oct = u >> 7;
        } else {
          row = u >> 3;
          oct = u & 7;
        }
        long long w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = 0;
        if (row < T.na) {
          if constexpr (MODE == OZ_TRSM || MODE == OZ_SYRK) {
            const longlong2* p = reinterpret_cast<const longlong2*>(
                S.C + (int64_t)(T.ra + row) * ld + i0 + 8 * oct);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const longlong2 v = __ldcg(p + k);
              w[2 * k] = (v.x + 64) >> 7;
              w[2 * k + 1] = (v.y + 64) >> 7;
            }
          } else if constexpr (MODE == OZ_INV1) {      // X11[k][j], k >= j
            const int j = T.ra + row;
            const int ex = 55 - S.xc[i0 + j];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int kr = kk + 8 * oct + k;
              if (kr >= j) w[k] = to_fix(S.X[(int64_t)(i0 + kr) * ld + i0 + j], ex);
            }
          } else {                                     // X22[i][k], k <= i
            const int i = T.ra + row;
            const int ex = 55 - S.xr[i0 + arg + i];
            const double2* p = reinterpret_cast<const double2*>(
                S.X + (int64_t)(i0 + arg + i) * ld + i0 + arg + kk + 8 * oct);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int kc = kk + 8 * oct + 2 * k;
              if (kc <= i) {
                const double2 v = p[k];
                w[2 * k] = to_fix(v.x, ex);
                if (kc + 1 <= i) w[2 * k + 1] = to_fix(v.y, ex);
              }
            }
          }
        }
        put_digits(pa, OPLANE, row, oct, w);
      }
      for (int u = t; u < BN * 8; u += WT) {
        const int row = u >> 3, oct = u & 7;
        long long w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = 0;
        if (row < T.nb) {
          if constexpr (MODE == OZ_TRSM || MODE == OZ_INV2) {
            const int ex = 55 - (MODE == OZ_TRSM ? S.f[i0 + row] : S.tr[i0 + T.rb + row]);
            const double2* p = reinterpret_cast<const double2*>(
                MODE == OZ_TRSM ? S.dinv + (int64_t)(i0 + row) * NB + 8 * oct
                                : (const double*)S.C + (int64_t)(i0 + T.rb + row) * ld + i0 + arg + kk + 8 * oct);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const double2 v = p[k];
              w[2 * k] = to_fix(v.x, ex);
              w[2 * k + 1] = to_fix(v.y, ex);
            }
          } else {
            const longlong2* p = reinterpret_cast<const longlong2*>(
                MODE == OZ_SYRK ? S.C + (int64_t)(T.rb + row) * ld + i0 + 8 * oct
                                : S.C + (int64_t)(i0 + arg + T.rb + row) * ld + i0 + kk + 8 * oct);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const longlong2 v = __ldcg(p + k);
              w[2 * k] = (v.x + 64) >> 7;
              w[2 * k + 1] = (v.y + 64) >> 7;
            }
          }
        }
        put_digits(pb, b_plane, row, oct, w);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (warp == WORKERS) {
      // ------------------------------------------------------------ products
      if (lane == 0 && issuing) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t da = smem_desc(smem_u32(pa)), db = smem_desc(smem_u32(pb));
        for (int s = 0; s < SLICES && issuing; ++s) {
          const int g = SLICES * ch + s, a = g & 3;
          if (g >= 4 && !oz_wait(&accE[a], (uint32_t)((g >> 2) - 1) & 1u, P.spin_cycles, abort_flag)) {
            if (!*abort_flag) timed_out();
            issuing = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          for (int i = 0; i <= s; ++i) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              mma_bf16(tmem + (uint32_t)(a * OT), da + (uint64_t)(i * (OPLANE >> 4) + 2 * k),
                       db + (uint64_t)((s - i) * (b_plane >> 4) + 2 * k), idesc_f16(OT, BN),
                       (i > 0 || k > 0) ? 1u : 0u);
          }
          mma_commit(&accF[a]);
        }
      }
      __syncwarp();
    } else if (warp < drains) {
      // ------------------------------------------- digit sums into 64 bits
      for (int s = 0; s < SLICES && !dead; ++s) {
        const int g = SLICES * ch + s, a = g & 3;
        int ok = 1;
        if (lane == 0) {
          ok = oz_wait(&accF[a], (uint32_t)(g >> 2) & 1u, P.spin_cycles, abort_flag) ? 1 : 0;
          if (!ok && !*abort_flag) timed_out();
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) {
          dead = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * OT + cg * 32);
        const int sh = 8 * (SLICES - 1 - s);
#pragma unroll
        for (int hlf = 0; hlf < 2; ++hlf) {
          uint32_t r[16];
          tmem_ld16(ta + 16 * hlf, r);
          tmem_wait_ld();
#pragma unroll
          for (int u = 0; u < 16; ++u)
            acc[16 * hlf + u] += (long long)__float2int_rn(__uint_as_float(r[u])) << sh;
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&accE[a]);
      }
    }
    __syncthreads();   // every MMA of the chunk is complete: its planes are free
  }
  if (warp == WORKERS && lane == 0) {
    mma_commit(done);
    if (!mbar_wait(done, 0, drain_limit)) timed_out();   // before anyone frees TMEM
  }
  __syncthreads();
  // ------------------------------------------------------------------- out
  long long* st = reinterpret_cast<long long*>(smem);
  if (warp < drains) {
    long long* o = st + (q * 32 + lane) * OUT_LD + cg * 32;
#pragma unroll
    for (int u = 0; u < 32; u += 2)
      *reinterpret_cast<longlong2*>(o + u) = make_longlong2(acc[u], acc[u + 1]);
  }
  __syncthreads();
  if (warp < WORKERS && !*abort_flag) {
    for (int r = warp; r < T.na; r += WORKERS) {
      const int er = MODE == OZ_INV1 ? S.xc[i0 + T.ra + r] : MODE == OZ_INV2 ? S.xr[i0 + arg + T.ra + r] : 0;
#pragma unroll
      for (int cb = 0; cb < BN / 64; ++cb) {
        const int c = 64 * cb + 2 * lane;
        if (c >= T.nb) continue;
        const longlong2 v = *reinterpret_cast<const longlong2*>(st + r * OUT_LD + c);
        if constexpr (MODE == OZ_TRSM) {
          const int f0 = min(max(S.f[i0 + c], 0), 62), f1 = min(max(S.f[i0 + c + 1], 0), 62);
          *reinterpret_cast<longlong2*>(S.C + (int64_t)(T.ra + r) * ld + i0 + c) =
              make_longlong2((long long)((unsigned long long)v.x << f0),
                             (long long)((unsigned long long)v.y << f1));
        } else if constexpr (MODE == OZ_SYRK) {
          longlong2* p = reinterpret_cast<longlong2*>(S.C + (int64_t)(T.ra + r) * ld + T.rb + c);
          const longlong2 old = __ldcg(p);
          *p = make_longlong2(old.x - v.x, old.y - v.y);
        } else if constexpr (MODE == OZ_INV1) {
          *reinterpret_cast<double2*>((double*)S.C + (int64_t)(i0 + T.ra + r) * ld + i0 + arg + T.rb + c) =
              make_double2(from_fix(v.x, er - 62), from_fix(v.y, er - 62));
        } else {
          const int e0 = S.tr[i0 + T.rb + c], e1 = S.tr[i0 + T.rb + c + 1];
          *reinterpret_cast<double2*>(S.X + (int64_t)(i0 + arg + T.ra + r) * ld + i0 + T.rb + c) =
              make_double2(from_fix(-v.x, er + e0 - 62), from_fix(-v.y, er + e1 - 62));
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == WORKERS)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  if constexpr (MODE == OZ_SYRK) {
    if (blockIdx.x == 0 && warp < WORKERS)
      potrf_block(S, arg + NB, *reinterpret_cast<PotrfSmem*>(smem), P.status);
  }
}

// ------------------------------------------------------------------ norms
// A power of two above the norm whose squared value (fp32) and largest entry
// (high word) are given; without a usable square, from the largest entry and n.
__device__ __forceinline__ int norm_exp(float ss, unsigned mx, int n) {
  if (isfinite(ss) && ss > 1e-30f) return exp_above_sqrt((double)ss * 1.01);
  if (mx == 0) return 0;
  return exp_above(__hiloint2double((int)mx, -1)) + (32 - __clz(n)) / 2 + 1;
}

// Node (i0 = 2 h blockIdx.y, h) of the inverse.  part 0: columns of X11 (32 a
// block); part 1: rows of X22; part 2: rows of R (8 a block).
__global__ void __launch_bounds__(256) k_prep_norms(const PrepArgs P, int h, int part, int blocks0) {
  pdl_wait();
  pdl_trigger();
  const PrepSide& S = P.side[blockIdx.z];
  const int i0 = 2 * h * (int)blockIdx.y, n2 = min(h, S.dp - i0 - h);
  if (n2 <= 0) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t ld = S.dp;
  if (part == 0 && (int)blockIdx.x < blocks0) {
    __shared__ float ssum[8][32];
    __shared__ unsigned smax[8][32];
    const int j0 = 32 * (int)blockIdx.x, j = j0 + lane;
    float ss = 0.f;
    unsigned mx = 0;
    for (int k = j0 + warp; k < h; k += 8) {
      if (k < j) continue;
      const double x = S.X[(int64_t)(i0 + k) * ld + i0 + j];
      const float xf = (float)x;
      ss = fmaf(xf, xf, ss);
      mx = max(mx, __double2hiint(x) & 0x7fffffffu);
    }
    ssum[warp][lane] = ss;
    smax[warp][lane] = mx;
    __syncthreads();
    if (warp == 0) {
      for (int w = 1; w < 8; ++w) {
        ss += ssum[w][lane];
        mx = max(mx, smax[w][lane]);
      }
      S.xc[i0 + j] = norm_exp(ss, mx, h);
    }
    return;
  }
  const bool rows_x = part == 0;
  const int r = 8 * ((int)blockIdx.x - (rows_x ? blocks0 : 0)) + warp;
  if (r >= (rows_x ? n2 : h)) return;
  const double* p = rows_x ? S.X + (int64_t)(i0 + h + r) * ld + i0 + h
                           : (const double*)S.C + (int64_t)(i0 + r) * ld + i0 + h;
  const int n = rows_x ? r + 1 : n2;
  float ss = 0.f;
  unsigned mx = 0;
  for (int k = lane; k < n; k += 32) {
    const double x = p[k];
    const float xf = (float)x;
    ss = fmaf(xf, xf, ss);
    mx = max(mx, __double2hiint(x) & 0x7fffffffu);
  }
  for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) (rows_x ? S.xr + i0 + h : S.tr + i0)[r] = norm_exp(ss, mx, n);
}

// --------------------------------------------------------------- assembly
// Lhat[i][j] = Xinv[d-1-j][d-1-i] * C[d-1-j][d-1-j]  (i > j), 1 on the
// diagonal, 0 above, identity on the padding; rdiag[i] = C[d-1-i][d-1-i]; Xinv
// and C of the unscaled matrix.  Overwrites S.C (the planes it was kept in).
__global__ void __launch_bounds__(256) k_assemble(const PrepSide S, float* L, float* Llo, float* rdiag) {
  __shared__ float tile[32][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  const int d = S.d, dp = S.dp;
  if (by + 31 >= bx) {
    for (int r = y; r < 32; r += 8) {
      const int j = bx + r, i = by + x;   // destination column and row
      float v = 0.f;
      if (i < d && j < d && i > j) {
        const int a = d - 1 - j, b = d - 1 - i;
        v = (float)times_pow2(S.X[(int64_t)a * dp + b] * S.ldiag[a], S.e[a] - S.e[b]);
      }
      tile[r][x] = v;
    }
  }
  __syncthreads();
  for (int r = y; r < 32; r += 8) {
    const int i = by + r, j = bx + x;
    float v = by + 31 >= bx ? tile[x][r] : 0.f;
    if (i == j) v = 1.f;
    const float hi = tf32_hi(v);
    L[(int64_t)i * dp + j] = hi;
    Llo[(int64_t)i * dp + j] = v - hi;
  }
  if (blockIdx.x == 0 && y == 0) {
    const int i = by + x;
    rdiag[i] = i < d ? (float)times_pow2(S.ldiag[d - 1 - i], S.e[d - 1 - i]) : 1.f;
  }
}

cudaError_t prep_attrs() {
  static std::mutex mu;
  static bool done = false;
  std::lock_guard<std::mutex> lk(mu);
  if (done) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k_prep_first, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(PotrfSmem));
  auto set = [&](const void* f) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM);
  };
  set((const void*)k_oz<OZ_TRSM>);
  set((const void*)k_oz<OZ_SYRK>);
  set((const void*)k_oz<OZ_INV1>);
  set((const void*)k_oz<OZ_INV2>);
  if (e == cudaSuccess) done = true;
  return e;
}

// Where one side keeps its matrices: C in the factor planes that the assembly
// writes last, small arrays in the leaf blocks (written after that), X in the
// workspace.
PrepSide make_side(const float* H, int d, int64_t dp, char* planes, char* scratch, char* x) {
  PrepSide S;
  S.H = H;
  S.d = d;
  S.dp = (int)dp;
  S.C = (long long*)planes;
  S.X = (double*)x;
  S.dinv = (double*)scratch;
  S.ldiag = S.dinv + dp * NB;
  S.mean = S.ldiag + dp;
  S.e = (int*)(S.mean + 2);
  S.f = S.e + dp;
  S.xc = S.f + dp;
  S.xr = S.xc + dp;
  S.tr = S.xr + dp;
  return S;
}
// bytes of `scratch` per row of a side: 64 + 1 fp64, five ints (and the mean)
static_assert((NB + 1) * 8 + 5 * 4 + 16 <= LEAF_BLOCKS * LEAF_BLOCK_FLOATS * 4 / TILE, "scratch fits the leaf blocks");

}  // namespace

int prepare_impl(const float* A, const float* B, int m, int n, float damp, void* factors,
                 void* workspace, cudaStream_t s) {
  FactorLayout fl(m, n);
  PrepareLayout pl(m, n);
  char* f = (char*)factors;
  char* ws = (char*)workspace;
  BK_CUDA_OK(prep_attrs());
  BK_CUDA_OK(cudaMemsetAsync(ws + pl.off_status, 0, 256, s));
  PrepArgs P;
  P.side[0] = make_side(A, n, fl.np, f + fl.off_LAH, f + fl.off_LAblk, ws + pl.off_X);
  P.side[1] = make_side(B, m, fl.mp, f + fl.off_LBH, f + fl.off_LBblk,
                        ws + pl.off_X + (size_t)(fl.np * fl.np) * 8);
  P.damp = damp;
  P.status = (int*)(ws + pl.off_status);
  P.spin_cycles = spin_cycles_from_env();
  const int dp = (int)(fl.np > fl.mp ? fl.np : fl.mp);   // both sides side by side (grid.z)
  auto up = [](int a, int b) { return (unsigned)((a + b - 1) / b); };
  k_prep_scale<<<2, 1024, 0, s>>>(P);
  k_prep_load<<<dim3(dp / 32, dp / 32, 2), 256, 0, s>>>(P);
  BK_CUDA_OK(cudaGetLastError());
  const dim3 oz(OZ_THREADS);
  BK_CUDA_OK(launch_pdl(k_prep_first, dim3(2), dim3(WT), sizeof(PotrfSmem), s, P));
  for (int k0 = 0; k0 + NB < dp; k0 += NB) {
    const unsigned nt = up(dp - k0 - NB, OT);
    BK_CUDA_OK(launch_pdl(k_oz<OZ_TRSM>, dim3(nt, 1, 2), oz, OZ_SMEM, s, P, k0));
    BK_CUDA_OK(launch_pdl(k_oz<OZ_SYRK>, dim3(nt * (nt + 1) / 2, 1, 2), oz, OZ_SMEM, s, P, k0));
  }
  for (int h = NB; h < dp; h *= 2) {
    const unsigned nodes = up(dp, 2 * h), tiles = up(h, OT) * up(h, OT);
    BK_CUDA_OK(launch_pdl(k_prep_norms, dim3(up(h, 32) + up(h, 8), nodes, 2), dim3(256), 0, s, P, h,
                          0, (int)up(h, 32)));
    BK_CUDA_OK(launch_pdl(k_oz<OZ_INV1>, dim3(tiles, nodes, 2), oz, OZ_SMEM, s, P, h));
    BK_CUDA_OK(launch_pdl(k_prep_norms, dim3(up(h, 8), nodes, 2), dim3(256), 0, s, P, h, 1, 0));
    BK_CUDA_OK(launch_pdl(k_oz<OZ_INV2>, dim3(tiles, nodes, 2), oz, OZ_SMEM, s, P, h));
  }
  k_assemble<<<dim3((unsigned)(fl.np / 32), (unsigned)(fl.np / 32)), 256, 0, s>>>(
      P.side[0], (float*)(f + fl.off_LAH), (float*)(f + fl.off_LAL), (float*)(f + fl.off_rA));
  k_assemble<<<dim3((unsigned)(fl.mp / 32), (unsigned)(fl.mp / 32)), 256, 0, s>>>(
      P.side[1], (float*)(f + fl.off_LBH), (float*)(f + fl.off_LBL), (float*)(f + fl.off_rB));
  BK_CUDA_OK(cudaGetLastError());
  return build_leaf_blocks(fl, f, s);
}

}  // namespace bakron
