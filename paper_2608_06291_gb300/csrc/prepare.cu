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
// on 4096-wide problems.  So the factors have to be as good as fp64's, but the
// GPU's fp64 units do 2 multiply-adds a cycle and SM (1.2 TFLOP/s in all), so
// all products of matrices run on the tensor cores, on exact slices (Ozaki et
// al. 2012, error-free transformations of matrix multiplication):
//   * Row and column i of the matrix are scaled by 2^-e_i (exact) so that the
//     diagonal lies in [1/4, 1): then |H_ij| < 1 and the rows of its Cholesky
//     factor have norm < 1, and both are kept as 64-bit fixed point, unit 2^-63
//     ("Q63"), which loses less than an fp64 of the same matrix would.
//   * An operand is cut into seven balanced base-256 digits, its upper 56 bits (Q63
//     as it is; fp64 matrices relative to a power of two above each row's norm),
//     each an fp16 integer of [-128, 127].  The 34 products of digit planes (i, j) with
//     i + j <= 7 are exact in the tensor cores' fp32 accumulators over 64 terms
//     (7 * 64 * 2^14 < 2^23); planes of equal i + j share one.  Their sum, shifted
//     8 bits apart (the last one rounded to the unit), is formed in 64-bit integers
//     modulo 2^64, which is right where the result itself fits.  The digit products
//     that are dropped are at most 2^-55 of the product of the norms per 64 terms and
//     some 2^-61 typically, the operands' rounding to 56 bits 2^-52 and 2^-56.  (With
//     the 28 products of i + j <= 6 the dropped ones were 2^-53 typically, and the
//     factors five to fifteen times further off than an fp64 factorisation's.)
//   * Of a positive definite matrix every result fits: entries of the factor and of
//     the Schur complements, and sums over a factor's rows, are below 0.976
//     (Cauchy-Schwarz).  Of another it need not, and a wrapped pivot could look
//     positive.  So each step raises NOT_SPD where its own result does not fit: the
//     sums of a panel's products by their leading digits (OZ_FIT), a factor's entries
//     by their size, a Schur complement by its subtraction's overflow and by a
//     diagonal that is not positive.  Nothing that wrapped is used unnoticed.
// Diagonal 64 x 64 blocks are factored and inverted by one CTA, in fp64 and 56-bit
// integers.
//
// Measured on GB300, both sides 4096: 160.2 ms with the products on the fp64 units,
// 10.5 so; 1531 + 1000: 26.7 -> 3.1.  (Of the 10.5, 0.65 are the last six digit
// products, 0.25 the looks at what fits, 0.27 CUDA's reciprocal and root.)
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "common.cuh"
#include "tc_gemm.cuh"
#include "tcgen05.cuh"

namespace bakron {

namespace {

constexpr int NB = 64;            // Cholesky panel width, contraction chunk
constexpr int OT = 128;           // output tile of the sliced products
constexpr int SLICES = 7;
// Sixteen warps cut operands and sum accumulators; thread 0 issues the MMAs
// between its other work (a warp of its own would leave 96 registers a thread).
constexpr int WORKERS = 16;
constexpr int WT = 32 * WORKERS;
constexpr uint32_t OPLANE = OT * 128;           // 128 rows of 64 fp16
constexpr uint32_t OZ_SMEM = 2 * SLICES * OPLANE + 1024 /*align*/ + 256 /*barriers*/;
constexpr int OUT_LD = OT + 2;                  // staged output row, 8-byte words
static_assert(OT * OUT_LD * 8 <= 2 * SLICES * OPLANE, "the output is staged over the planes");

// One side (A or B) of a prepare call.  C is dp x dp, row-major, 64-bit words:
// lower triangle and diagonal blocks Q63, first the scaled matrix, then its
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
// caller's bounds keep it below 2^63, larger magnitudes give garbage.
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
    const int u = 63 - S.e[i] - S.e[j], ex = (__double2hiint(h) >> 20) & 0x7ff;
    long long v = ex - 1023 + u >= 63 ? 0x7fffffffffffffffLL : to_fix(h, u);
    const long long lim = 0x7eLL << 56;   // 0.984
    if (v > lim || v < -lim) {
      bad = true;
      v = 0;
    }
    S.C[(int64_t)i * S.dp + j] = v;
  }
  if (bad) raise_status(P.status, BAKRON_ERR_NOT_SPD);
}

// ------------------------------------------------------- diagonal blocks
// A Q63 value for products in integers: ah * 2^25 + al, unit 2^-56 (ah 32 bits
// with the sign, al 25).
__device__ __forceinline__ int2 split56(long long v) {
  const long long u = v + 64;   // rounded
  return make_int2((int)(u >> 32), (int)((uint32_t)u >> 7));
}
// sum += a b, in two parts: s1 of unit 2^-62, s2 of unit 2^-87 (al * bl, below
// 2^-62, is left out).  The sums are right modulo 2^64: the products' sum itself
// is below 1 by the norms of the rows that are multiplied.
__device__ __forceinline__ void mac56(long long& s1, long long& s2, int2 a, int2 b) {
  s1 += (long long)a.x * b.x;
  s2 += (long long)a.x * b.y;
  s2 += (long long)a.y * b.x;
}
__device__ __forceinline__ long long sum56(long long s1, long long s2) {   // Q63
  return (long long)((unsigned long long)s1 << 1) + (s2 >> 24);
}

constexpr int PH = NB / 2;       // the inverse's last halving, in integers
struct PotrfSmem {
  long long a[NB][NB + 1];       // Q63: the block, then its factor
  double inv[NB][NB + 1];        // the inverse; above the diagonal, products of its halving
  double cur[NB][9];             // the eight columns being factored
  __align__(16) int2 l8[2][NB][10]; // the same, factored, split (rows of 80 bytes: no conflicts);
                                    // by the parity of the eight
  int2 xs[PH][PH + 1];           // columns of X11, then rows of X22 (split)
  int2 ts[PH][PH + 1];           // L21, then columns of L21 X11 (split)
  int ec[PH], er[PH], et[PH];
  double col[8][NB];             // their entries as each became the pivot column
  double rinv[NB], diag[NB];
};

__device__ __forceinline__ void workers_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(WT) : "memory");
}

// An exponent above three times the largest magnitude of a warp's values (32
// values of that exponent have a norm below one: sqrt(32) < 2^3 / 1.05).
__device__ __forceinline__ int warp_exp8(double x) {
  const unsigned m = __reduce_max_sync(0xffffffffu, (unsigned)__double2hiint(x) & 0x7fffffffu);
  return (int)(m >> 20) - 1022 + 3;
}

// Factors the block of C at (k0, k0) and inverts the factor, by all WT threads
// of the CTA.  Writes the factor to C, its inverse to dinv and to X's diagonal
// block, the exponents of the inverse's rows to f.  A pivot that is not positive
// raises NOT_SPD and is replaced by 1; so does anything that does not fit.
//
// The fp64 units take a warp's instruction every 64 cycles per scheduler, so
// the count of those sets the time, and what can be is done in integers.  Eight
// columns at a time in fp64: four warps, two threads a row with every other column
// in registers; per column the entries are published, and a row's entry over the
// pivot (a reciprocal) times the eight rows' entries updates what it holds, so that
// the square roots wait for the end, a lane each (with the quotient itself in place
// of the reciprocal both sides 4096 took 12.23 ms, not 10.47).  Then one update of the
// rest by all warps on split 56-bit values (three 32 x 32 + 64 multiply-adds each).
// The inverse by halving: 8 x 8 blocks and the first two levels in fp64, the last
// in integers.
__device__ void potrf_block(const PrepSide& S, int k0, PotrfSmem& M, int* status) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  bool bad = false;
  // this thread's entries of a lower triangle of up to 63 rows, row by row
  constexpr int TRI = ((NB - 8) * (NB - 7) / 2 + WT - 1) / WT;
  int tr[TRI], tc[TRI];
#pragma unroll
  for (int i = 0; i < TRI; ++i) {
    const int e = t + WT * i;
    int r = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= e) ++r;
    while (r * (r + 1) / 2 > e) --r;
    tr[i] = r;
    tc[i] = e - r * (r + 1) / 2;
  }
#pragma unroll
  for (int i = 0; i < NB * NB / WT; ++i) {
    const int e = t + WT * i, r = e / NB, c = e % NB;
    const long long v = c <= r ? __ldcg(S.C + (int64_t)(k0 + r) * S.dp + k0 + c) : 0;
    M.a[r][c] = v;
    if (c < 8) M.cur[r][c] = from_fix(v, -63);
  }
  workers_sync();
  // Whether row r of the eight columns from c on, and the update by them, fit: entries
  // below one, their norm too (0.99, to 2^-11), and a positive diagonal left.
  auto fits = [&](int r, int c, bool diagonal) {
    const int2* l = M.l8[(c >> 3) & 1][r];
    unsigned norm = 0;                                  // unit 2^-28
    bool ok = !diagonal || M.a[r][r] > 0;
    for (int j = 0; j < 8; ++j) {
      if (c + j > r) break;
      ok &= (__double2hiint(M.inv[r][c + j]) & 0x7fffffff) < 0x3ff00000;
      const int l14 = l[j].x >> 17;                     // unit 2^-14
      norm += (unsigned)(l14 * l14);
    }
    return ok && (r < c + 8 || norm <= 265751040u);
  };
  for (int c0 = 0; c0 < NB; c0 += 8) {
    int2 (*l8)[10] = M.l8[(c0 >> 3) & 1];
    // what the last eight columns left is looked over by two idle warps
    if (c0 > 0 && t >= 2 * NB && t < 3 * NB && t - 2 * NB >= c0 - 8)
      bad |= !fits(t - 2 * NB, c0 - 8, t - 2 * NB >= c0 + 8);
    // thread (row r, half hc): columns c0 + hc, + 2, + 4, + 6; a warp whose rows are
    // all done stays away
    if (t < 2 * NB && (t & (NB - 1)) >= (c0 & 32)) {
      const int r = t & (NB - 1), hc = t / NB, live = 2 * (NB - (c0 & 32));
      double a[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = r >= c0 ? M.cur[r][2 * i + hc] : 0.0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (hc == (j & 1)) M.col[j][r] = a[j / 2];
        asm volatile("bar.sync 2, %0;" ::"r"(live) : "memory");
        if (j == 7) break;
        double p = M.col[j][c0 + j];
        if (!(p > 0.0)) p = 1.0;
        const double lr = M.col[j][r] * (1.0 / p);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (2 * i + hc > j) a[i] = fma(-lr, M.col[j][c0 + 2 * i + hc], a[i]);
      }
      if (hc == 0 && r >= c0 && r < c0 + 8) {   // a pivot per lane
        double p = M.col[r - c0][r];
        if (!(p > 0.0)) {
          raise_status(status, BAKRON_ERR_NOT_SPD);
          p = 1.0;
        }
        const double ri = rsqrt(p);
        M.rinv[r] = ri;
        M.diag[r] = p * ri;
        S.ldiag[k0 + r] = p * ri;
      }
      asm volatile("bar.sync 2, %0;" ::"r"(live) : "memory");
      if (r >= c0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int j = 2 * i + hc;
          const double l = r == c0 + j ? M.diag[r] : a[i] * M.rinv[c0 + j];
          const long long v = c0 + j <= r ? to_fix(l, 63) : 0;
          if (c0 + j <= r) M.a[r][c0 + j] = v;
          l8[r][j] = split56(v);
          M.inv[r][c0 + j] = l;            // the factor in fp64, for the halving
        }
      }
    }
    workers_sync();
    const int b0 = c0 + 8, rem = NB - b0;
#pragma unroll
    for (int i = 0; i < TRI; ++i) {
      if (t + WT * i >= rem * (rem + 1) / 2) continue;
      const int r = b0 + tr[i], c = b0 + tc[i];
      const int4* lr = reinterpret_cast<const int4*>(l8[r]);
      const int4* lc = reinterpret_cast<const int4*>(l8[c]);
      long long s1 = 0, s2 = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int4 x = lr[k], y = lc[k];
        mac56(s1, s2, make_int2(x.x, x.y), make_int2(y.x, y.y));
        mac56(s1, s2, make_int2(x.z, x.w), make_int2(y.z, y.w));
      }
      const long long old = M.a[r][c], sum = sum56(s1, s2);
      const long long v = (long long)((unsigned long long)old - (unsigned long long)sum);
      bad |= ((old ^ sum) & (old ^ v)) < 0;
      M.a[r][c] = v;
      if (tc[i] < 8) M.cur[r][tc[i]] = from_fix(v, -63);
    }
    if (rem == 0 && t >= 3 * NB - 8 && t < 3 * NB) bad |= !fits(t - 2 * NB, c0, false);
    workers_sync();
  }
  if (bad) raise_status(status, BAKRON_ERR_NOT_SPD);
  // M.inv holds the factor (fp64).  The inverse: 8 x 8 diagonal blocks, a thread
  // per column ...
  double x8[8];
  if (t < NB) {
    const int b = t & ~7, c = t & 7;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < r; ++k) v = fma(M.inv[b + r][b + k], x8[k], v);
      x8[r] = r == c ? M.rinv[b + r] : -v * M.rinv[b + r];
      if (r < c) x8[r] = 0.0;
    }
    asm volatile("bar.sync 2, %0;" ::"n"(NB) : "memory");
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r >= c) M.inv[b + r][b + c] = x8[r];
  }
  workers_sync();
  // ... then [[X11, 0], [-X22 L21 X11, X22]] at 8 and 16: L21 is read where X21 goes
#pragma unroll
  for (int h = 8; h < PH; h *= 2) {
    for (int e = t; e < NB / 2 * h; e += WT) {
      const int i0 = 2 * h * (e / (h * h)), c = (e / h) % h, r = e % h;
      double v = 0.0;
      for (int k = c; k < h; ++k) v = fma(M.inv[i0 + h + r][i0 + k], M.inv[i0 + k][i0 + c], v);
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
  // at 32, in integers relative to the norms of X11's columns, X22's rows and the
  // columns of L21 X11 (a warp per column or row)
  for (int c = warp; c < PH; c += WORKERS) {
    const double x = lane >= c ? M.inv[lane][c] : 0.0;
    const int e = warp_exp8(x);
    M.xs[c][lane] = split56(to_fix(x, 63 - e));
    M.ts[c][lane] = split56(M.a[PH + c][lane]);        // row c of L21
    if (lane == 0) M.ec[c] = e;
  }
  workers_sync();
  long long tv[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {                        // column c of L21 X11, lane = row
    const int c = warp + WORKERS * i;
    long long s1 = 0, s2 = 0;
    for (int k = c; k < PH; ++k) mac56(s1, s2, M.ts[lane][k], M.xs[c][k]);
    tv[i] = sum56(s1, s2);
  }
  workers_sync();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int c = warp + WORKERS * i;
    const unsigned long long mag = (unsigned long long)(tv[i] < 0 ? -tv[i] : tv[i]);
    const int z = max(__clz((int)__reduce_max_sync(0xffffffffu, (unsigned)(mag >> 32))) - 1, 0);
    // up by z bits to the top, then 3 down for the norm
    M.ts[c][lane] = split56((long long)((unsigned long long)tv[i] << z) >> 3);
    if (lane == 0) M.et[c] = M.ec[c] - z + 3;
    const double x = lane <= c ? M.inv[PH + c][PH + lane] : 0.0;   // row c of X22
    const int e = warp_exp8(x);
    M.xs[c][lane] = split56(to_fix(x, 63 - e));
    if (lane == 0) M.er[c] = e;
  }
  workers_sync();
#pragma unroll
  for (int i = 0; i < 2; ++i) {                        // row r of X21, lane = column
    const int r = warp + WORKERS * i;
    long long s1 = 0, s2 = 0;
    for (int k = 0; k <= r; ++k) mac56(s1, s2, M.xs[r][k], M.ts[lane][k]);
    M.inv[PH + r][lane] = from_fix(-sum56(s1, s2), M.er[r] + M.et[lane] - 63);
  }
  workers_sync();
#pragma unroll
  for (int i = 0; i < NB * NB / WT; ++i) {
    const int e = t + WT * i, r = e / NB, c = e % NB;
    const double x = c <= r ? M.inv[r][c] : 0.0;
    const int64_t o = (int64_t)(k0 + r) * S.dp + k0 + c;
    S.dinv[(int64_t)(k0 + r) * NB + c] = x;
    S.X[o] = x;
    S.C[o] = M.a[r][c];
  }
  for (int r = warp; r < NB; r += WORKERS) {
    unsigned m = lane <= r ? __double2hiint(M.inv[r][lane]) & 0x7fffffff : 0;
    if (lane + 32 <= r) m = max(m, __double2hiint(M.inv[r][lane + 32]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) S.f[k0 + r] = min(exp_above(__hiloint2double((int)m, -1)), 300);
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
// 128 x 128 tiles and 64-deep chunks, because the fourteen digit planes of one chunk
// just fit shared memory.  What bounds a chunk: cutting the operands (6 to 9 thousand
// cycles, integer work and the loads' latency), then 136 MMAs of 62 cycles and the
// sums, which partly run beside them (some 14 thousand); nothing of the next chunk can
// start meanwhile.  10 to 11.5 us, against 20 to 28 with shifts by run-time counts and
// a warp of its own for the MMAs.  Sixteen warps leave 128 registers a thread, over
// which OZ_INV1, with its strided loads, spills 160 bytes.
enum OzMode { OZ_TRSM, OZ_SYRK, OZ_INV1, OZ_INV2 };

// Seven digits of eight values (Q63) to the planes: 16 bytes of a row each, in
// the 128-byte swizzled layout.  The 128s added to every byte make the digits
// balanced (the last one rounds the byte that is dropped).
__device__ __forceinline__ void put_digits(unsigned char* planes, uint32_t plane, int row, int oct,
                                           const long long (&w)[8]) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const unsigned long long u = (unsigned long long)w[k] + 0x8080808080808080ULL;
    lo[k] = (uint32_t)u;
    hi[k] = (uint32_t)(u >> 32);
  }
  unsigned char* dst = planes + row * 128 + ((oct ^ (row & 7)) << 4);
#pragma unroll
  for (int s = 0; s < SLICES; ++s) {
    const int b = SLICES - s;                          // byte of the digit, biased by 128
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

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                 "=r"(r[7])
               : "r"(taddr));
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

// An integer x, |x| <= 2^22, held in fp32: its bits after adding 1.5 * 2^23 are
// OZ_BIAS + x, for one addition instead of a conversion (a quarter of its rate).
constexpr uint32_t OZ_BIAS = 0x4B400000u;
__device__ __forceinline__ uint32_t biased_int(uint32_t f) {
  return __float_as_uint(__uint_as_float(f) + 12582912.f);
}

// An integer x, |x| < 2^23, held in fp32, by additions: its half rounded to an
// integer, and what is left (-1, 0 or 1).
__device__ __forceinline__ uint32_t wide_int(uint32_t f) {
  const float x = __uint_as_float(f), h = fmaf(x, 0.5f, 12582912.f);
  const float rest = fmaf(h - 12582912.f, -2.f, x);
  return 2 * (__float_as_uint(h) - OZ_BIAS) + (__float_as_uint(rest + 12582912.f) - OZ_BIAS);
}

// The sum of a panel's products over 64 terms, 2^-14 as the unit, from its two leading
// sums of digit products (the others add less than 49): up to this it is below 0.992
// and fits; a positive definite matrix has at most 0.953 (15 650).
constexpr float OZ_FIT = 16200.f;
__device__ __forceinline__ float leading(uint32_t f0, uint32_t f1) {
  return fabsf(fmaf(__uint_as_float(f1), 1.f / 256.f, __uint_as_float(f0)));
}

// Four 8-byte words, 32-byte aligned: whole sectors per lane.
__device__ __forceinline__ void ld4(const long long* p, long long& a, long long& b, long long& c, long long& d) {
  asm volatile("ld.global.v4.u64 {%0,%1,%2,%3}, [%4];" : "=l"(a), "=l"(b), "=l"(c), "=l"(d) : "l"(p) : "memory");
}

template <int V>
struct Int {
  static constexpr int value = V;
};

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
__global__ void __launch_bounds__(WT, 1) k_oz(const PrepArgs P, int arg) {
  extern __shared__ __align__(1024) unsigned char oz_smem[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)oz_smem + 1023) & ~(uintptr_t)1023);
  unsigned char* pa = smem;
  constexpr int BN = MODE == OZ_TRSM ? NB : OT;        // columns of the MMAs
  constexpr uint32_t b_plane = BN * 128;
  unsigned char* pb = smem + SLICES * OPLANE;
  // per chunk, the sums of digit products of equal weight s = 0 .. 7 are handed
  // over as {0, 1, 2}, {3, 4}, {5, 6}, {7}; sum s sits in accumulator s & 3
  constexpr int GROUPS = 4;
  uint64_t* accF = (uint64_t*)(smem + 2 * SLICES * OPLANE);   // [GROUPS] a group is complete
  uint64_t* accE = accF + GROUPS;                              // group 0, then 1, has been read out
  uint64_t* done = accE + 1;
  uint32_t* tmem_slot = (uint32_t*)(done + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const PrepSide& S = P.side[blockIdx.z];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  constexpr int drains = BN / 32 * 4;                  // warps that read accumulators
  OzTile T;
  int i0;
  if (((MODE == OZ_TRSM || MODE == OZ_SYRK) && arg + NB >= S.dp) || !oz_tile<MODE>(S, arg, T, i0)) {
    pdl_wait();                                        // uniform over the CTA
    pdl_trigger();
    return;
  }
  if (t == 0) {
    for (int a = 0; a < GROUPS; ++a) mbar_init(&accF[a], 1);
    mbar_init(accE, drains);
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
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
  pdl_wait();
  pdl_trigger();
  const int64_t ld = S.dp;
  const int q = warp & 3, cg = warp >> 2;              // lane quarter, 32 columns
  const long long drain_limit = 4000000000LL;
  if constexpr (MODE == OZ_SYRK) {   // the tile's old values on their way to L2
    for (int e = t; e < T.na * 8; e += WT)
      if (16 * (e & 7) < T.nb)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(S.C + (int64_t)(T.ra + (e >> 3)) * ld + T.rb + 16 * (e & 7)));
  }
  auto timed_out = [&]() {
    raise_status(P.status, BAKRON_ERR_TIMEOUT);
    *abort_flag = 1;
  };
  // operand words of one unit (a row's eight terms): raw, then Q63
  auto load_a = [&](int u, int kk, long long (&w)[8]) {
    const int row = MODE == OZ_INV1 ? u & (OT - 1) : u >> 3, oct = MODE == OZ_INV1 ? u >> 7 : u & 7;
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = 0;
    if (row >= T.na) return;
    if constexpr (MODE == OZ_INV1) {                   // X11[k][j], k >= j
      const int j = T.ra + row;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int kr = kk + 8 * oct + k;
        if (kr >= j) w[k] = __double_as_longlong(S.X[(int64_t)(i0 + kr) * ld + i0 + j]);
      }
    } else {                                           // C's panel, or X22[i][k], k <= i
      const long long* p =
          MODE == OZ_INV2 ? (const long long*)S.X + (int64_t)(i0 + arg + T.ra + row) * ld + i0 + arg + kk + 8 * oct
                          : S.C + (int64_t)(T.ra + row) * ld + i0 + 8 * oct;
      ld4(p, w[0], w[1], w[2], w[3]);
      ld4(p + 4, w[4], w[5], w[6], w[7]);
      if constexpr (MODE == OZ_INV2) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (kk + 8 * oct + k > T.ra + row) w[k] = 0;
      }
    }
  };
  auto load_b = [&](int u, int kk, long long (&w)[8]) {
    const int row = u >> 3, oct = u & 7;
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = 0;
    if (row >= T.nb) return;
    const long long* p =
        MODE == OZ_TRSM   ? (const long long*)S.dinv + (int64_t)(i0 + row) * NB + 8 * oct
        : MODE == OZ_SYRK ? S.C + (int64_t)(T.rb + row) * ld + i0 + 8 * oct
        : MODE == OZ_INV1 ? S.C + (int64_t)(i0 + arg + T.rb + row) * ld + i0 + kk + 8 * oct
                          : S.C + (int64_t)(i0 + T.rb + row) * ld + i0 + arg + kk + 8 * oct;
    ld4(p, w[0], w[1], w[2], w[3]);
    ld4(p + 4, w[4], w[5], w[6], w[7]);
  };
  auto put_a = [&](int u, long long (&w)[8]) {
    const int row = MODE == OZ_INV1 ? u & (OT - 1) : u >> 3, oct = MODE == OZ_INV1 ? u >> 7 : u & 7;
    if constexpr (MODE == OZ_INV1 || MODE == OZ_INV2) {
      const int ex = row >= T.na ? 0 : 63 - (MODE == OZ_INV1 ? S.xc[i0 + T.ra + row] : S.xr[i0 + arg + T.ra + row]);
#pragma unroll
      for (int k = 0; k < 8; ++k) w[k] = to_fix(__longlong_as_double(w[k]), ex);
    }
    put_digits(pa, OPLANE, row, oct, w);
  };
  auto put_b = [&](int u, long long (&w)[8]) {
    const int row = u >> 3, oct = u & 7;
    if constexpr (MODE == OZ_TRSM || MODE == OZ_INV2) {
      const int ex = row >= T.nb ? 0 : 63 - (MODE == OZ_TRSM ? S.f[i0 + row] : S.tr[i0 + T.rb + row]);
#pragma unroll
      for (int k = 0; k < 8; ++k) w[k] = to_fix(__longlong_as_double(w[k]), ex);
    }
    put_digits(pb, b_plane, row, oct, w);
  };
  const uint64_t da = smem_desc(smem_u32(pa)), db = smem_desc(smem_u32(pb));
  // the products of sums s0 .. s1 (compile-time digit planes)
  auto issue = [&](auto s0, auto s1) {
#pragma unroll
    for (int s = decltype(s0)::value; s <= decltype(s1)::value; ++s) {
      const int first = max(0, s - SLICES + 1);
#pragma unroll
      for (int i = first; i <= min(s, SLICES - 1); ++i) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          mma_bf16(tmem + (uint32_t)((s & 3) * OT), da + (uint64_t)(i * (OPLANE >> 4) + 2 * k),
                   db + (uint64_t)((s - i) * (b_plane >> 4) + 2 * k), idesc_f16(OT, BN),
                   (i > first || k > 0) ? 1u : 0u);
      }
    }
  };
  long long acc[32];
  bool dead = false;
  constexpr bool one_chunk = MODE == OZ_TRSM || MODE == OZ_SYRK;
  // the largest leading part of a sum, where sums are looked at: all of a TRSM's, and of a
  // SYRK's the rows' norms, which bound the others
  float most = 0.f;
  const bool fit = MODE == OZ_TRSM || (MODE == OZ_SYRK && T.ra == T.rb && q == cg);
  static_assert(OT * 8 == 2 * WT, "two units of a per thread, two (or one) of b");
  for (int ch = 0; ch < (one_chunk ? 1 : T.kn); ++ch) {
    const int kk = NB * (T.k0 + ch);
    // -------------------------------------------------------- cut the operands
    // the next unit's words are on their way while one is cut
    {
      long long w0[8], w1[8];
      load_a(t, kk, w0);
      load_a(t + WT, kk, w1);
      put_a(t, w0);
      load_b(t, kk, w0);
      put_a(t + WT, w1);
      if constexpr (BN == OT) load_b(t + WT, kk, w1);
      put_b(t, w0);
      if constexpr (BN == OT) put_b(t + WT, w1);
    }
    if (one_chunk || ch == 0) {
#pragma unroll
      for (int u = 0; u < 32; ++u) acc[u] = 0;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    // ---------------------------------------- products, digit sums into 64 bits
    if (t == 0 && !dead) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      issue(Int<0>{}, Int<2>{});
      mma_commit(&accF[0]);
      issue(Int<3>{}, Int<3>{});
    }
    __syncwarp();
    if (warp < drains) {
      // sum s counts 2^(8 (6 - s)); modulo 2^64, so the first three only reach
      // the upper word, pairs of the others fit 32 bits, and the last is rounded
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) {
        int ok = dead ? 0 : 1;
        if (lane == 0 && !dead) {
          ok = oz_wait(&accF[g], (uint32_t)ch & 1u, P.spin_cycles, abort_flag) ? 1 : 0;
          if (!ok && !*abort_flag) timed_out();
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) {
          dead = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cg * 32);
        if (g == 0) {
#pragma unroll
          for (int c = 0; c < 32; c += 8) {
            uint32_t r0[8], r1[8], r2[8];
            tmem_ld8(ta + c, r0);
            tmem_ld8(ta + OT + c, r1);
            tmem_ld8(ta + 2 * OT + c, r2);
            tmem_wait_ld();
            if (fit)
#pragma unroll
              for (int u = 0; u < 8; ++u) most = fmaxf(most, leading(r0[u], r1[u]));
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const uint32_t v = (((biased_int(r0[u]) << 8) + biased_int(r1[u])) << 8) + biased_int(r2[u]);
              acc[c + u] += (long long)((unsigned long long)(
                                v - ((OZ_BIAS << 16) + (OZ_BIAS << 8) + OZ_BIAS)) << 32);
            }
          }
        } else if (g == 3) {
#pragma unroll
          for (int c = 0; c < 32; c += 16) {
            uint32_t r[16];
            tmem_ld16(ta + 3 * OT + c, r);
            tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 16; ++u)
              acc[c + u] += (int)(__float_as_uint(fmaf(__uint_as_float(r[u]), 1.f / 256.f, 12582912.f)) - OZ_BIAS);
          }
        } else {
#pragma unroll
          for (int c = 0; c < 32; c += 16) {
            uint32_t r0[16], r1[16];
            tmem_ld16(ta + (g == 1 ? 3 * OT : OT) + c, r0);
            tmem_ld16(ta + (g == 1 ? 0 : 2 * OT) + c, r1);
            tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const int lo = __float2int_rn(__uint_as_float(r1[u]));
              if (g == 1)
                acc[c + u] += (long long)((int)((biased_int(r0[u]) - OZ_BIAS) << 8) + lo) * 65536;
              else
                acc[c + u] += (long long)((int)(wide_int(r0[u]) << 8) + lo);
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        if (g < 2) {
          __syncwarp();
          if (lane == 0) mbar_arrive(accE);
          if (t == 0) {   // accumulators 0 .. 2 again, then 3
            if (oz_wait(accE, (uint32_t)g, P.spin_cycles, abort_flag)) {   // two phases a chunk
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              if (g == 0) {
                issue(Int<4>{}, Int<4>{});
                mma_commit(&accF[1]);
                issue(Int<5>{}, Int<6>{});
                mma_commit(&accF[2]);
              } else {
                issue(Int<7>{}, Int<7>{});
                mma_commit(&accF[3]);
              }
            } else if (!*abort_flag) {
              timed_out();
            }
          }
          __syncwarp();
        }
      }
    }
    __syncthreads();   // every MMA of the chunk is complete: its planes are free
  }
  if (t == 0) {
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
  if (!*abort_flag) {
    bool bad = most > OZ_FIT;
    // a warp's eight rows, four at a time (old values in flight together)
#pragma unroll
    for (int rr = 0; rr < OT / WORKERS; rr += 4) {
      longlong2 old[4][BN / 64];
      if constexpr (MODE == OZ_SYRK) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int cb = 0; cb < BN / 64; ++cb) {
            const int r = warp + WORKERS * (rr + j), c = 64 * cb + 2 * lane;
            if (r < T.na && c < T.nb)
              old[j][cb] = __ldcg(reinterpret_cast<longlong2*>(S.C + (int64_t)(T.ra + r) * ld + T.rb + c));
          }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int cb = 0; cb < BN / 64; ++cb) {
          const int r = warp + WORKERS * (rr + j), c = 64 * cb + 2 * lane;
          if (r >= T.na || c >= T.nb) continue;
          const longlong2 v = *reinterpret_cast<const longlong2*>(st + r * OUT_LD + c);
          if constexpr (MODE == OZ_TRSM) {
            const int f0 = min(max(S.f[i0 + c] + 1, 0), 63), f1 = min(max(S.f[i0 + c + 1] + 1, 0), 63);
            const longlong2 l = make_longlong2((long long)((unsigned long long)v.x << f0),
                                               (long long)((unsigned long long)v.y << f1));
            bad |= l.x >> f0 != v.x || l.y >> f1 != v.y;   // an entry of 1 or more
            *reinterpret_cast<longlong2*>(S.C + (int64_t)(T.ra + r) * ld + i0 + c) = l;
          } else if constexpr (MODE == OZ_SYRK) {
            // `left`: columns to the diagonal; above it C holds nothing yet
            auto less = [&](long long o, long long x, int left) -> long long {
              const long long y = (long long)(2 * (unsigned long long)x),
                              w = (long long)((unsigned long long)o - (unsigned long long)y);
              bad |= (left >= 0 && ((o ^ y) & (o ^ w)) < 0) || (left == 0 && w <= 0);
              return w;
            };
            const int left = T.ra + r - T.rb - c;
            *reinterpret_cast<longlong2*>(S.C + (int64_t)(T.ra + r) * ld + T.rb + c) =
                make_longlong2(less(old[j][cb].x, v.x, left), less(old[j][cb].y, v.y, left - 1));
          } else if constexpr (MODE == OZ_INV1) {
            const int er = S.xc[i0 + T.ra + r] - 62;
            *reinterpret_cast<double2*>((double*)S.C + (int64_t)(i0 + T.ra + r) * ld + i0 + arg + T.rb + c) =
                make_double2(from_fix(v.x, er), from_fix(v.y, er));
          } else {
            const int er = S.xr[i0 + arg + T.ra + r] - 62;
            const int e0 = S.tr[i0 + T.rb + c], e1 = S.tr[i0 + T.rb + c + 1];
            *reinterpret_cast<double2*>(S.X + (int64_t)(i0 + arg + T.ra + r) * ld + i0 + T.rb + c) =
                make_double2(from_fix(-v.x, er + e0), from_fix(-v.y, er + e1));
          }
        }
    }
    if (bad) raise_status(P.status, BAKRON_ERR_NOT_SPD);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
  if constexpr (MODE == OZ_SYRK) {
    if (blockIdx.x == 0)
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
  static OncePerDevice once;
  return once([] {
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
    return e;
  });
}

// One side from where its matrices are (PrepareScratch).
PrepSide make_side(const float* H, int d, int64_t dp, char* c, char* scratch, char* x) {
  PrepSide S;
  S.H = H;
  S.d = d;
  S.dp = (int)dp;
  S.C = (long long*)c;
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
// bytes of `scratch` per row of a side: 64 + 1 fp64, five ints (and the mean, and the
// shift to a 32-byte boundary)
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
  const PrepareScratch at(fl, pl, f, ws);
  P.side[0] = make_side(A, n, fl.np, at.CA, at.smallA, at.XA);
  P.side[1] = make_side(B, m, fl.mp, at.CB, at.smallB, at.XB);
  P.damp = damp;
  P.status = (int*)(ws + pl.off_status);
  P.spin_cycles = spin_cycles_from_env();
  const int dp = (int)(fl.np > fl.mp ? fl.np : fl.mp);   // both sides side by side (grid.z)
  auto up = [](int a, int b) { return (unsigned)((a + b - 1) / b); };
  k_prep_scale<<<2, 1024, 0, s>>>(P);
  k_prep_load<<<dim3(dp / 32, dp / 32, 2), 256, 0, s>>>(P);
  BK_CUDA_OK(cudaGetLastError());
  const dim3 oz(WT);
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
