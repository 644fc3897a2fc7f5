// Blocked Cholesky of the scaled covariance in 64-bit fixed point (the S/N solve of the
// paper's Sec. 5, Eqs. SNprim and eq:SN, and the factor of the PCA).
//
// The rows and columns are scaled, C' = S C S, with scales of 24 bits close to C_ii^-1/2 and
// the entries' products formed exactly: which scale is taken matters little, that it is the
// same for every entry does (with FP64 products all of the S/N's error, 1.4e-14 at M = 632,
// came from their roundings).  Every entry of the matrix, of each Schur complement and of the
// factor is then below 1 in magnitude, and so is the 2-norm of every factor row.  So the
// working matrix is held as integers in units of 2^-62: its resolution is 2^-62 of the
// diagonal, where an FP64 entry near 1 has 2^-53, and the elimination runs on the integer
// units.  A dependent FP64 operation takes 64
// cycles on this part and an SM completes two per clock; a 64 x 64 -> 64-bit product is
// a few 4-cycle multiply-adds.
//
//   * k_fx_panel: one 64-column panel.  Every CTA factorises the 64 x 64 diagonal block
//     for itself (the block is 16 KB in L2, and no second launch or grid barrier has to
//     hand it over), then solves its share of the rows below by forward substitution,
//     eight lanes per row.  Solved rows are cut into base-256 digits (rounded to 2^-55;
//     digits.cuh) for the updates, and stored as the FP64 factor.
//   * k_fx_upd: C -= L L^T over a K range of panels on the tensor cores: exact digit
//     sums, added in registers to the 64-bit entries themselves.  There is no
//     conversion: the sums come in the entries' own unit.
//   * The data row: y = L^-1 D' in FP64 (its scale is not bounded by 1).  One warp of the
//     panel kernel solves y for the panel in step with the diagonal block's columns;
//     the rows then subtract their products from D'.
// Panels are grouped into super-panels of four (256 columns; eight from FX_WIDE rows):
// inside one, a panel updates only the super-panel's remaining columns; the rest of the
// matrix is updated once per super-panel (a quarter, an eighth of the passes over it).
//
// What bounds it: up to M ~ 10000 the chain of panels (M = 6375: 100 panels of ~45 us
// and their ~12 us inner updates of the 7.7 ms), beyond that the passes over the entries
// and the exact sums' additions in the updates' epilogue (M = 24400: 156 ms).  Against
// FP64 diagonal blocks and panel solves: the joint S/N of M = 6375 14.4 -> 7.9 ms, of
// M = 818 1.28 -> 0.78 ms, the one in place at M = 24400 268 -> 158 ms.
//
// The integers are modulo 2^64, i.e. modulo 4.  In a positive definite matrix
// nothing leaves [-1, 1]; in another one a row wraps only after its factor entries' squares
// have added up to more than its diagonal entry, so the panel kernel keeps that sum of every
// row (FP32) and raises the pivot status beyond FX_NORM.
//
// Error: entries 2^-62, factor entries 2^-58 inside a panel, updates 2^-56 per
// digit row and 2^-53 per product, against the diagonal, i.e. below that of an FP64
// factorisation (2^-53 per operation).  S/N against 80-bit factorisations of 24 matrices of 144
// to 818 rows: the survey's 2e-16 .. 2.5e-15 (FP64 panels with slices of 2^-48: 9e-16 .. 1.7e-14),
// Wishart matrices with pivots down to 5e-4 2e-13 .. 2e-11 (3e-11 .. 2e-9).
#include <algorithm>

#include "digits.cuh"

#define FX_NB 64
#define FX_THREADS 256
// rows from which a super-panel has eight panels (M = 24400: 168 ms with four, 156 with
// eight; no difference at 6375, where the scratch is then smaller)
#define FX_WIDE 12288
#define FX_ONE (1ll << 62)
#define FX_NORM 1.0625f  // (below 1 but for the FP32 sums' rounding, ~2e-4 at 2800 panels)

// RN(c s t 2^62) for |c s t| < 1, s and t scales of 24 bits (variance_scale): the 101-bit
// product of the significands, of which 61 bits and more are kept before the rounding.
// Anything else, NaN included, cannot be an entry of a scaled positive definite matrix: status
__device__ __forceinline__ long long fx_fixed(double c, double s, double t, int* status) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(c);
  const unsigned sh_ = (unsigned)__double2hiint(s), th = (unsigned)__double2hiint(t);
  const int E = (int)((b >> 52) & 0x7FFu), Es = (int)(sh_ >> 20), Et = (int)(th >> 20);
  if (E == 0x7FF) {
    atomicExch(status, 1);
    return 0;
  }
  if (E == 0 || Es == 0 || Et == 0) return 0;  // (a scale of 0 has raised the status)
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const unsigned long long u = (unsigned long long)(((sh_ & 0xFFFFFu) | 0x100000u) << 3 | (unsigned)__double2loint(s) >> 29) *
                               (((th & 0xFFFFFu) | 0x100000u) << 3 | (unsigned)__double2loint(t) >> 29);
  const unsigned long long hi = __umul64hi(m << 11, u << 16);  // m u 2^-37: 61 to 64 bits
  const int sh = 3068 - E - Es - Et;
  unsigned long long q = 0;
  if (sh > 0 && sh < 64) q = (hi >> sh) + ((hi >> (sh - 1)) & 1ull);
  if (sh == 0) q = hi;
  if (sh < 0 || q >= (unsigned long long)FX_ONE) {
    atomicExch(status, 1);
    return 0;
  }
  return (b >> 63) ? -(long long)q : (long long)q;
}

// two neighbouring entries; `wide`: the pair is 16-byte aligned (COV_CHOL_TILE also takes
// packed tiles that are not)
__device__ __forceinline__ ulonglong2 fx_ld2(const double* p, int wide) {
  if (wide) return *(const ulonglong2*)p;
  const unsigned long long* q = (const unsigned long long*)p;
  return make_ulonglong2(q[0], q[1]);
}
__device__ __forceinline__ void fx_st2(double* p, unsigned long long a, unsigned long long b, int wide) {
  if (wide) {
    *(ulonglong2*)p = make_ulonglong2(a, b);
  } else {
    unsigned long long* q = (unsigned long long*)p;
    q[0] = a;
    q[1] = b;
  }
}

// ---------------------------------------------------------------- scaling
// The scales rs[i] of the selected entries (perm null: row i of W, FP64).  A variance that is
// no positive finite number is caught here.
__global__ void k_fx_rs(int64_t Ms, const int* __restrict__ perm, const double* __restrict__ C, int64_t ldc, OutMap W,
                        double* rs, float* nrm, int* status) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Ms) return;
  const double d = perm ? C[(int64_t)perm[i] * ldc + perm[i]] : *W.at(i, i);
  if (!(d > 0.0 && isfinite(d))) atomicExch(status, 1);
  rs[i] = variance_scale(d);
  nrm[i] = 0.0f;
}

// the selected rows, reordered and scaled, as integers; row Ms: D' (FP64)
__global__ void __launch_bounds__(256) k_fx_pack(int64_t Ms, const int* __restrict__ perm, const double* __restrict__ C,
                                                 int64_t ldc, const double* __restrict__ D,
                                                 const double* __restrict__ rs, double* Wk, int64_t ldw, int* status) {
  const int64_t i = blockIdx.x;
  const int64_t j0 = (int64_t)blockIdx.y * 1024 + threadIdx.x;
  if (i == Ms) {
    for (int64_t j = j0; j < Ms && j < j0 + 1024; j += 256) Wk[i * ldw + j] = D[perm[j]] * rs[j];
    return;
  }
  const int64_t pi = perm[i];
  const double ri = rs[i];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t j = j0 + 256 * u;
    if (j > i) break;
    const int64_t pj = perm[j];
    const int64_t hi = pi > pj ? pi : pj, lo = pi > pj ? pj : pi;
    ((long long*)Wk)[i * ldw + j] = fx_fixed(C[hi * ldc + lo], ri, rs[j], status);
  }
}

// in place on lower-packed tiles (rows in cumulative order): one block per 32 x 32
// lower block of the leading M x M part, plus the D row
__global__ void __launch_bounds__(256) k_fx_pack_tiles(int64_t M, OutMap W, const double* __restrict__ rs,
                                                       const double* __restrict__ D, int* status) {
  const int64_t id = blockIdx.x;
  int64_t bi = (int64_t)((sqrtf(8.0f * (float)id + 1.0f) - 1.0f) * 0.5f);
  if (bi < 0) bi = 0;
  while (bi * (bi + 1) / 2 > id) --bi;
  while ((bi + 1) * (bi + 2) / 2 <= id) ++bi;
  const int64_t c = (id - bi * (bi + 1) / 2) * 32 + (threadIdx.x & 31);
  if (c >= M) return;
  const double rc = rs[c];
  for (int rr = threadIdx.x >> 5; rr < 32; rr += 8) {
    const int64_t r = bi * 32 + rr;
    if (c > r || r > M) continue;
    double* p = W.at(r, c);
    if (r == M)
      *p = D[c] * rc;
    else
      *(long long*)p = fx_fixed(*p, rc, rs[r], status);
  }
}

// ---------------------------------------------------------------- arithmetic
// Full products: a (units of 2^-62, |a| < 2^62) as two 31-bit halves, a = h 2^31 + l,
// 0 <= l < 2^31; a b 2^-62 = h h' + (h l' + l h') 2^-31 + l l' 2^-62, the last term
// (below one unit) dropped and the middle one rounded down: three 32 x 32 -> 64-bit
// multiply-adds.
__device__ __forceinline__ int2 fx_split(long long a) { return make_int2((int)(a >> 31), (int)(a & 0x7FFFFFFF)); }
__device__ __forceinline__ long long fx_mul(int2 a, int2 b) {
  const long long t = (long long)a.x * b.y + (long long)a.y * b.x;
  return (long long)a.x * b.x + (t >> 31);
}

// Factor entries are rounded to 2^-57 and held as h 2^-31 + l 2^-57, 0 <= l < 2^26, so
// that the middle terms of up to 16 products add up in one 64-bit word: three
// multiply-adds per product and one shift per eight.  (The trailing update takes them to
// 2^-55.)  An entry of 1, possible only in a singular matrix, wraps to -1: same square.
__device__ __forceinline__ int2 fx_entry(long long v) {
  const long long w = (v + 16) >> 5;
  return make_int2((int)(w >> 26), (int)(w & 0x3FFFFFF));
}
__device__ __forceinline__ long long fx_join(int2 a) { return ((long long)a.x << 26) + a.y; }  // units of 2^-57
__device__ __forceinline__ int2 fx_neg(int2 a) { return make_int2(-a.x, -a.y); }
struct FxAcc {
  long long h, m;  // units of 2^-62 and 2^-88
  __device__ __forceinline__ void add(int2 a, int2 b) {
    h += (long long)a.x * b.x;
    m += (long long)a.x * b.y;
    m += (long long)a.y * b.x;
  }
  __device__ __forceinline__ long long value() const { return h + (m >> 26); }
};

__device__ __forceinline__ long long fx_sub(long long v, int2 a, int2 b) {  // v - a b
  FxAcc t{v, 0};
  t.add(fx_neg(a), b);
  return t.value();
}

// v 2^-57 as FP64 (rounded to nearest), by integer operations: |v| <= 2^57
__device__ __forceinline__ double fx_double(long long v) {
  const unsigned long long u = v < 0 ? (unsigned long long)-v : (unsigned long long)v;
  const int lz = __clzll((long long)u);
  const unsigned long long m = (u << lz) + 1024;                // 53 bits, rounded half up
  const unsigned long long carry = m < 1024 ? 1ull : 0ull;      // up to the next power of two
  const unsigned long long e = (unsigned long long)(63 - lz - 57 + 1023 - 1);
  const unsigned long long q = carry ? (1ull << 53) : m >> 11;  // 2^52 .. 2^53: adds into the exponent
  const long long bits = (long long)((e << 52) + q) | (v < 0 ? (long long)(1ull << 63) : 0ll);
  return u == 0 ? 0.0 : __longlong_as_double(bits);
}

// 1 / sqrt(d 2^-62) = 2 r 2^(s - 62), r in (2^61, 2^62), for 0 < d < 2^62: a 22-bit
// seed from the FP32 unit and one third-order correction in integers (relative error
// below 2^-54).  The normalising shift comes from the converted value's exponent beside
// the seed's own latency, so the chain is one conversion, one reciprocal square root
// and ~20 dependent integer operations (the FP64 reciprocal square root: ~430 cycles).
__device__ __forceinline__ void fx_rsqrt(long long d, long long* r, int* s) {
  unsigned long long u = (unsigned long long)d;
  int up = 0;
  if (u < (1ull << 54)) {  // too few bits in the upper word for the seed
    up = (__clzll((long long)u) - 2) >> 1;
    u <<= 2 * up;
  }
  const float uf = __uint2float_rz((unsigned)(u >> 32));  // (rounded down: the exponent is that of u)
  float y0;                                                // 2^15 y0 = 1 / sqrt(u 2^-62)
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(uf));
  const int sh = (156 - (int)(__float_as_uint(uf) >> 23)) >> 1;  // u 4^sh in [2^60, 2^62)
  const unsigned long long x = u << (2 * sh);                    // Q62
  // 2^(15 - sh) y0 in [1, 2] as a 30-bit fraction
  const unsigned b = __float_as_uint(y0);
  const unsigned Y = ((b & 0x7FFFFFu) | 0x800000u) << ((int)(b >> 23) - 105 - sh);
  // e = 1 - x Y^2 (Q61)
  const unsigned long long z = (((x & 0xFFFFFFFFull) * Y) >> 32) + (x >> 32) * Y;           // x Y, Q60
  const unsigned long long t = (((z & 0xFFFFFFFFull) * Y) >> 29) + (((z >> 32) * Y) << 3);  // x Y^2, Q61
  const long long e = (long long)((1ull << 61) - t);
  const long long es = (long long)(int)(e >> 16);
  const long long f = (e >> 1) + ((3 * es * es) >> 32);  // e / 2 + 3 e^2 / 8, Q61
  // Y (1 + f), half of it in Q62; 64 units less, so that 2^62 is not reached
  const long long c = (f >> 32) * (long long)Y + (long long)(((f & 0xFFFFFFFFll) * (unsigned long long)Y) >> 32);  // Q59
  *r = (long long)(((unsigned long long)Y << 31) - 64) + (c << 2);
  *s = sh + up;
}

// a times 2 r 2^(s - 62), the reciprocal square root of a pivot d: |a| <= sqrt(d) in a
// positive definite matrix; bits of bad are raised where a or the result leaves the range.
__device__ __forceinline__ long long fx_scale(long long a, int2 r, int s, long long& bad) {
  const long long l = fx_mul(fx_split(a << s), r);  // half the result
  bad |= ((a >> (62 - s)) ^ (a >> 63)) | ((l >> 61) ^ (l >> 63));
  return l << 1;
}

__device__ __forceinline__ long long fx_bcast(long long v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
__device__ __forceinline__ int2 fx_bcast(int2 v, int lane) {
  return make_int2(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane));
}

// ---------------------------------------------------------------- panel
struct FxPanel {
  OutMap W;
  int64_t k0, Ms, rb0;   // first column; rows; first 128-row block of the digit buffer
  int kb, kblk, nkb;     // columns; first K block of the panel in the buffer; its K blocks per row block
  uint8_t* dig;
  double *y, *ld, *ld_prev;  // solved data vector; this and the previous panel's diagonal factor (64 x 64)
  float* nrm;                // squared norm of every row's factor entries so far
  int* status;
  int wide;  // the matrix is 16-byte aligned
};

// 1 / L_jj from the pivot's r (as two halves) and shift
__device__ __forceinline__ double fx_rpivot(int2 r, int s) {
  return (double)(((long long)r.x << 31) + r.y) * __hiloint2double((1023 - 61 + s) << 20, 0);
}

// the previous panel's diagonal factor into the matrix (its columns have no reader left)
__device__ __forceinline__ void fx_store_diag(const OutMap& W, int64_t k0, int kb, const double* ld) {
  for (int e = threadIdx.x; e < FX_NB * FX_NB; e += blockDim.x) {
    const int i = e >> 6, l = e & 63;
    if (i < kb && l <= i) *W.at(k0 + i, k0 + l) = ld[e];
  }
}

#define FX_LD (FX_NB + 1)
#define FX_RB 32                              // rows below the diagonal block per CTA
#define FX_ROWS (FX_NB + FX_RB)
#define FX_PSMEM (8 * FX_ROWS * FX_LD)        // 49 KB
#define FX_Q57 (1.0 / 144115188075855872.0)

// A CTA holds the diagonal block and 32 rows below it (the last CTA none: it stores the
// diagonal factor and y) and takes eight columns at a time, one block barrier each:
//  * warps 0-3 subtract the products of the eight columns before and factorise the eight
//    columns of every remaining row, one row per lane in registers, each warp with its
//    own copy of the 8 x 8 block in lanes 0-7: no barrier inside.  A warp may come to its
//    copy after warp 0 has finished the block (other kernels' CTAs on the SM), so the
//    factored entries inside an 8 x 8 block go to their mirror places above the diagonal,
//    which nobody reads in these eight columns.  The pivot's chain (the reciprocal square
//    root, one scaled entry, one shuffle, one product) is what bounds the panel;
//  * meanwhile warps 4-6 subtract the products of all earlier columns from the next eight,
//    and warp 7 advances y by the eight columns before.
// One panel of M = 6375 (cold): 51 us for the FP64 diagonal block and 37 us for the FP64
// panel solve before.
__global__ void __maxnreg__(104) k_fx_panel(FxPanel P) {
  extern __shared__ long long fx_smem[];
  // entries in units of 2^-62; factored entries as their two halves in place.  Rows 0-63:
  // the diagonal block; 64-95: this CTA's rows
  long long(*L)[FX_LD] = (long long(*)[FX_LD])fx_smem;
  __shared__ int2 rinv[FX_NB];
  __shared__ int rsh[FX_NB];
  __shared__ double ysh[FX_NB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const OutMap W = P.W;
  const int64_t k0 = P.k0;
  const int kb = P.kb;
  const bool storer = blockIdx.x + 1 == gridDim.x;
  const int64_t r0 = k0 + FX_NB + (int64_t)blockIdx.x * FX_RB;  // this CTA's rows (kb = 64 where there are any)
  const int nr = storer ? 0 : (int)(P.Ms - r0 < FX_RB ? P.Ms - r0 : FX_RB);
  {
    // all loads in flight before the first use
    const int c = tid & 63, i0 = tid >> 6;
    long long v[FX_ROWS / 4];
#pragma unroll
    for (int u = 0; u < FX_ROWS / 4; ++u) {
      const int i = i0 + 4 * u;
      if (i < FX_NB)
        v[u] = (i < kb && c <= i) ? *(const long long*)W.at(k0 + i, k0 + c) : (i == c ? FX_ONE - 1 : 0);
      else
        v[u] = i - FX_NB < nr ? *(const long long*)W.at(r0 + (i - FX_NB), k0 + c) : 0;
    }
#pragma unroll
    for (int u = 0; u < FX_ROWS / 4; ++u) L[i0 + 4 * u][c] = v[u];
  }
  double dv0 = 0.0, dv1 = 0.0;  // warp 7: D' of panel rows lane and lane + 32
  if (warp == 7) {
    if (lane < kb) dv0 = *W.at(P.Ms, k0 + lane);
    if (lane + 32 < kb) dv1 = *W.at(P.Ms, k0 + 32 + lane);
  }
  long long bad = 0;
  // factored entry (i, l), l < i < 64: mirrored inside its 8 x 8 block
  auto entry = [&](int i, int l) -> int2 { return *(const int2*)((i ^ l) < 8 ? &L[l][i] : &L[i][l]); };
  auto solve_y = [&](int c0) {  // warp 7: y of columns c0 .. c0 + 7, D' of the diagonal block's rows below
    double rd = 0.0;            // lane j < 8: 1 / L_jj
    if (lane < 8) rd = fx_rpivot(rinv[c0 + lane], rsh[c0 + lane]);
    // row lane (c0 < 32) or lane + 32: the columns c0 .. of the row, or of the block's mirror
    const bool m0 = (lane ^ c0) < 8, m1 = ((lane + 32) ^ c0) < 8;
    const long long *p0 = m0 ? &L[c0][lane] : &L[lane][c0], *p1 = m1 ? &L[c0][lane + 32] : &L[lane + 32][c0];
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
      const int c = c0 + j;
      const double yj = __shfl_sync(0xffffffffu, c < 32 ? dv0 : dv1, c & 31) * __shfl_sync(0xffffffffu, rd, j);
      if (lane == 0) ysh[c] = yj;
      const double ys = -yj * FX_Q57;
      if (c < 31 && lane > c) dv0 = fma((double)fx_join(*(const int2*)p0), ys, dv0);
      if (lane + 32 > c) dv1 = fma((double)fx_join(*(const int2*)p1), ys, dv1);
      p0 += m0 ? FX_LD : 1;
      p1 += m1 ? FX_LD : 1;
    }
  };
  __syncthreads();
#pragma unroll 1
  for (int c0 = 0; c0 < FX_NB; c0 += 8) {
    if (warp < 4) {
      // ---- columns c0 .. c0 + 7 of the remaining rows
      const int row = lane < 8 ? c0 + lane : c0 + 8 + warp * 24 + (lane - 8);
      const bool live = row < FX_ROWS;
      if (warp == 0 || c0 + 8 + warp * 24 < FX_ROWS) {
        const int ro = live ? row : c0, last = lane < 8 ? lane : (live ? 7 : 0);
        long long a[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) a[k] = k <= last ? L[ro][c0 + k] : 0;
        if (c0 > 0) {  // minus the products of the eight columns before (the earlier ones: warps 4-6)
          FxAcc v[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] = FxAcc{a[k], 0};
#pragma unroll 2
          for (int p = 0; p < 8; ++p) {
            const int2 x = fx_neg(*(const int2*)&L[ro][c0 - 8 + p]);
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k].add(x, *(const int2*)&L[c0 + k][c0 - 8 + p]);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) a[k] = v[k].value();
        }
        // where this lane's factored entries go, and the step from one column to the next
        int2* out = lane < 8 ? (int2*)&L[c0][row] : (int2*)&L[ro][c0];
        const int step = lane < 8 ? FX_LD : 1;
        const int upto = lane < 8 ? (warp == 0 ? lane : 0) : (live ? 8 : 0);  // columns below this one
        long long d = fx_bcast(a[0], 0);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (d <= 0) {
            bad = -1;
            d = FX_ONE - 1;
          }
          long long dn = 0;  // the next pivot before this column's product
          if (j < 7) dn = fx_bcast(a[j < 7 ? j + 1 : 7], j + 1);
          long long r;
          int s;
          fx_rsqrt(d, &r, &s);
          const int2 r2 = fx_split(r);
          long long b = 0;
          const int2 l = fx_entry(fx_scale(a[j], r2, s, b));
          if (live && lane > j) bad |= b;
          if (tid == 0) {
            rinv[c0 + j] = r2;
            rsh[c0 + j] = s;
          }
#pragma unroll
          for (int k = j + 1; k < 8; ++k) {
            const int2 y = fx_bcast(l, k);
            if (k == j + 1) d = fx_sub(dn, y, y);
            a[k] = fx_sub(a[k], l, y);
          }
          if (j < upto) out[j * step] = l;
        }
      }
    } else if (warp < 7) {
      // ---- columns c0 + 8 .. c0 + 15 minus the products of columns 0 .. c0 - 1: a lane takes
      // four columns of a row, both halves in turn while there are more than 48 rows
      const int t = tid - 128, n = FX_ROWS - 8 - c0;
      const bool two = n > 48;
      const int i = c0 + 8 + (two ? t : t % 48);
      if (c0 > 0 && c0 + 8 < FX_NB && i < FX_ROWS) {
#pragma unroll 1
        for (int h = two ? 0 : t / 48; h < (two ? 2 : t / 48 + 1); ++h) {
          const int l0 = c0 + 8 + 4 * h;
          long long a[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) a[k] = L[i][l0 + k];
#pragma unroll 1
          for (int p0 = 0; p0 < c0; p0 += 8) {
            FxAcc v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = FxAcc{a[k], 0};
#pragma unroll
            for (int p = p0; p < p0 + 8; ++p) {
              const int2 x = fx_neg(*(const int2*)&L[i][p]);
#pragma unroll
              for (int k = 0; k < 4; ++k) v[k].add(x, *(const int2*)&L[l0 + k][p]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) a[k] = v[k].value();
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) L[i][l0 + k] = a[k];  // (above the diagonal: never read)
        }
      }
    } else if (c0 > 0) {
      solve_y(c0 - 8);
    }
    __syncthreads();
  }
  if (warp == 7) solve_y(FX_NB - 8);
  __syncthreads();
  if (bad) atomicExch(P.status, 1);
  if (storer) {
    for (int e = tid; e < FX_NB * FX_NB; e += FX_THREADS) {
      const int i = e >> 6, l = e & 63;
      if (i < kb && l <= i)
        P.ld[e] = i == l ? 1.0 / fx_rpivot(rinv[i], rsh[i]) : (double)fx_join(entry(i, l)) * FX_Q57;
    }
    if (tid < kb) P.y[k0 + tid] = ysh[tid];
    {
      // the diagonal block's rows (the others: below), four threads each, without the pivot
      const int i = tid >> 2;
      float n2 = 0.0f;
      for (int l = tid & 3; l < i; l += 4) {
        const float f = __int2float_rn(entry(i, l).x);
        n2 = fmaf(f, f, n2);
      }
      n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
      n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
      if (i < kb && !(P.nrm[k0 + i] + n2 * 0x1p-62f <= FX_NORM)) atomicExch(P.status, 1);
    }
    if (k0 > 0) fx_store_diag(W, k0 - FX_NB, FX_NB, P.ld_prev);
    return;
  }
  // this CTA's rows: thread (row, k8) holds eight consecutive entries
  const int rl = tid >> 3, q = tid & 7;
  const int64_t row = r0 + rl;
  long long X[8];
  double xd[8], dot = 0.0;
  float n2 = 0.0f;
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int2 l = *(const int2*)&L[FX_NB + rl][8 * q + p];
    const long long v = fx_join(l);
    const float f = __int2float_rn(l.x);  // (units of 2^-31)
    n2 = fmaf(f, f, n2);
    X[p] = (v + 2) >> 2;  // to units of 2^-55
    xd[p] = fx_double(v);
    dot = fma(xd[p], ysh[8 * q + p], dot);
  }
  uint4 d[SL_S];
  sl_digits8(X, d);
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    dot += __shfl_xor_sync(0xffffffffu, dot, o);
    n2 += __shfl_xor_sync(0xffffffffu, n2, o);
  }
  if (rl < nr) {
    uint8_t* o = P.dig + ((size_t)((row >> 7) - P.rb0) * P.nkb + P.kblk + (q >> 2)) * SL_BLOCK +
                 (size_t)(row & 127) * (SL_BK * 2) + (q & 3) * 16;
#pragma unroll
    for (int t = 0; t < SL_S; ++t) *(uint4*)(o + (size_t)t * SL_DIGIT) = d[t];
    double* rowp = W.at(row, k0) + 8 * q;  // 64 consecutive entries (k0 is a multiple of 64)
#pragma unroll
    for (int p = 0; p < 8; p += 2)
      fx_st2(rowp + p, (unsigned long long)__double_as_longlong(xd[p]),
             (unsigned long long)__double_as_longlong(xd[p + 1]), P.wide);
    if (q == 0) {
      *W.at(P.Ms, row) -= dot;
      const float t = P.nrm[row] + n2 * 0x1p-62f;
      P.nrm[row] = t;
      if (!(t <= FX_NORM)) atomicExch(P.status, 1);
    }
  }
}

// the last panel's diagonal factor, and y as the data row
__global__ void k_fx_tail(OutMap W, int64_t Ms, int64_t k0, int kb, const double* ld, const double* y) {
  if (blockIdx.x == 0) fx_store_diag(W, k0, kb, ld);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < Ms; i += (int64_t)gridDim.x * blockDim.x)
    *W.at(Ms, i) = y[i];
}

// ---------------------------------------------------------------- trailing update
// Tiles of one launch: column tiles [j0, j0 + nj) of 64 columns, each with the 128-row
// blocks that reach its lower part, row block by row block.
struct FxTiles {
  int64_t j0, nj, i0, ni;
  __host__ __device__ int64_t cnt(int64_t i) const {
    const int64_t c = 2 * (i + 1) - j0;
    return c < nj ? c : nj;
  }
  __host__ __device__ int64_t cum(int64_t i) const {  // tiles of row blocks i0 .. i - 1
    int64_t st = (nj + j0 + 1) / 2 - 1;               // first row block with all nj tiles
    if (st < i0) st = i0;
    const int64_t b = i < st ? i : st, a = i0;
    const int64_t tri = b > a ? (b * (b + 1) - a * (a + 1)) - j0 * (b - a) : 0;
    return tri + (i > st ? (i - st) * nj : 0);
  }
  __device__ void at(int64_t id, int64_t* ib, int64_t* jt) const {
    int64_t lo = i0, hi = i0 + ni;  // cum(lo) <= id < cum(hi)
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (cum(mid) <= id)
        lo = mid;
      else
        hi = mid;
    }
    *ib = lo;
    *jt = j0 + (id - cum(lo));
  }
};

struct FxUpd {
  OutMap W;
  int64_t Ms, rb0;
  int kblk, nk, nkb;  // K blocks kblk .. kblk + nk - 1 of the buffer's nkb
  FxTiles t;
  int64_t ntiles;
  int* status;
  int wide;  // the matrix is 16-byte aligned
};

// A CTA takes every gridDim-th tile of 128 x 64.  The accumulators start as the tile's
// own entries and are stored at its end; meanwhile the loads and MMAs of the next tile's
// first K blocks proceed (a CTA per tile paid ~14 us of set-up, first loads, entry reads
// and writes beside ~11 us of products at K = 256).  Elements above the diagonal are left
// alone (a pair of entries is moved at a time: the entry right of the diagonal may be
// rewritten, no kernel reads it).
#define FX_NG 2
// (120 registers: with the panel kernel's 104 both fit an SM's register file, see fx_update)
__global__ void __maxnreg__(120)
    k_fx_upd(const __grid_constant__ CUtensorMap map_i, const __grid_constant__ CUtensorMap map_j, FxUpd A) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) SlBars bars;
  __shared__ uint32_t tmem_sh;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) sl_bars_init(&bars);
  if (warp == 0) sl_tmem_alloc(&tmem_sh);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_sh;
  int it = 0;
  if (warp == 0 && lane == 0) {
    for (int64_t id = blockIdx.x; id < A.ntiles; id += gridDim.x) {
      int64_t ib, jt;
      A.t.at(id, &ib, &jt);
      if (!sl_produce<FX_NG>(&map_i, &map_j, smem, &bars, (int)((ib - A.rb0) * A.nkb) + A.kblk,
                             (int)(((jt >> 1) - A.rb0) * A.nkb) + A.kblk, (int)(jt & 1) * 64, A.nk, it, A.status))
        break;
    }
  } else if (warp == 1) {
    for (int64_t id = blockIdx.x; id < A.ntiles; id += gridDim.x)
      if (!sl_issue<FX_NG, true>(smem, &bars, A.nk, it, A.status)) break;
    sl_issue_end(&bars, lane);
  } else if (warp >= 2) {
    const int q = warp & 3, half = (warp - 2) >> 2;
    const unsigned long long off = SL_BIAS * (unsigned long long)A.nk;
    sl_drain_init<true>(&bars, tmem, q, half, lane);
    for (int64_t id = blockIdx.x; id < A.ntiles; id += gridDim.x) {
      int64_t ib, jt;
      A.t.at(id, &ib, &jt);
      const int64_t col0 = jt * 64;
      // this thread's rows: c of acc[j][c] in pairs {0, 1, 4, 5}, {2, 3, 6, 7} and these + 8
      double* p[4];
      int nc[4];  // last live column of the tile in the row, less this thread's first
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t gr = ib * SL_BM + sl_row<true>(q, lane, 2 * (u & 1) + 8 * (u >> 1));
        const bool in = gr < A.Ms && gr >= col0;
        p[u] = in ? A.W.at(gr, col0) + sl_col<true>(half, lane, 0, 0) : nullptr;
        nc[u] = in ? (int)(gr - col0 < 64 ? gr - col0 : 64) - sl_col<true>(half, lane, 0, 0) : -1;
      }
      unsigned long long acc[FX_NG][16];
#pragma unroll
      for (int j = 0; j < FX_NG; ++j)
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const int u = ((c >> 1) & 1) + 2 * (c >> 3), o = j * SL_BN + 8 * ((c >> 2) & 1);
          ulonglong2 v = make_ulonglong2(0ull, 0ull);
          if (o <= nc[u]) v = fx_ld2(p[u] + o, A.wide);
          acc[j][c] = v.x - off;
          acc[j][c + 1] = v.y - off;
        }
      if (!sl_drain<FX_NG, true>(acc, &bars, tmem, q, half, lane, A.nk, it, A.status)) break;
#pragma unroll
      for (int j = 0; j < FX_NG; ++j)
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const int u = ((c >> 1) & 1) + 2 * (c >> 3), o = j * SL_BN + 8 * ((c >> 2) & 1);
          if (o <= nc[u]) fx_st2(p[u] + o, acc[j][c], acc[j][c + 1], A.wide);
        }
    }
  }
  __syncwarp();
  if (warp == 0 && lane == 0) sl_pause(A.status);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) sl_tmem_free(tmem);
}

// ---------------------------------------------------------------- host side
int wl_num_sms() {
  static std::once_flag once[WL_MAX_DEVICES];
  static int n[WL_MAX_DEVICES];
  int d = 0;
  cudaGetDevice(&d);
  if (d < 0 || d >= WL_MAX_DEVICES) return 1;
  std::call_once(once[d], [&] {
    n[d] = 1;
    cudaDeviceGetAttribute(&n[d], cudaDevAttrMultiProcessorCount, d);
    if (n[d] < 1) n[d] = 1;
  });
  return n[d];
}

// scratch of a factorisation of n rows with super-panels of w panels: two digit
// buffers, the diagonal factors of two panels, the solved data vector, the scaling, the rows'
// norms
size_t wl_fx_bytes(int64_t n, int w) {
  const size_t dig = (size_t)((n + SL_BM - 1) / SL_BM) * (size_t)(2 * w) * SL_BLOCK;
  return 2 * dig + 2 * FX_NB * FX_NB * 8 + 16 * (size_t)((n + 1) / 2 * 2) + 4 * (size_t)((n + 1) / 2 * 2);
}

// The scratch, grown on demand: super-panels of four panels (eight for matrices whose
// trailing update bounds the factorisation: half the passes over the entries), fewer
// where the memory (or the server's reservation) does not hold them.  A captured step
// keeps to what the eager one before it allocated.
static int fx_scratch(cov_handle* h, int64_t n, int* w_out, cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (h->deferred) WL_CHECK(h, cudaStreamIsCapturing(s, &cap));
  for (int w = n >= FX_WIDE ? 8 : 4; w >= 1; w >>= 1) {
    const size_t need = wl_fx_bytes(n, w);
    if (w > 1 && h->chol_scratch_cap && need > h->chol_scratch_cap) continue;
    if (need <= h->chol_scratch_n) {
      *w_out = w;
      return COV_OK;
    }
    if (cap != cudaStreamCaptureStatusNone) continue;
    if (w > 1) {
      size_t fr = 0, tot = 0;
      const bool known = cudaMemGetInfo(&fr, &tot) == cudaSuccess;
      if (!known || need > fr / 16 ||
          (h->budget && h->allocated - h->chol_scratch_n + need + ((size_t)64 << 20) > h->budget))
        continue;
    }
    if (h->chol_scratch) {  // given back first: never the old and the new buffer at the same time
      cudaFree(h->chol_scratch);
      h->allocated -= h->chol_scratch_n;
      h->chol_scratch = nullptr;
      h->chol_scratch_n = 0;
    }
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, need);
    if (e != cudaSuccess) {
      cudaGetLastError();
      if (w > 1) continue;
      return wl_cuda(h, e, "cudaMalloc (Cholesky scratch)");
    }
    h->chol_scratch = p;
    h->chol_scratch_n = need;
    h->allocated += need;
    *w_out = w;
    return COV_OK;
  }
  return wl_fail(h, COV_ERR_INVALID, "Cholesky scratch not allocated before stream capture");
}

// Whether `extra` bytes more are beyond the handle's budget.  The Cholesky's scratch is
// given back first where it stands in the way: it is wider than it has to be, and the
// next factorisation takes what then fits.
bool wl_over_budget(cov_handle* h, size_t extra) {
  if (!h->budget || h->allocated + extra <= h->budget) return false;
  if (h->chol_scratch && !h->deferred) {
    cudaFree(h->chol_scratch);
    h->allocated -= h->chol_scratch_n;
    h->chol_scratch = nullptr;
    h->chol_scratch_n = 0;
  }
  return h->allocated + extra > h->budget;
}

static uint8_t* fx_dig(cov_handle* h, int64_t n, int w, int b) {
  const size_t dig = (size_t)((n + SL_BM - 1) / SL_BM) * (size_t)(2 * w) * SL_BLOCK;
  return (uint8_t*)h->chol_scratch + (size_t)b * dig;
}
static double* fx_tail_mem(cov_handle* h, int64_t n, int w) { return (double*)fx_dig(h, n, w, 2); }

struct FxMaps {
  CUtensorMap i, j;
};

static int fx_attributes(cov_handle* h) {
  static std::once_flag attr_once[WL_MAX_DEVICES];
  static int attr_rc[WL_MAX_DEVICES];
  if (wl_once_per_device(attr_once, attr_rc, [] {
        int e = (int)cudaFuncSetAttribute(k_fx_upd, cudaFuncAttributeMaxDynamicSharedMemorySize, SlShape<FX_NG>::kSmem);
        if (!e) e = (int)cudaFuncSetAttribute(k_fx_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, FX_PSMEM);
        return e;
      }) != 0)
    return wl_fail(h, COV_ERR_CUDA, "cudaFuncSetAttribute (Cholesky kernels) failed");
  return COV_OK;
}

static int fx_wide(const OutMap& W) { return ((uintptr_t)W.C & 15) == 0 && (W.tiled || W.ldc % 2 == 0); }

// columns [c0, c1) of the trailing matrix of rows c0 .. Ms - 1, on at most `sms` SMs
static int fx_update(cov_handle* h, OutMap W, int64_t Ms, int64_t rb0, int kblk, int nk, int nkb, int64_t c0, int64_t c1,
                     const FxMaps& m, int64_t sms, cudaStream_t s) {
  if (c0 >= c1 || c0 >= Ms) return COV_OK;
  FxUpd a{W, Ms, rb0, kblk, nk, nkb, {}, 0, h->chol_status, fx_wide(W)};
  a.t.j0 = c0 / 64;
  a.t.nj = (c1 + 63) / 64 - a.t.j0;
  a.t.i0 = c0 / SL_BM;
  a.t.ni = (Ms + SL_BM - 1) / SL_BM - a.t.i0;
  a.ntiles = a.t.cum(a.t.i0 + a.t.ni);
  if (a.ntiles <= 0) return COV_OK;
  const int64_t grid = h->chol_kernel == 1 ? a.ntiles : std::min(a.ntiles, sms);
  k_fx_upd<<<(unsigned)grid, SL_THREADS, SlShape<FX_NG>::kSmem, s>>>(m.i, m.j, a);
  WL_LAUNCH(h, "k_fx_upd");
  return COV_OK;
}

// The scaling factors and integers of the selected entries (perm: dense source C into
// the workspace; null: W's own FP64 tiles in place), then the factorisation of rows
// 0 .. Ms - 1 with the data row Ms, which ends as y = L^-1 D'; the factor is left in
// FP64.  Everything stays on the device; the status words are the caller's.
int wl_fx_factor(cov_handle* h, OutMap W, int64_t Ms, const int* perm, const double* C, int64_t ldc, const double* D,
                 cudaStream_t s) {
  int rc, w = 4;
  if (h->chol_kernel != 1 && !fx_wide(W))
    return wl_fail(h, COV_ERR_CUDA, "Cholesky: the matrix is not 16-byte aligned");
  if ((rc = fx_attributes(h))) return rc;
  if ((rc = fx_scratch(h, Ms, &w, s))) return rc;
  if ((rc = wl_side_stream(h))) return rc;
  const int64_t nb = (Ms + SL_BM - 1) / SL_BM;
  const int nkb = 2 * w;
  double* ld = fx_tail_mem(h, Ms, w);
  double* y = ld + 2 * FX_NB * FX_NB;
  double* rs = y + (Ms + 1) / 2 * 2;
  float* nrm = (float*)(rs + (Ms + 1) / 2 * 2);
  int* st = h->piv_status;
  int tk = wl_stage_begin(h, ST_SNR_PACK, s);
  k_fx_rs<<<(unsigned)((Ms + 255) / 256), 256, 0, s>>>(Ms, perm, C, ldc, W, rs, nrm, st);
  if (perm) {
    k_fx_pack<<<dim3((unsigned)(Ms + 1), (unsigned)((Ms + 1023) / 1024)), 256, 0, s>>>(Ms, perm, C, ldc, D, rs, W.C, W.ldc,
                                                                                     st);
  } else {
    const int64_t b = (Ms + 1 + 31) / 32;
    k_fx_pack_tiles<<<(unsigned)(b * (b + 1) / 2), 256, 0, s>>>(Ms, W, rs, D, st);
  }
  WL_LAUNCH(h, "Cholesky scaling");
  wl_stage_end(h, tk, s);
  FxMaps m[2];
  for (int b = 0; b < 2; ++b)
    if ((rc = wl_sl_map(h, &m[b].i, fx_dig(h, Ms, w, b), nb * nkb, SL_BM)) ||
        (rc = wl_sl_map(h, &m[b].j, fx_dig(h, Ms, w, b), nb * nkb, SL_BN)))
      return rc;
  tk = wl_stage_begin(h, ST_SNR_CHOL, s);
  const int64_t SP = (int64_t)w * FX_NB, sms = wl_num_sms();
  // the panels of the super-panel at S0, in order
  auto chain = [&](int64_t S0, cudaStream_t st_) -> int {
    const int b = (int)((S0 / SP) & 1);
    const int64_t S1 = std::min(S0 + SP, Ms);
    for (int p = 0; p < w && S0 + (int64_t)p * FX_NB < Ms; ++p) {
      const int64_t k0 = S0 + (int64_t)p * FX_NB;
      const int slot = (int)((k0 / FX_NB) & 1);
      FxPanel a{W, k0, Ms, S0 / SL_BM, (int)std::min<int64_t>(FX_NB, Ms - k0), 2 * p, nkb, fx_dig(h, Ms, w, b), y,
                ld + slot * FX_NB * FX_NB, ld + (slot ^ 1) * FX_NB * FX_NB, nrm, st, fx_wide(W)};
      const int64_t groups = std::max<int64_t>(0, (Ms - k0 - FX_NB + FX_RB - 1) / FX_RB);
      k_fx_panel<<<(unsigned)(groups + 1), FX_THREADS, FX_PSMEM, st_>>>(a);
      WL_LAUNCH(h, "k_fx_panel");
      int r;
      if ((r = fx_update(h, W, Ms, S0 / SL_BM, 2 * p, 2, nkb, k0 + FX_NB, S1, m[b], sms, st_))) return r;
    }
    return COV_OK;
  };
  if ((rc = chain(0, s))) return rc;
  for (int64_t S0 = 0; S0 + SP < Ms; S0 += SP) {
    const int b = (int)((S0 / SP) & 1);
    const int64_t S1 = S0 + SP, S2 = S1 + SP;
    const int64_t rest = (Ms - S2 + SL_BM - 1) / SL_BM;  // row blocks beyond the next super-panel
    if (h->chol_lookahead && S2 < Ms && rest * (rest + 1) >= sms) {
      // look-ahead: the next super-panel's columns first; its panels then run on the side
      // stream beside the rest of this update.  A panel CTA (52 KB of shared memory, 104
      // registers) fits an SM beside an update CTA (174 KB, 120); the inner updates need
      // SMs of their own: as many as finish their ~6 us tiles in the time that the rest (~4
      // us per tile and panel) leaves over the panels' own ~45 us each
      const double t_rest = 4.0 * w * (double)(rest * (rest + 1)) / (double)sms;
      const double inner = 6.0 * (double)(w * (w - 1) / 2 * ((Ms - S1 + SL_BM - 1) / SL_BM));
      const int64_t free_sms =
          std::max<int64_t>(sms / 19, std::min<int64_t>(sms / 2, (int64_t)(inner / std::max(t_rest - 45.0 * w, 1.0))));
      if ((rc = fx_update(h, W, Ms, S0 / SL_BM, 0, nkb, nkb, S1, std::min(S2, Ms), m[b], sms, s))) return rc;
      WL_CHECK(h, cudaEventRecord(h->ev_cols, s));
      WL_CHECK(h, cudaStreamWaitEvent(h->side, h->ev_cols, 0));
      if ((rc = chain(S1, h->side))) return rc;
      WL_CHECK(h, cudaEventRecord(h->ev_panel, h->side));
      if ((rc = fx_update(h, W, Ms, S0 / SL_BM, 0, nkb, nkb, S2, nb * SL_BM, m[b], sms - free_sms, s)))
        return rc;
      WL_CHECK(h, cudaStreamWaitEvent(s, h->ev_panel, 0));
    } else {
      if ((rc = fx_update(h, W, Ms, S0 / SL_BM, 0, nkb, nkb, S1, nb * SL_BM, m[b], sms, s))) return rc;
      if ((rc = chain(S1, s))) return rc;
    }
  }
  const int64_t kl = (Ms - 1) / FX_NB * FX_NB;
  k_fx_tail<<<(unsigned)std::min<int64_t>(sms, (Ms + 255) / 256), 256, 0, s>>>(
      W, Ms, kl, (int)(Ms - kl), ld + ((kl / FX_NB) & 1) * FX_NB * FX_NB, y);
  WL_LAUNCH(h, "k_fx_tail");
  wl_stage_end(h, tk, s);
  return COV_OK;
}
