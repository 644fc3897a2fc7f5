// FP64 form of the 1-halo (chi, M) contraction on the tcgen05 tensor cores
// (paper Eqs. CovPPNG, Ins5P, Ins6P as C_1h = A A^T with A the factor rows, the
// super-sample rows of Eq. WLSSCflatskyLimber as further columns, and the 1-halo
// trispectrum table of Eq. CovBB), by integer slicing in the manner of Ozaki,
// Ogita & Oishi (2012).  This part multiplies FP64 at ~1.2 TFLOP/s, BF16 at ~1900.
//
//   * Rows.  Every K block (32 entries) of a factor row is scaled by a power of two 2^-e
//     that brings its 2-norm below sqrt(2), rounded to x = X 2^-55 with an integer X, and
//     cut into the seven balanced base-256 digits of X: x = sum_t d_t 2^(-7-8t),
//     |d_0| <= 182, |d_t| <= 128, each exact in BF16 (k_sl_rows).  The entries of a row
//     span many decades along K, and two rows may overlap only where both are small: with
//     one exponent per row such an element kept the bits of its rows' norms, not its own
//     (relative error up to 2e-12 for the paper's two bins, 4e-12 for narrow bins and a wide
//     ell range).
//   * Products as described in digits.cuh, exact per K block.  By Cauchy-Schwarz a block's
//     sum is below 2^63 in units of 2^-62 (that is what the scaling is for).
//   * Recombination (sl_drain_aligned): the block sums of an element are shifted to one
//     unit per element, chosen from a bound of their total by the block exponents of its
//     row and column (sl_bound), rounded, and added as 64-bit integers: any order gives the
//     same value.  One rounding to FP64 at the end.
// Error of an element against 80-bit sums, relative to the sum of its terms' magnitudes, in
// units of 2^-53, on a CPU replica (200 rows each of the paper's 2 and 5 bins and of 1 to 10 bins
// with and without photo-z, ell from 2 to 2e4, N_chi 2 .. 256, N_M 2 .. 128): at most 27, 2-norm
// 0.4-1.4, where sequential FP64 sums of the same rows have 96 and 16; in every set-up both are
// below those of the sequential sums.  What is left out are the digit products of the levels
// t + u > 6, 2^-54 of a block's norms each.  Sequential sums of fewer than SL_FULL entries err less
// than that where few nodes are far apart (N_chi = 16, N_M = 20: 16 against 50), so there the
// level 7 is formed too (6; 34 instead of 28 digit products).
//
// Bound: the recombination (~25 integer operations per element and K block, two epilogue warps
// per scheduler), close behind the tensor pipe and L2 (a 128 x 128 tile reads 112 KB per K
// block).  K blocks that add nothing to a tile are not read (SlLive).  M = 6375, 400 K blocks:
// contraction 7.1 ms where k_gemm_lower took 415 + 4.4 ms (1.2 TFLOP/s), trispectrum table
// 37 -> 1.0 ms, rows 0.51 ms, whole FP64 assembly 464 -> 9.0 ms.  M = 818 (28 tiles in 5 parts
// each): contraction 0.29 ms, assembly 27.1 -> 0.66 ms.  (With one exponent per row: 11.8 and
// 0.63 ms.)
#include "digits.cuh"

#define SL_NG 4               // a tile is 128 x 128
#define SL_SPLIT_TILES 304                          // largest tile count whose K range is cut over several CTAs
#define SL_FULL 4096                                // entries per row below which the eighth level is formed

__global__ void k_rows_prep(int nchi, int nm, double inv_omega, const cov_cosmology* __restrict__ cosmo_p,
                            const double* chi, const double* wchi, const double* m, const double* om, const double* f,
                            double* g2, double* g3, double* c2, double* c3);

// ---------------------------------------------------------------- rows
// Descriptors of the trispectrum rows in the form of the data vector's: one per leg
// pair (L1 <= L2), L = bin * n_t + tomo: type, three bins, three tomographic bins
// (the third unused), index of the bin pair.
__global__ void k_sl_trd(int64_t ntrow, int nleg, int nt, int nl, int32_t* rd) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= ntrow) return;
  int L1 = 0;
  int64_t base = 0;
  while (base + (nleg - L1) <= r) {
    base += nleg - L1;
    ++L1;
  }
  const int L2 = L1 + (int)(r - base), b1 = L1 / nt, b2 = L2 / nt;  // L1 <= L2, so b1 <= b2
  int32_t* o = rd + 8 * r;
  o[0] = 0;
  o[1] = b1;
  o[2] = b2;
  o[3] = b2;
  o[4] = L1 % nt;
  o[5] = L2 % nt;
  o[6] = -1;
  o[7] = b1 * nl - b1 * (b1 - 1) / 2 + (b2 - b1);
}

// The (n, q) part of a row depends on its ell bins alone (its signature): bin b for P
// rows, triangle nl + t for B rows, bin pair for trispectrum rows (pairs != 0).
struct SlSig {
  int nl, nchi, nm, pairs;
  const double *U, *g2, *g3, *c2, *c3;
};
__device__ __forceinline__ int sl_sig(const SlSig& g, const int32_t* r) {
  return g.pairs ? r[7] : (r[0] == 0 ? r[1] : g.nl + r[7]);
}
__device__ __forceinline__ double sl_factor(const SlSig& g, int isB, int a, int b, int c, int n, int64_t kk) {
  const int64_t K = (int64_t)g.nchi * g.nm;
  return isB ? g.g3[kk] * g.c3[n] * g.U[a * K + kk] * g.U[b * K + kk] * g.U[c * K + kk]
             : g.g2[kk] * g.c2[n] * g.U[a * K + kk] * g.U[b * K + kk];
}

// Where a row's entries lie in its K blocks.  The masses of a node follow those of the node
// before; fewer than SL_FEW of them get a K block of their own, since rows that overlap in one
// node of a block only keep the bits of the whole block there (N_M = 12, N_chi = 16: 14 units
// of 2^-53 against 1.6; sequential sums 13).  The super-sample entries, one per node, come SL_SSC to a block for the same reason (N_chi =
// 64, narrow bins: 49 with 32 to a block, 4.6 with 8).
#define SL_FEW 16
#define SL_SSC 8
struct SlCols {
  int np, n1, nk;  // slots per node; K blocks of the factor row; all K blocks
};
__host__ __device__ static inline SlCols sl_cols(int nchi, int nm, bool ssc) {
  SlCols c;
  c.np = nm < SL_FEW ? SL_BK : nm;
  c.n1 = (int)(((int64_t)nchi * c.np + SL_BK - 1) / SL_BK);
  c.nk = c.n1 + (ssc ? (nchi + SL_SSC - 1) / SL_SSC : 0);
  return c;
}

struct SlSsc {
  int nssc;  // super-sample columns (N_chi or 0)
  const double *wchi, *sigw2, *chi, *RP3, *RB3;
};

// The lensing weight and super-sample entry of every row at every node
__global__ void __launch_bounds__(256) k_sl_weights(SlSig g, int64_t rows, const int32_t* __restrict__ rd,
                                                    const double* __restrict__ W, double wscale, SlSsc ss,
                                                    double* __restrict__ wrow, double* __restrict__ srow) {
  const int64_t id = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (id >= rows * g.nchi) return;
  const int64_t a = id / g.nchi;
  const int n = (int)(id % g.nchi), nchi = g.nchi;
  const int32_t* r = rd + 8 * a;
  const bool isB = r[0] != 0;
  double w = W[r[4] * nchi + n] * W[r[5] * nchi + n];
  if (isB) w *= W[r[6] * nchi + n];
  wrow[id] = w * wscale;
  if (ss.nssc) {
    const double c2 = ss.chi[n] * ss.chi[n], t = sqrt(ss.wchi[n] * ss.sigw2[n]) * w;
    srow[id] = isB ? t / (c2 * c2) * ss.RB3[r[7] * nchi + n] : t / c2 * ss.RP3[r[1] * nchi + n];
  }
}

// Exponents of a set of rows, behind its digit blocks: of every (row block, K block, row),
// an int16 (SL_EMPTY: no entry, SL_BAD: an infinity or NaN) and its distance below the row's
// largest in a byte, SL_NONE for an empty block and beyond SL_FAR; the least distance in every
// (row block, K block); and of every (row block, group of K blocks, row).  A group is one K
// block where there are few (nodes far apart: a group of four costs up to 6 bits of an
// element's unit at N_chi = 16), else four (1 bit).
#define SL_FINE 128      // K blocks up to which a group is one of them
#define SL_GB 4
#define SL_SG 8          // groups per term of the bound (sl_bound)
#define SL_EMPTY (-20000)
#define SL_BAD 20000
#define SL_FAR 104
#define SL_NONE 112
struct SlExp {
  int16_t* e;
  uint16_t* gd;
  uint8_t *d, *bd;
  int nk, gb, ng;  // K blocks, K blocks per group, groups
};
__host__ __device__ static inline SlExp sl_exp(uint8_t* dig, int64_t nb, int64_t nk) {
  SlExp x;
  x.nk = (int)nk;
  x.gb = nk <= SL_FINE ? 1 : SL_GB;
  x.ng = (int)((nk + x.gb - 1) / x.gb);
  x.gd = (uint16_t*)(dig + (size_t)nb * nk * SL_BLOCK);
  x.e = (int16_t*)(x.gd + (size_t)nb * x.ng * SL_BM);
  x.d = (uint8_t*)(x.e + (size_t)nb * nk * SL_BM);
  x.bd = x.d + (size_t)nb * nk * SL_BM;
  return x;
}

// The distances, and the row's largest exponent (0 for an empty row, SL_BAD for one that is
// not finite).  One CTA per row block; a warp holds all 128 rows, four to a lane, of every 32nd
// K block or group (bound by the latency of its passes: 16 us with a row to a thread).
__global__ void __launch_bounds__(1024) k_sl_exp(SlExp x, int64_t rows, int* rexp) {
  __shared__ int4 mx[32][SL_BM / 4];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t rb = blockIdx.x;
  const short4* e = (const short4*)(x.e + (size_t)rb * x.nk * SL_BM) + lane;
  int m[4] = {SL_EMPTY, SL_EMPTY, SL_EMPTY, SL_EMPTY};
#pragma unroll 4
  for (int k = warp; k < x.nk; k += 32) {
    const short4 v = e[(size_t)k * (SL_BM / 4)];
    m[0] = max(m[0], (int)v.x);
    m[1] = max(m[1], (int)v.y);
    m[2] = max(m[2], (int)v.z);
    m[3] = max(m[3], (int)v.w);
  }
  mx[warp][lane] = make_int4(m[0], m[1], m[2], m[3]);
  __syncthreads();
#pragma unroll 8
  for (int i = 0; i < 32; ++i) {
    const int4 v = mx[i][lane];
    m[0] = max(m[0], v.x);
    m[1] = max(m[1], v.y);
    m[2] = max(m[2], v.z);
    m[3] = max(m[3], v.w);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (m[c] == SL_EMPTY) m[c] = 0;
    const int64_t r = rb * SL_BM + 4 * lane + c;
    if (warp == 0 && r < rows) rexp[r] = m[c];
  }
  uchar4* d = (uchar4*)(x.d + (size_t)rb * x.nk * SL_BM) + lane;
#pragma unroll 2
  for (int g = warp; g < x.ng; g += 32) {
    int lo[4] = {SL_NONE, SL_NONE, SL_NONE, SL_NONE};
#pragma unroll
    for (int i = 0; i < SL_GB; ++i) {
      const int k = g * x.gb + i;
      if (i < x.gb && k < x.nk) {
        const short4 s = e[(size_t)k * (SL_BM / 4)];
        const int at[4] = {s.x, s.y, s.z, s.w};
        int v[4], least = SL_NONE;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          v[c] = m[c] - at[c] > SL_FAR ? SL_NONE : m[c] - at[c];
          lo[c] = min(lo[c], v[c]);
          least = min(least, v[c]);
        }
        d[(size_t)k * (SL_BM / 4)] = make_uchar4((uint8_t)v[0], (uint8_t)v[1], (uint8_t)v[2], (uint8_t)v[3]);
        least = __reduce_min_sync(0xffffffffu, least);
        if (lane == 0) x.bd[(size_t)rb * x.nk + k] = (uint8_t)least;
      }
    }
    *((ushort4*)(x.gd + ((size_t)rb * x.ng + g) * SL_BM) + lane) =
        make_ushort4((uint16_t)lo[0], (uint16_t)lo[1], (uint16_t)lo[2], (uint16_t)lo[3]);
  }
}

// Digits of 128 rows x 32 K, one contiguous 56 KB block per (row block, K block):
// [digit][row][k].  The factor of each signature present among the rows is formed
// once in shared memory; an entry is then one FP64 product (the bound here beside the
// 14 bytes written per entry: 5-bin rows, 7.9e7 entries).  A thread holds 8
// consecutive k of one row and stores each digit's 16 bytes at once; the four threads of a
// row's K block agree on its exponent from its largest entry's and an FP32 sum of squares
// (mantissas cut to 24 bits: 2^-17 in all, inside the margin of 2^-11).
#define SR_THREADS 256
__global__ void __launch_bounds__(SR_THREADS)
    k_sl_rows(SlSig g, int64_t rows, SlCols cols, const int32_t* __restrict__ rd,
              const double* __restrict__ wrow, const double* __restrict__ srow, uint8_t* __restrict__ out,
              int16_t* __restrict__ ex) {
  __shared__ double F[SL_BM][SL_BK + 1];
  __shared__ int slot[SL_BM];
  __shared__ int first[SL_BM];  // a row of each signature slot
  __shared__ int nslot_sh[SL_BM / 32];
  const int64_t rb = blockIdx.y, kb = blockIdx.x, r0 = rb * SL_BM;
  const bool ssc = kb >= cols.n1;
  const int n0 = ssc ? (int)(kb - cols.n1) * SL_SSC : 0;  // first node of a super-sample block
  const int64_t k0 = kb * SL_BK;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // rows with equal signatures are consecutive: number the runs
  if (tid < SL_BM) {
    const int64_t r = r0 + tid;
    bool head = false;
    if (r < rows) {
      const int s = sl_sig(g, rd + 8 * r);
      head = tid == 0 || sl_sig(g, rd + 8 * (r - 1)) != s;
    }
    const unsigned mk = __ballot_sync(0xffffffffu, head);
    slot[tid] = __popc(mk & (0xffffffffu >> (31 - lane)));
    if (lane == 0) nslot_sh[warp] = __popc(mk);
  }
  __syncthreads();
  int nslot = 0;
  for (int w = 0; w < SL_BM / 32; ++w) nslot += nslot_sh[w];
  if (tid < SL_BM) {
    int base = 0;
    for (int w = 0; w < warp; ++w) base += nslot_sh[w];
    const int s = slot[tid] + base - 1;  // >= 0: the block's first row is a head
    const int64_t r = r0 + tid;
    slot[tid] = s;
    if (r < rows && (tid == 0 || sl_sig(g, rd + 8 * (r - 1)) != sl_sig(g, rd + 8 * r))) first[s] = tid;
  }
  __syncthreads();
  for (int e = tid; e < (ssc ? 0 : nslot * SL_BK); e += SR_THREADS) {
    const int s = e / SL_BK, k = e % SL_BK;
    const int n = (int)((k0 + k) / cols.np), q = (int)((k0 + k) % cols.np);
    if (n < g.nchi && q < g.nm) {
      const int32_t* r = rd + 8 * (r0 + first[s]);
      F[s][k] = sl_factor(g, r[0] != 0, r[1], r[2], r[3], n, (int64_t)n * g.nm + q);
    }
  }
  __syncthreads();
  uint8_t* o = out + ((size_t)rb * cols.nk + kb) * SL_BLOCK;
  for (int e = tid; e < SL_BM * (SL_BK / 8); e += SR_THREADS) {
    const int row = e >> 2, k8 = (e & 3) * 8;
    const int64_t r = r0 + row;
    const double* wr = wrow + r * g.nchi;
    const double* sr = srow + r * g.nchi;
    double v[8];
    long long X[8];
    uint4 d[SL_S];
    int n = (int)((k0 + k8) / cols.np), q = (int)((k0 + k8) % cols.np), E = 0;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      v[p] = 0.0;
      if (r < rows) {
        if (ssc) {
          if (k8 + p < SL_SSC && n0 + k8 + p < g.nchi) v[p] = sr[n0 + k8 + p];
        } else if (n < g.nchi && q < g.nm) {
          v[p] = F[slot[row]][k8 + p] * wr[n];
        }
      }
      if (++q == cols.np) {
        q = 0;
        ++n;
      }
      E = max(E, (__double2hiint(v[p]) >> 20) & 0x7FF);
    }
    E = max(E, __shfl_xor_sync(0xffffffffu, E, 1));
    E = max(E, __shfl_xor_sync(0xffffffffu, E, 2));
    float s2 = 0.0f;  // squares in units of the largest entry's power of two: 1 .. 128
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const unsigned long long b = (unsigned long long)__double_as_longlong(v[p]);
      const int below = E - (int)((b >> 52) & 0x7FFu);
      const float f =
          below < 40 ? __uint_as_float((unsigned)(127 - below) << 23 | ((unsigned)(b >> 29) & 0x7FFFFFu)) : 0.0f;
      s2 = fmaf(f, f, s2);
    }
    s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 2);
    s2 *= 1.0f + 0x1p-11f;
    int e2 = E - 1023 + (s2 > 2.0f) + (s2 > 8.0f) + (s2 > 32.0f) + (s2 > 128.0f);
    if (E == 0x7FF) e2 = SL_BAD;
    if (E == 0) e2 = SL_EMPTY;  // (subnormal entries count as 0)
    if ((e & 3) == 0) ex[((size_t)rb * cols.nk + kb) * SL_BM + row] = (int16_t)e2;
#pragma unroll
    for (int p = 0; p < 8; ++p) X[p] = E == 0 || E == 0x7FF ? 0 : sl_int(v[p], e2);
    sl_digits8(X, d);
#pragma unroll
    for (int t = 0; t < SL_S; ++t)
      *(uint4*)(o + (size_t)t * SL_DIGIT + row * (SL_BK * 2) + k8 * 2) = d[t];
  }
}

// ---------------------------------------------------------------- contraction
// Launch order of the lower 128 x 128 tiles of tile rows [t0, t1): groups of 8 tile
// rows, column by column inside a group, so that the CTAs of a wave share few row
// and column blocks in L2.
#define SL_ORDER 8
__device__ __forceinline__ void sl_tile(int64_t id, int64_t t0, int64_t t1, int64_t* ti, int64_t* tj) {
  const int64_t base = t0 * (t0 + 1) / 2;
  int64_t lo = 0, hi = (t1 - t0 + SL_ORDER - 1) / SL_ORDER;  // group of id by bisection on the tiles before it
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1, r = t0 + mid * SL_ORDER;
    if (r * (r + 1) / 2 - base <= id)
      lo = mid;
    else
      hi = mid;
  }
  const int64_t r = t0 + lo * SL_ORDER, nr = t1 - r < SL_ORDER ? t1 - r : SL_ORDER;
  int64_t o = id - (r * (r + 1) / 2 - base);
  if (o < (r + 1) * nr) {  // columns 0 .. r: all nr rows
    *tj = o / nr;
    *ti = r + o % nr;
    return;
  }
  o -= (r + 1) * nr;
  int64_t c = 1;  // column r + c holds rows r + c .. r + nr - 1
  while (o >= nr - c) {
    o -= nr - c;
    ++c;
  }
  *tj = r + c;
  *ti = r + c + o;
}

// An element's sum to FP64: e the exponents of its row and column, H as sl_bound gives it.
// An infinity or NaN in either row, and a sum left incomplete (e = SL_BAD): NaN.  (An element
// whose rows overlap in no block above 2^-112 of their largest has H = 0 and sum 0.)
__device__ __forceinline__ double sl_value(unsigned long long sum, int e, int H) {
  return e > SL_BAD / 2 ? __longlong_as_double(0x7FF8000000000000ll) : scaled_to_double_rn((long long)sum, e - H - 42);
}

// Units of this thread's 64 elements (row: the lane's, columns 16 half .. of each group).
// With block exponents d (distance below the row's largest) a block's sum is below
// 2^63 2^-(d_i + d_j) in units of 2^-62 of the rows' largest; the unit 2^(-H + 20 - 62) is the
// finest for which the sum of these bounds over the K blocks stays below 2^63.  The bound
// takes the largest term of SL_SG groups times the number of their K blocks, with the
// groups' least distances: ~1.2 operations per group and element.  H = 246 - exponent
// field of (2^100 bound), 0 .. 130, four to a word; 0 where all distances are SL_NONE or more (no
// shift is below 64 then).  Returns the largest H.  The distances come through shared
// memory (from L2 in the loop, every group waited for it: 70 us per tile of 388 K blocks
// against 10).  gi, gj: of the row blocks; called by the epilogue warps together.
#define SL_CHUNK 256  // groups staged at a time: 64 KB for the rows, 64 KB for the columns
__device__ __forceinline__ int sl_bound(const uint16_t* gi, const uint16_t* gj, const SlExp& x, uint8_t* smem, int row,
                                        int half, uint32_t (*H)[4]) {
  float B[SL_NG][16];
  uint32_t lo[SL_NG][8];
#pragma unroll
  for (int j = 0; j < SL_NG; ++j) {
#pragma unroll
    for (int c = 0; c < 16; ++c) B[j][c] = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; ++c) lo[j][c] = 0x00FF00FFu;
  }
  uint4 *si = (uint4*)smem, *sj = si + SL_CHUNK * (SL_BM / 8);
  for (int c0 = 0; c0 < x.ng; c0 += SL_CHUNK) {
    const int cn = min(SL_CHUNK, x.ng - c0);
    if (c0) asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll 4
    for (int e = threadIdx.x & 255; e < cn * (SL_BM / 8); e += 256) {
      si[e] = __ldg((const uint4*)(gi + (size_t)c0 * SL_BM) + e);
      sj[e] = __ldg((const uint4*)(gj + (size_t)c0 * SL_BM) + e);
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll 1
    for (int s0 = 0; s0 < cn; s0 += SL_SG) {
      const int s1 = min(cn, s0 + SL_SG);
      const float cnt = (float)(min(x.nk, (c0 + s1) * x.gb) - (c0 + s0) * x.gb);
      uint32_t m[SL_NG][8];
#pragma unroll
      for (int j = 0; j < SL_NG; ++j)
#pragma unroll
        for (int c = 0; c < 8; ++c) m[j][c] = 0x00FF00FFu;
#pragma unroll 1
      for (int g = s0; g < s1; ++g) {
        const uint32_t a = ((const uint16_t*)si)[g * SL_BM + row] * 0x10001u;
        const uint4* q = sj + g * (SL_BM / 8) + 2 * half;
#pragma unroll
        for (int j = 0; j < SL_NG; ++j) {
          const uint4 b0 = q[j * (SL_BN / 8)], b1 = q[j * (SL_BN / 8) + 1];
          const uint32_t b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
          for (int c = 0; c < 8; ++c) m[j][c] = __viaddmin_u16x2(b[c], a, m[j][c]);
        }
      }
#pragma unroll
      for (int j = 0; j < SL_NG; ++j) {
#pragma unroll
        for (int c = 0; c < 8; ++c) lo[j][c] = __vminu2(lo[j][c], m[j][c]);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int v = (int)((m[j][c >> 1] >> (16 * (c & 1))) & 0xFFFFu);
          B[j][c] = fmaf(cnt, __int_as_float((227 - v) << 23), B[j][c]);
        }
      }
    }
  }
  uint32_t top = 0;
#pragma unroll
  for (int j = 0; j < SL_NG; ++j)
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      uint32_t w = 0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int e = 246 - (int)(__float_as_uint(B[j][4 * h + c] * (1.0f + 0x1p-10f)) >> 23);
        const uint32_t least = (lo[j][(4 * h + c) >> 1] >> (16 * (c & 1))) & 0xFFFFu;
        w |= (least < SL_NONE ? (uint32_t)max(e, 0) : 0u) << (8 * c);
      }
      top = __vmaxu4(top, w);
      H[j][h] = w;
    }
  top = __vmaxu4(top, top >> 16);
  return (int)max(top & 255u, (top >> 8) & 255u);
}

// The K blocks that reach a tile's elements, in order: the others' shifts are 64 or more
// throughout (d_i + d_j >= limit = 44 + the largest H), they add exactly 0 and are neither
// read nor multiplied.  The masses of a node span up to 15 decades in the rows: ~0.6 of the K
// blocks are left (the paper's and the 5-bin rows).  Part sp of ns takes an equal share of what
// is left.  Run by a whole warp; the first SL_WORDS words of 32 blocks lie in shared memory.
#define SL_WORDS 64
struct SlLive {
  const uint8_t *bi, *bj;
  int nk, limit;
  __device__ __forceinline__ SlLive(const SlExp& x, int64_t ti, int64_t tj, int hmax)
      : bi(x.bd + (size_t)ti * x.nk), bj(x.bd + (size_t)tj * x.nk), nk(x.nk), limit(44 + hmax) {}
  __device__ __forceinline__ uint32_t word(int w) const {
    const int i = 32 * w + (threadIdx.x & 31);
    return __ballot_sync(0xffffffffu, i < nk && (int)__ldg(bi + i) + (int)__ldg(bj + i) < limit);
  }
};
struct SlWalk {
  SlLive live;
  const uint32_t* sh;
  int w, nw, left;
  uint32_t mask;
  __device__ __forceinline__ SlWalk(const SlLive& l, const uint32_t* words, int sp, int ns)
      : live(l), sh(words), w(0), nw((l.nk + 31) / 32), left(l.nk), mask(0) {
    if (ns == 1) return;
    int64_t n = 0;
    for (int i = 0; i < nw; ++i) n += __popc(word(i));
    int skip = (int)(n * sp / ns);
    left = (int)(n * (sp + 1) / ns) - skip;
    while (skip > 0) {
      mask = word(w++);
      const int c = __popc(mask);
      if (c <= skip) {
        skip -= c;
        mask = 0;
      } else {
        for (; skip > 0; --skip) mask &= mask - 1;
      }
    }
  }
  __device__ __forceinline__ uint32_t word(int i) const { return i < SL_WORDS ? sh[i] : live.word(i); }
  __device__ __forceinline__ int next() {  // -1 at the end
    if (left == 0) return -1;
    while (mask == 0) {
      if (w >= nw) return -1;
      mask = word(w++);
    }
    const int b = __ffs((int)mask) - 1;
    mask &= mask - 1;
    --left;
    return 32 * (w - 1) + b;
  }
};

// Epilogue warps: acc[j][c] += the level sums of a K block (S, units of 2^-62) shifted right by
// s = d_i + d_j + 20 - H, rounded: t = floor(S 2^-s) plus its lowest bit, i.e. twice the
// integer nearest to S 2^(-s-1) (a plain floor would leave half a unit per block: 1e-14 of an
// element after 388 blocks).  di: the distances of this thread's row in K block 0, dj: of its
// columns.  Otherwise as sl_drain.
template <int LV>
__device__ __forceinline__ bool sl_drain_aligned(unsigned long long (&acc)[SL_NG][16], const uint32_t (&H)[SL_NG][4],
                                                 const uint8_t* di, const uint8_t* dj, SlWalk walk, SlBars* B,
                                                 int q, int half, int* status) {
  int ok = 1;
  const int lane = threadIdx.x & 31;
  const uint32_t tbase = ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 16);  // (the 512 columns start at 0)
  int k = walk.next();
  uint4 nb = make_uint4(0, 0, 0, 0);
  uint32_t na = 0;
  if (k >= 0) {
    nb = __ldg((const uint4*)(dj + (size_t)k * SL_BM));
    na = __ldg(di + (size_t)k * SL_BM);
  }
  for (int w = 0; k >= 0 && ok; ++w) {
    const uint32_t a = (na + 20u) * 0x01010101u;
    const int k1 = walk.next();
    if (k1 >= 0) na = __ldg(di + (size_t)k1 * SL_BM);
    uint32_t r[2][LV][4];  // the levels of four columns; the next four are on their way meanwhile
    auto load = [&](int j, int h) {
#pragma unroll
      for (int g = 0; g < LV; ++g)
        sl_tmem_ld4<false>(tbase + (uint32_t)((j & 1) * 256) + sl_part<false>(h) + g * SL_BN, r[h & 1][g]);
    };
#pragma unroll
    for (int j = 0; j < SL_NG; ++j) {
      const uint32_t b[4] = {nb.x, nb.y, nb.z, nb.w};
      // the next group's distances, on their way while this one waits
      const uint8_t* next = dj + (size_t)(j + 1 < SL_NG ? k : k1) * SL_BM + (j + 1 < SL_NG ? (j + 1) * SL_BN : 0);
      if (j + 1 < SL_NG || k1 >= 0) nb = __ldg((const uint4*)next);
      if (ok) {  // (warp-uniform: the TMEM accesses are warp-collective)
        if (lane == 0) ok = sl_wait(&B->tfull[j & 1], (uint32_t)(((SL_NG / 2) * w + (j >> 1)) & 1), status);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
      }
      if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        load(j, 0);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          uint32_t(&x4)[LV][4] = r[h & 1];
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int g = 0; g < LV; ++g)
#pragma unroll
            for (int c = 0; c < 4; ++c) asm volatile("" : "+r"(x4[g][c]));
          if (h < 3) {
            load(j, h + 1);
          } else {  // the set has been read: its constants, on their way while the last columns are added
#pragma unroll
            for (int g = 0; g < LV; ++g)
#pragma unroll
              for (int i = 0; i < 16; i += 4) sl_tmem_st4<false>(tbase + (uint32_t)((j & 1) * 256 + g * SL_BN + i), SL_MAGIC);
          }
          const uint32_t s4 = b[h] + a - H[j][h];  // four shifts, 1 .. 244
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            unsigned long long x = 0ull - SL_BIAS;
            x += (unsigned long long)(x4[3][c] * 256u + x4[4][c]) * 65536ull;
            uint32_t y = x4[5][c] * 256u + x4[6][c];
            if (LV > SL_S) y += (uint32_t)((int)(x4[LV - 1][c] - (SL_MAGIC - 128u)) >> 8);  // the eighth level, rounded
            x += (unsigned long long)y;
            x += (unsigned long long)(x4[0][c] * 65536u + x4[1][c] * 256u + x4[2][c]) << 32;
            long long t;
            asm("shr.s64 %0, %1, %2;" : "=l"(t) : "l"(x), "r"((s4 >> (8 * c)) & 255u));  // (64 and more: the sign)
            acc[j][h * 4 + c] += (unsigned long long)t + (unsigned long long)(t & 1);
          }
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) sl_arrive(&B->tempty[j & 1]);
      }
    }
    k = k1;
  }
  return ok != 0;
}

struct SlArgs {
  int64_t row1, t0, t1;
  int nk, ns;                 // K blocks; CTAs that share a tile's K range
  const int* rexp;
  SlExp x;
  OutMap out;
  int *status, *report;       // an expired wait of this assembly; of any since the host last read it
  unsigned long long* part;   // [tile][column][row] exact partial sums (ns > 1), zero at launch
  int* ticket;                // [tile] CTAs that have delivered (ns > 1), 2^16 for each that gave up, zero at launch
};

// One CTA per (128 x 128 lower tile, part of its live K blocks).  Warp 0 loads (TMA, two
// stages of a K block: the I block in one box, the J block as four groups of 32 rows), warp
// 1 issues the MMAs of the four column groups in turn into two accumulator sets (LV x 32
// columns each), warps 4-11 recombine the set of the group before in registers (64
// 64-bit sums per thread).  Where a launch has too few tiles for the SMs, ns CTAs take
// parts of a tile's K range, add their 64-bit sums atomically (integers: any order
// gives the same value) and the last one converts.  The host does not wait for this kernel:
// where a wait expires, the elements that it leaves incomplete are stored as NaN.
// An epilogue thread holds 64 64-bit sums, their units and a K block's levels (~190
// registers, of 168 that 12 warps can have each): the first four warps hand over what they do
// not need (128 x 56 + 256 x 224 = 384 x 168 registers).
#define SC_THREADS 384
template <int LV>
__global__ void __launch_bounds__(SC_THREADS, 1)
    k_syrk_sl(const __grid_constant__ CUtensorMap map_i, const __grid_constant__ CUtensorMap map_j, SlArgs A) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) SlBars bars;
  __shared__ uint32_t tmem_sh;
  __shared__ int last_sh, gave_up, hmax;
  __shared__ uint32_t words[SL_WORDS];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  // (the same in every lane: TMEM addresses stay in uniform registers)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int64_t tile = blockIdx.x / A.ns;
  const int sp = (int)(blockIdx.x % A.ns);
  int64_t ti, tj;
  sl_tile(tile, A.t0, A.t1, &ti, &tj);
  if (threadIdx.x == 0) {
    sl_bars_init(&bars);
    gave_up = hmax = 0;
  }
  if (warp == 0) sl_tmem_alloc(&tmem_sh);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_sh;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    __syncthreads();  // the largest H, the live K blocks
    SlWalk walk(SlLive(A.x, ti, tj, hmax), words, sp, A.ns);
    int it = 0, ok = 1;
    if (warp == 0) {
      const int bi = (int)(ti * A.nk), bj = (int)(tj * A.nk);
      int k = walk.next(), k1 = k < 0 ? -1 : walk.next();
      while (k >= 0 && ok) {
        const int k2 = k1 < 0 ? -1 : walk.next();
        if (lane == 0) {
          ok = sl_produce<SL_NG>(&map_i, &map_j, smem, &bars, bi + k, bj + k, 0, 1, it, A.status);
          if (k2 >= 0) {
            sl_prefetch(&map_i, 0, bi + k2);
            if (bi != bj) sl_prefetch(&map_i, 0, bj + k2);
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        k = k1;
        k1 = k2;
      }
    } else if (warp == 1) {
      while (ok && walk.next() >= 0) ok = sl_issue<SL_NG, false, LV>(smem, &bars, 1, it, A.status);
      if (it > 0 || !ok) sl_issue_end(&bars, lane);
    }
    __syncwarp();
    if (warp == 0 && lane == 0) sl_pause(A.status);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) sl_tmem_free(tmem);
    if (threadIdx.x == 0) {
      if (*(volatile int*)A.status != 0) atomicExch(A.report, 1);
      if (A.ns > 1) {  // 1: the last CTA of the tile, 2: and one of them gave up
        const int add = gave_up ? 65537 : 1, t = atomicAdd(A.ticket + tile, add) + add;
        last_sh = (t & 65535) != A.ns ? 0 : t > 65535 ? 2 : 1;
      }
    }
    if (A.ns > 1) __syncthreads();
    return;
  }

  asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
  const int q = warp & 3, half = (warp - 4) >> 2;  // TMEM lanes 32 q .., columns 16 half .. of a group
  unsigned long long acc[SL_NG][16];               // this thread's sums
  uint32_t H[SL_NG][4] = {};                       // and their units
  auto store = [&](bool good) {
    const int64_t gr = ti * SL_BM + sl_row<false>(q, lane, 0);
    if (gr >= A.row1) return;
    const int er = good ? A.rexp[gr] : SL_BAD;
    double* p = A.out.at(gr, tj * SL_BM);
#pragma unroll
    for (int j = 0; j < SL_NG; ++j)
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int lc = sl_col<false>(half, lane, j, c);
        const int64_t gc = tj * SL_BM + lc;
        if (gc <= gr) p[lc] = sl_value(acc[j][c], er + __ldg(A.rexp + gc), (int)((H[j][c >> 2] >> (8 * (c & 3))) & 255u));
      }
  };
#pragma unroll
  for (int j = 0; j < SL_NG; ++j)
#pragma unroll
    for (int c = 0; c < 16; ++c) acc[j][c] = 0ull;
  sl_drain_init<false, LV>(&bars, tmem, q, half, lane);
  const int top = sl_bound(A.x.gd + (size_t)ti * A.x.ng * SL_BM, A.x.gd + (size_t)tj * A.x.ng * SL_BM, A.x, smem,
                           q * 32 + lane, half, H);
  const int wtop = __reduce_max_sync(0xffffffffu, top);
  if (lane == 0) atomicMax(&hmax, wtop);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the copies overwrite what sl_bound has staged
  asm volatile("bar.sync 1, 256;" ::: "memory");
  const SlLive live(A.x, ti, tj, hmax);
  for (int w = warp - 4; w < SL_WORDS && 32 * w < A.nk; w += 8) {
    const uint32_t m = live.word(w);
    if (lane == 0) words[w] = m;
  }
  __syncthreads();
  const bool ok = sl_drain_aligned<LV>(acc, H, A.x.d + (size_t)ti * A.nk * SL_BM + q * 32 + lane,
                                       A.x.d + (size_t)tj * A.nk * SL_BM + half * 16,
                                       SlWalk(live, words, sp, A.ns), &bars, q, half, A.status);
  if (!ok) gave_up = 1;
  unsigned long long* part = A.part + (size_t)tile * (SL_BM * SL_BM);
  if (A.ns == 1) {
    store(ok);
  } else if (ok) {
#pragma unroll
    for (int j = 0; j < SL_NG; ++j)
#pragma unroll
      for (int c = 0; c < 16; ++c)
        atomicAdd(part + (size_t)sl_col<false>(half, lane, j, c) * SL_BM + sl_row<false>(q, lane, c), acc[j][c]);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (A.ns > 1) __threadfence();
  __syncthreads();
  if (A.ns == 1) return;
  __syncthreads();
  if (last_sh == 0) return;
  __threadfence();
#pragma unroll
  for (int j = 0; j < SL_NG; ++j)
#pragma unroll
    for (int c = 0; c < 16; ++c)
      acc[j][c] = __ldcg(part + (size_t)sl_col<false>(half, lane, j, c) * SL_BM + sl_row<false>(q, lane, c));
  store(last_sh == 1);
}

// ---------------------------------------------------------------- host side
// bytes of the digits of the factor rows (with super-sample columns) or the trispectrum rows
// (tri) and their exponents
size_t wl_sl_bytes(const cov_handle* h, bool tri) {
  const size_t nb = (size_t)(((tri ? h->ntrow : h->M) + SL_BM - 1) / SL_BM);
  const size_t nk = (size_t)sl_cols(h->nchi, h->nm, !tri).nk;
  // (the groups of the columns with or without the super-sample ones)
  return nb * (nk * (SL_BLOCK + 3 * SL_BM + 1) + (std::min<size_t>(nk, SL_FINE) + nk / SL_GB + 1) * 2 * SL_BM);
}

// upper bound of what wl_sl_alloc takes beside the digits themselves
size_t wl_sl_fixed_bytes(const cov_handle* h) {
  const size_t M = (size_t)h->M, T = (size_t)h->ntrow, nchi = (size_t)h->nchi;
  return 8 * (std::max(M, T) + M) * nchi + 4 * M + 36 * T + 16 * ((size_t)h->K + nchi) +
         (size_t)SL_SPLIT_TILES * (SL_BM * SL_BM * 8 + sizeof(int));
}

int wl_sl_map(cov_handle* h, CUtensorMap* map, void* base, int64_t blocks, int box_rows) {
  auto fn = wl_encode_tiled();
  if (!fn) return wl_fail(h, COV_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
  cuuint64_t dims[4] = {SL_BK, SL_BM, SL_S, (cuuint64_t)blocks};
  cuuint64_t strides[3] = {SL_BK * 2, SL_DIGIT, SL_BLOCK};
  cuuint32_t box[4] = {SL_BK, (cuuint32_t)box_rows, SL_S, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return wl_fail(h, COV_ERR_CUDA, "cuTensorMapEncodeTiled failed (digit blocks)");
  return COV_OK;
}

// Digits of the 1-halo factor rows (with nssc super-sample columns) or of the
// trispectrum rows (tri).  The buffers exist already (wl_sl_alloc).
int wl_sl_rows(cov_handle* h, bool tri, int nssc, cudaStream_t s) {
  SlSig g{h->nl, h->nchi, h->nm, tri ? 1 : 0, h->U, h->G2, h->G3, h->C2, h->C3};
  const int64_t rows = tri ? h->ntrow : h->M;
  const int32_t* rd = tri ? h->trd : h->rowdesc_d;
  const SlCols cols = sl_cols(h->nchi, h->nm, nssc > 0);
  int* rexp = tri ? h->Texp : h->Aexp;
  k_rows_prep<<<(h->K + 255) / 256, 256, 0, s>>>(h->nchi, h->nm, 1.0 / h->omega, h->cosmo_d, h->chi, h->wchi, h->m,
                                                 h->om, h->f, h->G2, h->G3, h->C2, h->C3);
  SlSsc ss{nssc, h->wchi, h->sigw2, h->chi, h->RP3, h->RB3};
  k_sl_weights<<<(unsigned)((rows * h->nchi + 255) / 256), 256, 0, s>>>(g, rows, rd, h->W, tri ? sqrt(h->omega) : 1.0, ss,
                                                                        h->sl_w, h->sl_sr);
  const int64_t nb = (rows + SL_BM - 1) / SL_BM;
  uint8_t* dig = tri ? h->Tsl : h->Asl;
  const SlExp x = sl_exp(dig, nb, cols.nk);
  k_sl_rows<<<dim3((unsigned)cols.nk, (unsigned)nb), SR_THREADS, 0, s>>>(g, rows, cols, rd, h->sl_w, h->sl_sr, dig, x.e);
  k_sl_exp<<<(unsigned)nb, 1024, 0, s>>>(x, rows, rexp);
  WL_LAUNCH(h, "digit row kernels");
  return COV_OK;
}

// Whether the tensor-core FP64 form serves the handle's rows (tri: its trispectrum
// rows), and its buffers.  The digits take 14 bytes per entry where the FP64 rows of
// k_gemm_lower take 8; where they do not fit (in hbm_budget, or the free memory, beside
// all that the handle's other calls may still allocate) the FP64 rows and that kernel
// serve the handle as before.  A served request's reservation was made with the digits in it,
// so there they only have to fit.  Decided once per handle: a later call with more
// super-sample columns finds room for them.
int wl_sl_alloc(cov_handle* h, bool tri, bool* use, cudaStream_t s) {
  int& state = tri ? h->sl_tri : h->sl_rows;
  if (state) {
    *use = state > 0;
    return COV_OK;
  }
  const int64_t rows = tri ? h->ntrow : h->M;
  const size_t d = sizeof(double), K = (size_t)h->K;
  const size_t wmax = (size_t)std::max<int64_t>(h->M, h->ntrow) * h->nchi;
  struct {
    void** p;
    size_t n;
  } al[] = {{(void**)(tri ? &h->Tsl : &h->Asl), wl_sl_bytes(h, tri)},
            {(void**)(tri ? &h->Texp : &h->Aexp), sizeof(int) * (size_t)rows},
            {(void**)&h->trd, tri ? sizeof(int32_t) * 8 * (size_t)rows : 0},
            {(void**)&h->sl_w, d * wmax},
            {(void**)&h->sl_sr, d * (size_t)h->M * h->nchi},
            {(void**)&h->G2, d * K},
            {(void**)&h->G3, d * K},
            {(void**)&h->C2, d * h->nchi},
            {(void**)&h->C3, d * h->nchi},
            {(void**)&h->sl_part, (size_t)SL_SPLIT_TILES * (SL_BM * SL_BM * 8 + sizeof(int))}};
  size_t need = 0;
  for (auto& a : al)
    if (!*a.p) need += a.n;
  size_t fr = 0, tot = 0;
  WL_CHECK(h, cudaMemGetInfo(&fr, &tot));
  const size_t late = wl_late_bytes(h);
  bool ok = need <= fr / 4 * 3 && need + late <= fr && !(h->budget && h->allocated + need + late > h->budget);
  if (h->sl_reserved) ok = need <= fr;  // (what the request allocates besides is in the same reservation)
  const bool had_trd = h->trd != nullptr;
  std::vector<void**> got;
  for (auto& a : al) {
    if (!ok) break;
    if (*a.p || a.n == 0) continue;
    if (wl_ensure(h, a.p, a.n, "digit rows") != COV_OK)
      ok = false;
    else
      got.push_back(a.p);
  }
  if (!ok) {
    for (auto p : got) {  // give back what the attempt took
      for (auto& a : al)
        if (a.p == p) h->allocated -= a.n;
      cudaFree(*p);
      *p = nullptr;
    }
    h->err.clear();
    state = -1;
    *use = false;
    return COV_OK;
  }
  if (tri && !had_trd) {
    k_sl_trd<<<(unsigned)((rows + 127) / 128), 128, 0, s>>>(rows, h->nleg, h->nt, h->nl, h->trd);
    WL_LAUNCH(h, "k_sl_trd");
  }
  state = 1;
  *use = true;
  return COV_OK;
}

// Lower part of rows [out.row0, row1) of the contraction (tri: the trispectrum table)
// into out: the first writer.  The caller resets the status word; what the launch reports is
// read by the next call that waits for the device (wl_snr_status).
int wl_sl_syrk(cov_handle* h, bool tri, int nssc, OutMap out, int64_t row1, cudaStream_t s) {
  const int64_t rows = tri ? h->ntrow : h->M;
  const int64_t nb = (rows + SL_BM - 1) / SL_BM, nk = sl_cols(h->nchi, h->nm, nssc > 0).nk;
  const int64_t t0 = out.row0 / SL_BM, t1 = (row1 + SL_BM - 1) / SL_BM;
  const int64_t ntiles = t1 * (t1 + 1) / 2 - t0 * (t0 + 1) / 2;
  if (ntiles <= 0) return COV_OK;
  CUtensorMap mi, mj;
  int rc;
  if ((rc = wl_status_words(h, s))) return rc;
  uint8_t* sl = tri ? h->Tsl : h->Asl;
  if ((rc = wl_sl_map(h, &mi, sl, nb * nk, SL_BM)) || (rc = wl_sl_map(h, &mj, sl, nb * nk, SL_BN))) return rc;
  const SlExp x = sl_exp(sl, nb, nk);
  // CTAs per tile: with one per SM, the parts (of at least 16 K blocks) that finish in
  // the fewest waves of K blocks
  const int64_t sms = wl_num_sms();
  int ns = 1;
  if (ntiles <= SL_SPLIT_TILES) {
    double best = 1e300;
    for (int c = 1; c <= 64 && (c == 1 || nk / c >= 16); ++c) {
      const int64_t waves = (ntiles * c + sms - 1) / sms;
      // a part costs its K blocks (~2.3 us each, ~0.6 of them read), its bound and, where parts are added, ~8 us for that
      const double t = (double)waves * (0.6 * (double)((nk + c - 1) / c) + 1.0 + (double)x.ng / 40.0 + (c > 1 ? 4.0 : 0.0));
      if (t < best) {
        best = t;
        ns = c;
      }
    }
  }
  SlArgs a{row1, t0, t1, (int)nk, ns, tri ? h->Texp : h->Aexp, x, out, h->tc_status,
           h->sl_report, h->sl_part, nullptr};
  a.ticket = (int*)(h->sl_part + (size_t)SL_SPLIT_TILES * SL_BM * SL_BM);
  if (ns > 1) {
    WL_CHECK(h, cudaMemsetAsync(h->sl_part, 0, (size_t)ntiles * SL_BM * SL_BM * 8, s));
    WL_CHECK(h, cudaMemsetAsync(a.ticket, 0, sizeof(int) * (size_t)ntiles, s));
  }
  static std::once_flag attr_once[WL_MAX_DEVICES];
  static int attr_rc[WL_MAX_DEVICES];
  constexpr int smem = SlShape<SL_NG>::kSmem;
  if (wl_once_per_device(attr_once, attr_rc, [] {
        int e = (int)cudaFuncSetAttribute(k_syrk_sl<SL_S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (!e) e = (int)cudaFuncSetAttribute(k_syrk_sl<SL_S + 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return e;
      }) != 0)
    return wl_fail(h, COV_ERR_CUDA, "cudaFuncSetAttribute(k_syrk_sl) failed");
  if (h->K < SL_FULL)
    k_syrk_sl<SL_S + 1><<<(unsigned)(ntiles * ns), SC_THREADS, smem, s>>>(mi, mj, a);
  else
    k_syrk_sl<SL_S><<<(unsigned)(ntiles * ns), SC_THREADS, smem, s>>>(mi, mj, a);
  WL_LAUNCH(h, "k_syrk_sl");
  return COV_OK;
}
