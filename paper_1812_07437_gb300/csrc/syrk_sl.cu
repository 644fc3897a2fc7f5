// FP64 form of the 1-halo (chi, M) contraction on the tcgen05 tensor cores
// (paper Eqs. CovPPNG, Ins5P, Ins6P as C_1h = A A^T with A the factor rows, the
// super-sample rows of Eq. WLSSCflatskyLimber as further columns, and the 1-halo
// trispectrum table of Eq. CovBB), by integer slicing in the manner of Ozaki,
// Ogita & Oishi (2012).  This part multiplies FP64 at ~1.2 TFLOP/s, BF16 at ~1900.
//
//   * Rows.  Every factor row is scaled by a power of two 2^-e that brings its
//     2-norm below sqrt(2) (k_sl_norm), rounded to x = X 2^-55 with an integer X,
//     and cut into the seven balanced base-256 digits of X: x = sum_t d_t 2^(-7-8t),
//     |d_0| <= 182, |d_t| <= 128, each exact in BF16 (k_sl_rows).
//   * Products.  d_t(i) d_u(j) and their sums over a K block of 32 at equal
//     t + u = g, g = 0..6, stay below 2^22: exact in the FP32 accumulators.  The 28
//     pairs t + u <= 6 are formed by 7 MMAs per K step instead of 28: the J digits
//     u = 0..6 of a group of 32 columns are stacked in shared memory, the accumulators
//     of the seven levels lie side by side in TMEM, and one MMA of digit t against the
//     first 32 (7 - t) stacked rows lands on the levels t..6 (N = 224, 192, ..., 32).
//     Small-N MMAs would read the 4 KB of the I digit from shared memory for 8 cycles
//     of work each.
//   * Recombination.  The level sums of a K block are added exactly to one 64-bit
//     integer per element, sum_g a_g 2^(8 (6 - g)), modulo 2^64.  By Cauchy-Schwarz the
//     complete sum is below 2^63 (that is what the norm scaling is for), so partial
//     sums may wrap and need no second word.  One rounding to FP64 at the end.
// What is dropped (levels above 6, digits beyond 2^-55 of the norm) is ~1e-15 of
// sqrt(C_aa C_bb); against extended precision on the paper's and the 5-bin rows the
// error is 0.8-1.4e-15 in the 2-norm where the FP64 FMA chain of k_gemm_lower, one
// rounding per term, has 4.3-8.0e-15 (largest normalised element 0.7-0.9e-14 against
// 1.2-1.3e-14).
//
// Bound: the tensor pipe and, close behind, L2 (a 128 x 128 tile reads 112 KB per K
// block of 32, 32 bytes per clock and SM at the full MMA rate).  M = 6375, K = 12288 +
// 128: contraction 10.7 ms = 1.36 PFLOP/s issued (48 TFLOP/s FP64) where k_gemm_lower
// took 415 + 4.4 ms (1.2 TFLOP/s); trispectrum table 37 -> 1.0 ms, rows 0.55 ms; whole
// FP64 assembly 464 -> 12.6 ms.  M = 818 (28 tiles, 11 K parts each): 27.2 -> 0.65 ms.
#include <cuda_bf16.h>

#include "common.cuh"

#define SL_S 7
#define SL_BM 128                                   // tile rows, and tile columns
#define SL_BK 32                                    // K block
#define SL_BN 32                                    // columns per accumulator group
#define SL_NG (SL_BM / SL_BN)
#define SL_DIGIT (SL_BM * SL_BK * 2)                // 8 KB: one digit of 128 rows x 32 K
#define SL_BLOCK (SL_S * SL_DIGIT)                  // 56 KB: one (row block, K block)
#define SL_GROUP (SL_S * SL_BN * SL_BK * 2)         // 14 KB: the digits of 32 rows
#define SL_STAGE (SL_BLOCK + SL_NG * SL_GROUP)      // 112 KB
#define SL_STAGES 2
#define SL_SMEM (SL_STAGES * SL_STAGE + 1024)
#define SL_EPI 8                                    // epilogue warps: two per TMEM lane quarter, 16 columns each
#define SL_THREADS (64 + 32 * SL_EPI)
#define SL_SPIN (1u << 22)
#define SL_MAGIC 0x4B400000u                        // bits of 1.5 2^23: f + 1.5 2^23 holds the integer f in its low bits
#define SL_SPLIT_TILES 304                          // largest tile count whose K range is cut over several CTAs

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

// sum over q of the squared factor, one warp per (signature, node)
__global__ void __launch_bounds__(256) k_sl_norm2(SlSig g, int nsig, const int32_t* __restrict__ tris, double* s2) {
  const int id = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (id >= nsig * g.nchi) return;
  const int s = id / g.nchi, n = id % g.nchi;
  int a = s, b = s, c = s, isB = 0;
  if (g.pairs) {
    a = 0;
    int r = s;
    while (r >= g.nl - a) {
      r -= g.nl - a;
      ++a;
    }
    b = c = a + r;
  } else if (s >= g.nl) {
    const int32_t* t = tris + 3 * (s - g.nl);
    a = t[0];
    b = t[1];
    c = t[2];
    isB = 1;
  }
  double acc = 0.0;
  for (int q = lane; q < g.nm; q += 32) {
    const double v = sl_factor(g, isB, a, b, c, n, (int64_t)n * g.nm + q);
    acc = fma(v, v, acc);
  }
  acc = warp_sum(acc);
  if (lane == 0) s2[id] = acc;
}

struct SlSsc {
  int nssc;  // super-sample columns (N_chi or 0)
  const double *wchi, *sigw2, *chi, *RP3, *RB3;
};

// One warp per row: its lensing weight and super-sample entry at every node, scaled by
// the row's power of two (exponent in rexp).
__global__ void __launch_bounds__(256) k_sl_norm(SlSig g, int64_t rows, const int32_t* __restrict__ rd,
                                                 const double* __restrict__ W, double wscale,
                                                 const double* __restrict__ s2, SlSsc ss, double* wrow, double* srow,
                                                 int* rexp) {
  const int64_t a = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (a >= rows) return;
  const int32_t* r = rd + 8 * a;
  const bool isB = r[0] != 0;
  const int nchi = g.nchi;
  const double *W1 = W + r[4] * nchi, *W2 = W + r[5] * nchi, *W3 = W + (isB ? r[6] : r[4]) * nchi;
  const double* sq = s2 + (size_t)sl_sig(g, r) * nchi;
  double* wo = wrow + a * nchi;
  double* so = srow + a * nchi;
  double acc = 0.0;
  for (int n = lane; n < nchi; n += 32) {
    double w = W1[n] * W2[n];
    if (isB) w *= W3[n];
    if (ss.nssc) {
      const double c2 = ss.chi[n] * ss.chi[n], t = sqrt(ss.wchi[n] * ss.sigw2[n]) * w;
      const double v = isB ? t / (c2 * c2) * ss.RB3[r[7] * nchi + n] : t / c2 * ss.RP3[r[1] * nchi + n];
      so[n] = v;
      acc = fma(v, v, acc);
    }
    w *= wscale;
    wo[n] = w;
    acc = fma(w * w, sq[n], acc);
  }
  acc = warp_sum(acc);
  int e = 0;
  if (acc > 0.0) frexp(sqrt(acc) * (0.70710678118654752440 * (1.0 + 1e-9)), &e);
  const double sc = ldexp(1.0, -e);
  for (int n = lane; n < nchi; n += 32) {
    wo[n] *= sc;
    if (ss.nssc) so[n] *= sc;
  }
  if (lane == 0) rexp[a] = e;
}

// X = RN(x 2^55) (ties to even) for |x| < 2, by integer operations on the bits of x
__device__ __forceinline__ long long sl_int(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FFu);
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);  // (subnormals round to 0 either way)
  const int sh = 1020 - E;  // X = RN(m / 2^sh); sh >= -3
  unsigned long long q;
  if (sh <= 0) {
    q = m << -sh;
  } else if (sh >= 64) {
    q = 0;
  } else {
    q = m >> sh;
    const unsigned long long rem = m & ((1ull << sh) - 1), half = 1ull << (sh - 1);
    q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;
  }
  return (b >> 63) ? -(long long)q : (long long)q;
}

// Digits of 128 rows x 32 K, one contiguous 56 KB block per (row block, K block):
// [digit][row][k].  The factor of each signature present among the rows is formed
// once in shared memory; an entry is then one FP64 product (the bound here beside the
// 14 bytes written per entry: 5-bin rows, 7.9e7 entries).  A thread holds 8
// consecutive k of one row and stores each digit's 16 bytes at once.
#define SR_THREADS 256
__global__ void __launch_bounds__(SR_THREADS)
    k_sl_rows(SlSig g, int64_t rows, int nssc, int nk, const int32_t* __restrict__ rd,
              const double* __restrict__ wrow, const double* __restrict__ srow, uint8_t* __restrict__ out) {
  __shared__ double F[SL_BM][SL_BK + 1];
  __shared__ int slot[SL_BM];
  __shared__ int first[SL_BM];  // a row of each signature slot
  __shared__ int nslot_sh[SL_BM / 32];
  const int64_t rb = blockIdx.y, kb = blockIdx.x, r0 = rb * SL_BM;
  const int64_t K = (int64_t)g.nchi * g.nm, k0 = kb * SL_BK;
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
  for (int e = tid; e < nslot * SL_BK; e += SR_THREADS) {
    const int s = e / SL_BK, k = e % SL_BK;
    const int64_t kk = k0 + k;
    if (kk < K) {
      const int32_t* r = rd + 8 * (r0 + first[s]);
      F[s][k] = sl_factor(g, r[0] != 0, r[1], r[2], r[3], (int)(kk / g.nm), kk);
    }
  }
  __syncthreads();
  uint8_t* o = out + ((size_t)rb * nk + kb) * SL_BLOCK;
  for (int e = tid; e < SL_BM * (SL_BK / 8); e += SR_THREADS) {
    const int row = e >> 2, k8 = (e & 3) * 8;
    const int64_t r = r0 + row;
    const double* wr = wrow + r * g.nchi;
    const double* sr = srow + r * g.nchi;
    uint32_t d[SL_S][4];
    int n = (int)((k0 + k8) / g.nm), q = (int)((k0 + k8) % g.nm);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      unsigned long long y[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t kk = k0 + k8 + 2 * p + h;
        double v = 0.0;
        if (r < rows) {
          if (kk < K)
            v = F[slot[row]][k8 + 2 * p + h] * wr[n];
          else if (kk < K + nssc)
            v = sr[kk - K];
        }
        if (++q == g.nm) {
          q = 0;
          ++n;
        }
        // balanced digits d_t = byte_t(X + 128 sum_t 256^t) - 128
        y[h] = (unsigned long long)sl_int(v) + 0x0080808080808080ull;
      }
#pragma unroll
      for (int t = 0; t < SL_S; ++t) {
        float f[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // the top digit keeps its sign and ninth bit
          const int by = t == 0 ? (int)((long long)y[h] >> 48) : (int)((y[h] >> (8 * (SL_S - 1 - t))) & 255u);
          f[h] = __int_as_float(SL_MAGIC + by) - (12582912.0f + 128.0f);
        }
        // |d| <= 256 has at most 8 significant bits: the upper half of the FP32 value is its BF16 form
        d[t][p] = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632);
      }
    }
#pragma unroll
    for (int t = 0; t < SL_S; ++t)
      *(uint4*)(o + (size_t)t * SL_DIGIT + row * (SL_BK * 2) + k8 * 2) = make_uint4(d[t][0], d[t][1], d[t][2], d[t][3]);
  }
}

// ---------------------------------------------------------------- contraction
__device__ __forceinline__ uint32_t sl_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void sl_init(uint64_t* bar, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sl_u32(bar)), "r"(n) : "memory");
}
__device__ __forceinline__ void sl_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sl_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void sl_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sl_u32(bar)) : "memory");
}
__device__ __forceinline__ void sl_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sl_u32(bar))
               : "memory");
}
__device__ __forceinline__ uint32_t sl_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(sl_u32(bar)), "r"(parity)
      : "memory");
  return ok;
}
// bounded wait that also gives up once any CTA has raised the status word
__device__ __forceinline__ bool sl_wait(uint64_t* bar, uint32_t parity, int* status) {
  for (uint32_t i = 0; i < SL_SPIN; ++i) {
    if (sl_try(bar, parity)) return true;
    if ((i & 1023u) == 1023u && *(volatile int*)status) return false;
  }
  atomicExch(status, 1);
  return false;
}
__device__ __forceinline__ void sl_tma(const CUtensorMap* map, uint64_t* bar, void* dst, int row, int blk) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
      "[%2];" ::"r"(sl_u32(dst)),
      "l"((uint64_t)map), "r"(sl_u32(bar)), "r"(0), "r"(row), "r"(0), "r"(blk)
      : "memory");
}
__device__ __forceinline__ void sl_prefetch(const CUtensorMap* map, int row, int blk) {
  asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"((uint64_t)map), "r"(0),
               "r"(row), "r"(0), "r"(blk)
               : "memory");
}
__device__ __forceinline__ uint64_t sl_desc(uint32_t saddr) {  // K-major, 64-byte rows, SWIZZLE_64B
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;  // 8 rows x 64 B
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}
__device__ __forceinline__ void sl_tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}

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

struct SlArgs {
  int64_t rows, row1, t0, t1;
  int nk, ns;                 // K blocks; CTAs that share a tile's K range
  const int* rexp;
  OutMap out;
  int* status;
  unsigned long long* part;   // [tile][column][row] exact partial sums (ns > 1), zero at launch
  int* ticket;                // [tile] CTAs that have delivered (ns > 1), zero at launch
};

// One CTA per (128 x 128 lower tile, K range).  Warp 0 loads (TMA, two stages of a K
// block: the I block in one box, the J block as four groups of 32 rows), warp 1 issues
// the MMAs of the four column groups in turn into two accumulator sets (7 x 32
// columns each), eight warps recombine the set of the group before: 14 integer and
// FP32 operations per element and K block, in registers (64 64-bit sums per thread).
// The exact FP32 integers become integers by adding 1.5 2^23 (full rate; the
// conversion instruction is not); the biases this leaves are removed once at the end.
// Where a launch has too few tiles for the SMs, ns CTAs take parts of a tile's K
// range, add their 64-bit sums atomically (integers: any order gives the same value)
// and the last one converts.
__global__ void __launch_bounds__(SL_THREADS, 1)
    k_syrk_sl(const __grid_constant__ CUtensorMap map_i, const __grid_constant__ CUtensorMap map_j, SlArgs A) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[SL_STAGES], empty[SL_STAGES], tfull[2], tempty[2], mma_done;
  __shared__ uint32_t tmem_sh;
  __shared__ int last_sh;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tile = blockIdx.x / A.ns;
  const int sp = (int)(blockIdx.x % A.ns);
  const int kb0 = (int)((int64_t)A.nk * sp / A.ns), kb1 = (int)((int64_t)A.nk * (sp + 1) / A.ns);
  int64_t ti, tj;
  sl_tile(tile, A.t0, A.t1, &ti, &tj);
  if (threadIdx.x == 0) {
    for (int s = 0; s < SL_STAGES; ++s) {
      sl_init(&full[s], 1);
      sl_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      sl_init(&tfull[b], 1);
      sl_init(&tempty[b], SL_EPI);
    }
    sl_init(&mma_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sl_u32(&tmem_sh)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_sh;
  const int q = warp & 3, half = (warp - 2) >> 2;  // epilogue warp: TMEM lanes 32 q .., columns 16 half .. of a group
  const int row = q * 32 + lane;
  const unsigned long long bias = ((unsigned long long)SL_MAGIC << 48) + ((257ull * SL_MAGIC) << 32) +
                                  ((257ull * SL_MAGIC & 0xFFFFFFFFull) << 16) + (257ull * SL_MAGIC & 0xFFFFFFFFull);

  if (warp == 0 && lane == 0) {
    for (int kb = kb0; kb < kb1; ++kb) {
      const int w = kb - kb0, s = w % SL_STAGES;
      if (!sl_wait(&empty[s], (uint32_t)((w / SL_STAGES) & 1) ^ 1u, A.status)) break;
      uint8_t* st = smem + (size_t)s * SL_STAGE;
      const int bi = (int)(ti * A.nk + kb), bj = (int)(tj * A.nk + kb);
      sl_expect(&full[s], SL_STAGE);
      sl_tma(&map_i, &full[s], st, 0, bi);
      for (int j = 0; j < SL_NG; ++j) sl_tma(&map_j, &full[s], st + SL_BLOCK + j * SL_GROUP, j * SL_BN, bj);
      if (kb + 2 < kb1) {
        sl_prefetch(&map_i, 0, bi + 2);
        if (ti != tj) sl_prefetch(&map_i, 0, bj + 2);
      }
    }
  } else if (warp == 1 && lane == 0) {
    for (int kb = kb0; kb < kb1; ++kb) {
      const int w = kb - kb0, s = w % SL_STAGES;
      if (!sl_wait(&full[s], (uint32_t)((w / SL_STAGES) & 1), A.status)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t base_i = sl_u32(smem + (size_t)s * SL_STAGE);
      bool ok = true;
#pragma unroll 1
      for (int j = 0; j < SL_NG && ok; ++j) {
        const int b = j & 1, use = 2 * w + (j >> 1);  // use-th filling of accumulator set b
        ok = sl_wait(&tempty[b], (uint32_t)(use & 1) ^ 1u, A.status);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t base_j = base_i + SL_BLOCK + j * SL_GROUP, dt = tmem + (uint32_t)(b * 256);
#pragma unroll
        for (int k = 0; k < SL_BK / 16; ++k)
#pragma unroll
          for (int t = 0; t < SL_S; ++t) {
            // BF16 x BF16 -> FP32, K-major, M = 128, N = 32 (7 - t): digit t against the digits 0 .. 6 - t
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                   ((uint32_t)((SL_BN * (SL_S - t)) >> 3) << 17) | ((uint32_t)(SL_BM >> 4) << 24);
            const uint32_t acc = (k == 0 && t == 0) ? 0u : 1u;
            asm volatile(
                "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, "
                "p;\n}\n" ::"r"(dt + (uint32_t)(t * SL_BN)),
                "l"(sl_desc(base_i + t * SL_DIGIT + k * 32)), "l"(sl_desc(base_j + k * 32)), "r"(idesc), "r"(acc)
                : "memory");
          }
        sl_commit(&tfull[b]);
      }
      if (!ok) break;
      sl_commit(&empty[s]);
    }
    // every MMA of this CTA has completed before its TMEM is released
    sl_commit(&mma_done);
    for (uint32_t i = 0; i < SL_SPIN && !sl_try(&mma_done, 0u); ++i) {
    }
  } else if (warp >= 2) {
    unsigned long long acc[SL_NG][16];
#pragma unroll
    for (int j = 0; j < SL_NG; ++j)
#pragma unroll
      for (int c = 0; c < 16; ++c) acc[j][c] = 0ull;
    int ok = 1;
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 16);
    for (int kb = kb0; kb < kb1 && ok; ++kb) {
#pragma unroll
      for (int j = 0; j < SL_NG; ++j) {
        if (ok) {  // (warp-uniform: the TMEM loads are warp-collective)
          const int b = j & 1;
          if (lane == 0) ok = sl_wait(&tfull[b], (uint32_t)(j >> 1), A.status);
          ok = __shfl_sync(0xffffffffu, ok, 0);
          __syncwarp();
        }
        if (ok) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t r[SL_S][8];
#pragma unroll
            for (int g = 0; g < SL_S; ++g) sl_tmem_ld8(tbase + (uint32_t)((j & 1) * 256 + g * SL_BN + h * 8), r[g]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int g = 0; g < SL_S; ++g)
#pragma unroll
              for (int c = 0; c < 8; ++c) asm volatile("" : "+r"(r[g][c]));
            if (h == 1) {  // the set's values are in registers
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0) sl_arrive(&tempty[j & 1]);
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              uint32_t v[SL_S];
#pragma unroll
              for (int g = 0; g < SL_S; ++g) v[g] = __float_as_uint(__uint_as_float(r[g][c]) + 12582912.0f);
              // a_0 2^48 + (a_1 2^8 + a_2) 2^32 + (a_3 2^8 + a_4) 2^16 + (a_5 2^8 + a_6), biased
              unsigned long long x = acc[j][h * 8 + c];
              x += (unsigned long long)(v[3] * 256u + v[4]) * 65536ull;
              x += (unsigned long long)(v[5] * 256u + v[6]);
              x += (unsigned long long)(v[0] * 65536u + v[1] * 256u + v[2]) << 32;
              acc[j][h * 8 + c] = x;
            }
          }
        }
      }
    }
    if (ok && *(volatile int*)A.status == 0) {
      if (A.ns == 1) {
        const unsigned long long off = bias * (unsigned long long)(kb1 - kb0);
        const int64_t gr = ti * SL_BM + row;
        if (gr < A.row1) {
          const int er = A.rexp[gr] - 62;
          double* p = A.out.at(gr, tj * SL_BM);
#pragma unroll
          for (int j = 0; j < SL_NG; ++j)
#pragma unroll
            for (int c = 0; c < 16; ++c) {
              const int lc = j * SL_BN + half * 16 + c;
              const int64_t gc = tj * SL_BM + lc;
              if (gc <= gr) p[lc] = scaled_to_double_rn((long long)(acc[j][c] - off), er + __ldg(A.rexp + gc));
            }
        }
      } else {
        unsigned long long* p = A.part + (size_t)tile * (SL_BM * SL_BM) + row;
#pragma unroll
        for (int j = 0; j < SL_NG; ++j)
#pragma unroll
          for (int c = 0; c < 16; ++c)
            atomicAdd(p + (size_t)(j * SL_BN + half * 16 + c) * SL_BM, acc[j][c]);
      }
    }
  }
  __syncwarp();
  // after an expired wait some copies may still be in flight: a bounded
  // pause (~1 ms) lets them land before the CTA's shared memory is released
  if (warp == 0 && lane == 0 && *(volatile int*)A.status != 0)
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (A.ns > 1) __threadfence();
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  if (A.ns > 1) {
    if (threadIdx.x == 0) last_sh = atomicAdd(A.ticket + tile, 1) == A.ns - 1;
    __syncthreads();
    if (last_sh && *(volatile int*)A.status == 0) {
      __threadfence();
      const unsigned long long off = bias * (unsigned long long)A.nk;
      const unsigned long long* p = A.part + (size_t)tile * (SL_BM * SL_BM);
      for (int e = threadIdx.x; e < SL_BM * SL_BM; e += SL_THREADS) {
        const int lr = e & (SL_BM - 1), lc = e >> 7;
        const int64_t gr = ti * SL_BM + lr, gc = tj * SL_BM + lc;
        if (gr < A.row1 && gc <= gr)
          *A.out.at(gr, gc) = scaled_to_double_rn((long long)(__ldcg(p + e) - off), A.rexp[gr] + A.rexp[gc] - 62);
      }
    }
  }
}

// ---------------------------------------------------------------- host side
static inline int64_t sl_nk(int64_t k) { return (k + SL_BK - 1) / SL_BK; }

// bytes of the digits of `rows` rows of k entries
size_t wl_sl_bytes(int64_t rows, int64_t k) {
  return (size_t)((rows + SL_BM - 1) / SL_BM) * (size_t)sl_nk(k) * SL_BLOCK;
}

// upper bound of what wl_sl_alloc takes beside the digits themselves
size_t wl_sl_fixed_bytes(const cov_handle* h) {
  const size_t M = (size_t)h->M, T = (size_t)h->ntrow, nchi = (size_t)h->nchi;
  const size_t nsig = (size_t)std::max(h->nl + h->ntri, h->nl * (h->nl + 1) / 2);
  return 8 * nsig * nchi + 8 * (std::max(M, T) + M) * nchi + 4 * M + 36 * T + 16 * ((size_t)h->K + nchi) +
         (size_t)SL_SPLIT_TILES * (SL_BM * SL_BM * 8 + sizeof(int));
}

static int sl_map(cov_handle* h, CUtensorMap* map, void* base, int64_t blocks, int box_rows) {
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
// trispectrum rows (tri).  The buffers exist already (wl_sl_rows_alloc).
int wl_sl_rows(cov_handle* h, bool tri, int nssc, cudaStream_t s) {
  SlSig g{h->nl, h->nchi, h->nm, tri ? 1 : 0, h->U, h->G2, h->G3, h->C2, h->C3};
  const int nsig = tri ? h->nl * (h->nl + 1) / 2 : h->nl + h->ntri;
  const int64_t rows = tri ? h->ntrow : h->M;
  const int32_t* rd = tri ? h->trd : h->rowdesc_d;
  const int nk = (int)sl_nk((int64_t)h->K + nssc);
  int* rexp = tri ? h->Texp : h->Aexp;
  k_rows_prep<<<(h->K + 255) / 256, 256, 0, s>>>(h->nchi, h->nm, 1.0 / h->omega, h->cosmo_d, h->chi, h->wchi, h->m,
                                                 h->om, h->f, h->G2, h->G3, h->C2, h->C3);
  k_sl_norm2<<<(nsig * h->nchi + 7) / 8, 256, 0, s>>>(g, nsig, h->tris_d, h->sl_s2);
  SlSsc ss{nssc, h->wchi, h->sigw2, h->chi, h->RP3, h->RB3};
  k_sl_norm<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(g, rows, rd, h->W, tri ? sqrt(h->omega) : 1.0, h->sl_s2, ss,
                                                       h->sl_w, h->sl_sr, rexp);
  k_sl_rows<<<dim3((unsigned)nk, (unsigned)((rows + SL_BM - 1) / SL_BM)), SR_THREADS, 0, s>>>(
      g, rows, nssc, nk, rd, h->sl_w, h->sl_sr, tri ? h->Tsl : h->Asl);
  WL_LAUNCH(h, "digit row kernels");
  return COV_OK;
}

// Whether the tensor-core FP64 form serves the handle's rows (tri: its trispectrum
// rows), and its buffers.  The digits take 14 bytes per entry where the FP64 rows of
// k_gemm_lower take 8; where they do not fit (hbm_budget, or three quarters of the
// free memory) the FP64 rows and that kernel serve the handle as before.  Decided
// once per handle: a later call with more super-sample columns finds room for them.
int wl_sl_alloc(cov_handle* h, bool tri, bool* use, cudaStream_t s) {
  int& state = tri ? h->sl_tri : h->sl_rows;
  if (state) {
    *use = state > 0;
    return COV_OK;
  }
  const int64_t rows = tri ? h->ntrow : h->M;
  const size_t d = sizeof(double), K = (size_t)h->K;
  const size_t nsig = (size_t)std::max(h->nl + h->ntri, h->nl * (h->nl + 1) / 2);
  const size_t wmax = (size_t)std::max<int64_t>(h->M, h->ntrow) * h->nchi;
  struct {
    void** p;
    size_t n;
  } al[] = {{(void**)(tri ? &h->Tsl : &h->Asl), wl_sl_bytes(rows, (int64_t)K + (tri ? 0 : h->nchi))},
            {(void**)(tri ? &h->Texp : &h->Aexp), sizeof(int) * (size_t)rows},
            {(void**)&h->trd, tri ? sizeof(int32_t) * 8 * (size_t)rows : 0},
            {(void**)&h->sl_s2, d * nsig * h->nchi},
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
  bool ok = need <= fr / 4 * 3 && !(h->budget && h->allocated + need > h->budget);
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
// into out: the first writer.  The status word is reset and checked by the caller.
int wl_sl_syrk(cov_handle* h, bool tri, int nssc, OutMap out, int64_t row1, cudaStream_t s) {
  const int64_t rows = tri ? h->ntrow : h->M;
  const int64_t nb = (rows + SL_BM - 1) / SL_BM, nk = sl_nk((int64_t)h->K + nssc);
  const int64_t t0 = out.row0 / SL_BM, t1 = (row1 + SL_BM - 1) / SL_BM;
  const int64_t ntiles = t1 * (t1 + 1) / 2 - t0 * (t0 + 1) / 2;
  if (ntiles <= 0) return COV_OK;
  CUtensorMap mi, mj;
  int rc;
  uint8_t* sl = tri ? h->Tsl : h->Asl;
  if ((rc = sl_map(h, &mi, sl, nb * nk, SL_BM)) || (rc = sl_map(h, &mj, sl, nb * nk, SL_BN))) return rc;
  // CTAs per tile: with one per SM, the parts (of at least 16 K blocks) that finish in
  // the fewest waves of K blocks
  const int64_t sms = wl_num_sms();
  int ns = 1;
  if (ntiles <= SL_SPLIT_TILES) {
    double best = 1e300;
    for (int c = 1; c <= 64 && (c == 1 || nk / c >= 16); ++c) {
      const int64_t waves = (ntiles * c + sms - 1) / sms;
      // a part costs its K blocks (~2.3 us each) and, where parts are added, about 8 us for that
      const double t = (double)waves * ((double)((nk + c - 1) / c) + (c > 1 ? 4.0 : 0.0));
      if (t < best) {
        best = t;
        ns = c;
      }
    }
  }
  SlArgs a{rows, row1, t0, t1, (int)nk, ns, tri ? h->Texp : h->Aexp, out, h->tc_status, h->sl_part, nullptr};
  a.ticket = (int*)(h->sl_part + (size_t)SL_SPLIT_TILES * SL_BM * SL_BM);
  if (ns > 1) {
    WL_CHECK(h, cudaMemsetAsync(h->sl_part, 0, (size_t)ntiles * SL_BM * SL_BM * 8, s));
    WL_CHECK(h, cudaMemsetAsync(a.ticket, 0, sizeof(int) * (size_t)ntiles, s));
  }
  static std::once_flag attr_once[WL_MAX_DEVICES];
  static int attr_rc[WL_MAX_DEVICES];
  if (wl_once_per_device(attr_once, attr_rc, [] {
        return (int)cudaFuncSetAttribute(k_syrk_sl, cudaFuncAttributeMaxDynamicSharedMemorySize, SL_SMEM);
      }) != 0)
    return wl_fail(h, COV_ERR_CUDA, "cudaFuncSetAttribute(k_syrk_sl) failed");
  k_syrk_sl<<<(unsigned)(ntiles * ns), SL_THREADS, SL_SMEM, s>>>(mi, mj, a);
  WL_LAUNCH(h, "k_syrk_sl");
  return COV_OK;
}
