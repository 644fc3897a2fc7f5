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
//   * Products and recombination as described in digits.cuh, modulo 2^64.  By
//     Cauchy-Schwarz the complete sum is below 2^63 (that is what the norm scaling is
//     for), so partial sums may wrap and need no second word.  One rounding to FP64 at
//     the end.
// What is dropped (levels above 6, digits beyond 2^-55 of the norm) is ~1e-15 of
// sqrt(C_aa C_bb); against extended precision on the paper's and the 5-bin rows the
// error is 0.8-1.4e-15 in the 2-norm where the FP64 FMA chain of k_gemm_lower, one
// rounding per term, has 4.3-8.0e-15 (largest normalised element 0.7-0.9e-14 against
// 1.2-1.3e-14).
//
// Bound: the tensor pipe and, close behind, L2 (a 128 x 128 tile reads 112 KB per K
// block of 32, 32 bytes per clock and SM at the full MMA rate).  M = 6375, K = 12288 +
// 128: contraction 10.0 ms = 1.45 PFLOP/s issued (51 TFLOP/s FP64) where k_gemm_lower
// took 415 + 4.4 ms (1.2 TFLOP/s); trispectrum table 37 -> 1.0 ms, rows 0.55 ms; whole
// FP64 assembly 464 -> 11.8 ms.  M = 818 (28 tiles, 11 K parts each): 27.1 -> 0.63 ms.
#include "digits.cuh"

#define SL_NG 4               // a tile is 128 x 128
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

// Exponent of a row that is not finite (an FP64 row's is below 1100 in magnitude): all
// elements of its row and column are NaN.
#define SL_BAD (1 << 20)
__device__ __forceinline__ double sl_value(unsigned long long sum, int ei, int ej) {
  const int e = ei + ej - 62;
  return e > SL_BAD / 2 ? __longlong_as_double(0x7FF8000000000000ll) : scaled_to_double_rn((long long)sum, e);
}

// One warp per row: its lensing weight and super-sample entry at every node, scaled by
// the row's power of two (exponent in rexp; SL_BAD where the row holds an infinity or NaN
// or its norm overflows).
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
  const bool bad = !isfinite(acc);
  int e = 0;
  if (!bad && acc > 0.0) frexp(sqrt(acc) * (0.70710678118654752440 * (1.0 + 1e-9)), &e);
  const double sc = bad ? 0.0 : ldexp(1.0, -e);  // (NaN and infinity stay what they are or become NaN: digits of 0)
  for (int n = lane; n < nchi; n += 32) {
    wo[n] *= sc;
    if (ss.nssc) so[n] *= sc;
  }
  if (lane == 0) rexp[a] = bad ? SL_BAD : e;
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
    long long X[8];
    uint4 d[SL_S];
    int n = (int)((k0 + k8) / g.nm), q = (int)((k0 + k8) % g.nm);
#pragma unroll
    for (int p = 0; p < 8; ++p) {
      const int64_t kk = k0 + k8 + p;
      double v = 0.0;
      if (r < rows) {
        if (kk < K)
          v = F[slot[row]][k8 + p] * wr[n];
        else if (kk < K + nssc)
          v = sr[kk - K];
      }
      if (++q == g.nm) {
        q = 0;
        ++n;
      }
      X[p] = sl_int(v);
    }
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

struct SlArgs {
  int64_t rows, row1, t0, t1;
  int nk, ns;                 // K blocks; CTAs that share a tile's K range
  const int* rexp;
  OutMap out;
  int *status, *report;       // an expired wait of this assembly; of any since the host last read it
  unsigned long long* part;   // [tile][column][row] exact partial sums (ns > 1), zero at launch
  int* ticket;                // [tile] CTAs that have delivered (ns > 1), 2^16 for each that gave up, zero at launch
};

// One CTA per (128 x 128 lower tile, K range).  Warp 0 loads (TMA, two stages of a K
// block: the I block in one box, the J block as four groups of 32 rows), warp 1 issues
// the MMAs of the four column groups in turn into two accumulator sets (7 x 32
// columns each), eight warps recombine the set of the group before in registers (64
// 64-bit sums per thread).  Where a launch has too few tiles for the SMs, ns CTAs take
// parts of a tile's K range, add their 64-bit sums atomically (integers: any order
// gives the same value) and the last one converts.  The host does not wait for this kernel:
// where a wait expires, the elements that it leaves incomplete are stored as NaN.
__global__ void __launch_bounds__(SL_THREADS, 1)
    k_syrk_sl(const __grid_constant__ CUtensorMap map_i, const __grid_constant__ CUtensorMap map_j, SlArgs A) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) SlBars bars;
  __shared__ uint32_t tmem_sh;
  __shared__ int last_sh, gave_up;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tile = blockIdx.x / A.ns;
  const int sp = (int)(blockIdx.x % A.ns);
  const int kb0 = (int)((int64_t)A.nk * sp / A.ns), kb1 = (int)((int64_t)A.nk * (sp + 1) / A.ns);
  int64_t ti, tj;
  sl_tile(tile, A.t0, A.t1, &ti, &tj);
  if (threadIdx.x == 0) {
    sl_bars_init(&bars);
    gave_up = 0;
  }
  if (warp == 0) sl_tmem_alloc(&tmem_sh);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_sh;
  const int q = warp & 3, half = (warp - 2) >> 2;  // epilogue warp: TMEM lanes 32 q .., columns 16 half .. of a group

  if (warp == 0 && lane == 0) {
    int it = 0;
    sl_produce<SL_NG>(&map_i, &map_j, smem, &bars, (int)(ti * A.nk) + kb0, (int)(tj * A.nk) + kb0, 0, kb1 - kb0, it, A.status);
  } else if (warp == 1) {
    int it = 0;
    sl_issue<SL_NG, false>(smem, &bars, kb1 - kb0, it, A.status);
    sl_issue_end(&bars, lane);
  } else if (warp >= 2) {
    unsigned long long acc[SL_NG][16];
#pragma unroll
    for (int j = 0; j < SL_NG; ++j)
#pragma unroll
      for (int c = 0; c < 16; ++c) acc[j][c] = 0ull;
    int it = 0;
    sl_drain_init<false>(&bars, tmem, q, half, lane);
    const bool ok = sl_drain<SL_NG, false>(acc, &bars, tmem, q, half, lane, kb1 - kb0, it, A.status);
    if (!ok) gave_up = 1;
    if (A.ns == 1) {
      const unsigned long long off = SL_BIAS * (unsigned long long)(kb1 - kb0);
      const int64_t gr = ti * SL_BM + sl_row<false>(q, lane, 0);
      if (gr < A.row1) {
        const int er = ok ? A.rexp[gr] : SL_BAD;
        double* p = A.out.at(gr, tj * SL_BM);
#pragma unroll
        for (int j = 0; j < SL_NG; ++j)
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const int lc = sl_col<false>(half, lane, j, c);
            const int64_t gc = tj * SL_BM + lc;
            if (gc <= gr) p[lc] = sl_value(acc[j][c] - off, er, __ldg(A.rexp + gc));
          }
      }
    } else if (ok) {
      unsigned long long* p = A.part + (size_t)tile * (SL_BM * SL_BM);
#pragma unroll
      for (int j = 0; j < SL_NG; ++j)
#pragma unroll
        for (int c = 0; c < 16; ++c)
          atomicAdd(p + (size_t)sl_col<false>(half, lane, j, c) * SL_BM + sl_row<false>(q, lane, c), acc[j][c]);
    }
  }
  __syncwarp();
  if (warp == 0 && lane == 0) sl_pause(A.status);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (A.ns > 1) __threadfence();
  __syncthreads();
  if (warp == 0) sl_tmem_free(tmem);
  if (threadIdx.x == 0 && *(volatile int*)A.status != 0) atomicExch(A.report, 1);
  if (A.ns > 1) {
    if (threadIdx.x == 0) {  // 1: the last CTA of the tile, 2: and one of them gave up
      const int add = gave_up ? 65537 : 1, t = atomicAdd(A.ticket + tile, add) + add;
      last_sh = (t & 65535) != A.ns ? 0 : t > 65535 ? 2 : 1;
    }
    __syncthreads();
    if (last_sh) {
      __threadfence();
      const unsigned long long off = SL_BIAS * (unsigned long long)A.nk;
      const unsigned long long* p = A.part + (size_t)tile * (SL_BM * SL_BM);
      for (int e = threadIdx.x; e < SL_BM * SL_BM; e += SL_THREADS) {
        const int lr = e & (SL_BM - 1), lc = e >> 7;
        const int64_t gr = ti * SL_BM + lr, gc = tj * SL_BM + lc;
        if (gr < A.row1 && gc <= gr)
          *A.out.at(gr, gc) = sl_value(__ldcg(p + e) - off, last_sh == 2 ? SL_BAD : A.rexp[gr], A.rexp[gc]);
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
// k_gemm_lower take 8; where they do not fit (in hbm_budget, or the free memory, beside
// all that the handle's other calls may still allocate) the FP64 rows and that kernel
// serve the handle as before.  Decided
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
  const size_t late = wl_late_bytes(h);
  bool ok = need <= fr / 4 * 3 && need + late <= fr && !(h->budget && h->allocated + need + late > h->budget);
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
  const int64_t nb = (rows + SL_BM - 1) / SL_BM, nk = sl_nk((int64_t)h->K + nssc);
  const int64_t t0 = out.row0 / SL_BM, t1 = (row1 + SL_BM - 1) / SL_BM;
  const int64_t ntiles = t1 * (t1 + 1) / 2 - t0 * (t0 + 1) / 2;
  if (ntiles <= 0) return COV_OK;
  CUtensorMap mi, mj;
  int rc;
  if ((rc = wl_status_words(h, s))) return rc;
  uint8_t* sl = tri ? h->Tsl : h->Asl;
  if ((rc = wl_sl_map(h, &mi, sl, nb * nk, SL_BM)) || (rc = wl_sl_map(h, &mj, sl, nb * nk, SL_BN))) return rc;
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
  SlArgs a{rows, row1, t0, t1, (int)nk, ns, tri ? h->Texp : h->Aexp, out, h->tc_status, h->sl_report,
           h->sl_part, nullptr};
  a.ticket = (int*)(h->sl_part + (size_t)SL_SPLIT_TILES * SL_BM * SL_BM);
  if (ns > 1) {
    WL_CHECK(h, cudaMemsetAsync(h->sl_part, 0, (size_t)ntiles * SL_BM * SL_BM * 8, s));
    WL_CHECK(h, cudaMemsetAsync(a.ticket, 0, sizeof(int) * (size_t)ntiles, s));
  }
  static std::once_flag attr_once[WL_MAX_DEVICES];
  static int attr_rc[WL_MAX_DEVICES];
  if (wl_once_per_device(attr_once, attr_rc, [] {
        return (int)cudaFuncSetAttribute(k_syrk_sl, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         SlShape<SL_NG>::kSmem);
      }) != 0)
    return wl_fail(h, COV_ERR_CUDA, "cudaFuncSetAttribute(k_syrk_sl) failed");
  k_syrk_sl<<<(unsigned)(ntiles * ns), SL_THREADS, SlShape<SL_NG>::kSmem, s>>>(mi, mj, a);
  WL_LAUNCH(h, "k_syrk_sl");
  return COV_OK;
}
