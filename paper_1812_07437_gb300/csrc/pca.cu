// Principal components of the joint covariance (paper Sec. 6, Eqs. SNPCA,
// NewObs, SNperEign, CumulSN) on the GPU, in FP64.
//
// The eigen-pairs of C come from one-sided Jacobi on its Cholesky factor
// (Demmel & Veselic 1992), which keeps high relative accuracy on every
// eigenvalue of a graded positive definite matrix, however small (the paper's
// covariances span ~23 decades):
//
//  * the FP64-accurate Cholesky of the S/N (cov_snr) on the scaled matrix C' = S C S
//    (S ~ d^-1/2), rows in order of descending C_aa, gives the factor L' and the
//    solved data row y = L'^-1 S D = L^-1 D with L = S^-1 L';
//  * sweeps of plane rotations of column pairs make the columns of L orthogonal:
//    L J = U diag(sigma), C = L L^T = U diag(sigma^2) U^T, so the eigenvalues are
//    lambda_a = |l_a|^2.  With the large variances first, L's columns are graded and
//    already closer to orthogonal than its rows (L^T L is one LR step from L L^T; Veselic
//    & Hari 1989): at M = 818, 8 sweeps where the rows in the S/N's order took 12;
//  * (S/N)^2 of mode a, (u_a . D)^2 / lambda_a, is (J^T y)_a^2, since D = L y =
//    U diag(sigma) J^T y: y is carried as one more entry of every column (not part of
//    its products), and no eigenvector needs to be accumulated;
//  * each sweep visits every pair once: blocks of b columns in round-robin order, a CTA
//    per pair of blocks, and inside it b disjoint pairs at a time (k_pca_round).  The
//    skip test is |c| <= tol sqrt(a b);
//  * eigenvalues sorted ascending by rank, the cumulative (S/N)^2 in both of
//    the paper's orders and the mode counts for 90/95/99% of the total S/N
//    computed on the device.
#include <algorithm>
#include <chrono>
#include <mutex>
#include <vector>

#include "common.cuh"

#define PCA_TOL 1e-15
#define PCA_MAX_SWEEPS 60

// Column j of L, contiguous: G[j][i] = factor entry (i, j) / scale of row p_i (i >= j,
// zero above), entry n the solved data row's y_j, the rest of the ld entries zero.
// One 32 x 32 tile per CTA, transposed in shared memory.
__global__ void __launch_bounds__(256) k_pca_build(int n, int ld, const double* __restrict__ W, int64_t ldw,
                                                   const int* __restrict__ perm, const double* __restrict__ C,
                                                   int64_t ldc, double* G, double* D) {
  __shared__ double t[32][33];
  const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int r = ty; r < 32; r += 8) {
    const int i = i0 + r, j = j0 + tx;
    double v = 0.0;
    if (i < n && j <= i) {
      const int64_t p = perm[i];
      v = W[(int64_t)i * ldw + j] / variance_scale(C[p * ldc + p]);
    } else if (i == n && j < n) {
      v = W[(int64_t)n * ldw + j];
    }
    t[r][tx] = v;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const int j = j0 + r, i = i0 + tx;
    if (j < n && i < ld) G[(int64_t)j * ld + i] = t[tx][r];
    if (j < n && i == 0) D[j] = 1.0;
  }
}

// a_j = |g_j|^2 of the stored column, after an exact scaling by a power of two to a_j in
// [1/4, 4) (D_j, the square of the column's scale factor, takes it up).  A zero column
// stays as it is: it is never rotated.
__global__ void __launch_bounds__(128) k_pca_norms(double* G, int n, int ld, double* D, double* a) {
  __shared__ double sh[32];
  double* g = G + (int64_t)blockIdx.x * ld;
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s = fma(g[i], g[i], s);
  s = block_sum(s, sh);
  __shared__ int e;
  if (threadIdx.x == 0) {
    e = s > 0.0 && isfinite(s) ? ilogb(s) / 2 : 0;
    a[blockIdx.x] = scalbn(s, -2 * e);
    D[blockIdx.x] = scalbn(D[blockIdx.x], 2 * e);
  }
  __syncthreads();
  if (e == 0) return;
  const double f = scalbn(1.0, -e);
  for (int i = threadIdx.x; i <= n; i += blockDim.x) g[i] *= f;
}

// One round of a sweep.  CTA k takes the column blocks at positions k and nblk - 1 - k of
// the round's arrangement (position 0 fixed, the others rotating) into shared memory and
// rotates all pairs between them, b disjoint pairs at a time (`all`: the pairs inside the
// blocks too; the first round of a sweep).  Four warps per pair, and one warp for the
// angles of all pairs, a lane each.
//
// FP64 bounds it (an SM completes two FP64 operations per clock, and a dependent one takes
// ~64 cycles), so a pair costs three operations per entry: the product c, and a rotation
// in scaled form.  The true columns are sqrt(D_p) x and sqrt(D_q) z (D_q <= D_p), and
//   x' = x - alpha z,  z' = z + beta x,  D' = D / (1 + alpha beta),  alpha = rho beta,
//   rho = D_q / D_p,   rho u beta^2 + g beta - u = 0,  u = x.z,  g = rho |z|^2 - |x|^2
// is the rotation by the angle of tan 2 theta = 2 c / (b - a).  It is a rotation to FP64
// rounding for any beta; beta itself is the smaller root by an FP32 estimate and one
// Newton step in FP64 (~1e-13: an FP64 divide or root is a dependent chain of ~0.3 us).
// |x|^2 and |z|^2 follow the rotations and are computed afresh once per sweep.
//
// M = 818: 17.9 ms per sweep (one launch per disjoint set, seven operations per entry,
// columns from L2) -> 4.6 ms, and the whole call 215.6 (12 sweeps) -> 37.9 ms (8); a step
// is ~3.3 us of FP64 work and the chain of the sum and the angle, a round ~5 us of launch,
// loads and stores more.  (Launching rounds programmatically early packs their CTAs
// unevenly on the SMs: 43 ms.)
#define PCA_TEAM 128
#define PCA_MAX_B 7  // 7 x 128 + 32 threads

struct PcaRound {
  double *G, *D, *a;
  int n, ld, b, nblk, round, all;
  int* rotated;
};

__device__ __forceinline__ void pca_cp16(double* dst, const double* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

template <bool SMEM>
__global__ void __launch_bounds__(PCA_TEAM* PCA_MAX_B + 32) k_pca_round(PcaRound A) {
  extern __shared__ double sm[];
  __shared__ double Ds[2 * PCA_MAX_B], as[2 * PCA_MAX_B], us[PCA_MAX_B], al[PCA_MAX_B], be[PCA_MAX_B];
  __shared__ int turn[PCA_MAX_B], dirty[2 * PCA_MAX_B], down[2 * PCA_MAX_B];
  const int n = A.n, b = A.b, tid = threadIdx.x, lane = tid & 31, team = tid / PCA_TEAM;
  auto block = [&](int i) { return i == 0 ? 0 : 1 + (i - 1 + A.round) % (A.nblk - 1); };
  const int B0 = block(blockIdx.x), B1 = block(A.nblk - 1 - blockIdx.x);
  const int P = min(B0, B1), Q = max(B0, B1);
  const int cP = min(b, n - P * b), cQ = min(b, n - Q * b);  // (Q, and with `all` P, may lie beyond the end)
  if (cP <= 0 || (cQ <= 0 && !A.all)) return;
  auto filled = [&](int s) { return s < b ? s < cP : s - b < cQ; };
  auto column = [&](int s) { return s < b ? P * b + s : Q * b + s - b; };
  double* red = SMEM ? sm + (size_t)2 * b * A.ld : sm;  // [pair][thread]
  auto at = [&](int s) { return SMEM ? sm + (size_t)s * A.ld : A.G + (int64_t)column(s) * A.ld; };
  if (SMEM) {
    for (int s = 0; s < 2 * b; ++s)
      if (filled(s)) {
        const double* src = A.G + (int64_t)column(s) * A.ld;
        for (int i = 2 * tid; i < A.ld; i += 2 * blockDim.x) pca_cp16(sm + (size_t)s * A.ld + i, src + i);
      }
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  if (tid < 2 * b) {
    Ds[tid] = filled(tid) ? A.D[column(tid)] : 1.0;
    as[tid] = filled(tid) ? A.a[column(tid)] : 0.0;
    dirty[tid] = 0;
    down[tid] = 0;
  }
  __syncthreads();
  const int steps = A.all ? 2 * b - 1 : b;
  // slots of pair i at a step
  auto pair = [&](int i, int step, int* s0, int* s1) {
    if (A.all) {
      const int m = 2 * b;
      auto pos = [&](int k) { return k == 0 ? 0 : 1 + (k - 1 + step) % (m - 1); };
      *s0 = pos(i);
      *s1 = pos(m - 1 - i);
    } else {
      *s0 = i;
      *s1 = b + (i + step) % b;
    }
    return filled(*s0) && filled(*s1);
  };
  const int wt = (tid >> 5) & 3;
  const int e0 = ((wt + team) & 3) * 32 + lane;  // the odd chunks of the pairs on different schedulers
  int turns = 0;
  for (int step = 0; step < steps; ++step) {
    int s0 = 0, s1 = 0;
    double *x = nullptr, *z = nullptr, rho = 1.0;
    bool on = false, swapped = false;
    if (team < b) {
      on = pair(team, step, &s0, &s1);
      if (on) {
        x = at(s0);
        z = at(s1);
        double u0 = 0.0, u1 = 0.0;
        int i = e0;
        for (; i + PCA_TEAM < n; i += 2 * PCA_TEAM) {
          u0 = fma(x[i], z[i], u0);
          u1 = fma(x[i + PCA_TEAM], z[i + PCA_TEAM], u1);
        }
        if (i < n) u0 = fma(x[i], z[i], u0);
        red[tid] = u0 + u1;
        asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(PCA_TEAM) : "memory");
        if (wt == (team & 3)) {
          const double* r = red + team * PCA_TEAM + lane;
          const double v = warp_sum((r[0] + r[32]) + (r[64] + r[96]));
          if (lane == 0) us[team] = v;
        }
      }
    } else if (lane < b) {
      on = pair(lane, step, &s0, &s1);
      swapped = Ds[s0] < Ds[s1];
      if (swapped) {
        const int t = s0;
        s0 = s1;
        s1 = t;
      }
      if (on) rho = Ds[s1] / Ds[s0];
    }
    __syncthreads();
    double q = 0.0, u = 0.0, ax = 0.0, az = 0.0, alpha = 0.0, beta = 0.0;
    if (team == b && lane < b) {
      if (on) {
        u = us[lane];
        ax = as[s0];
        az = as[s1];
        const double g = fma(rho, az, -ax), r1 = rho * u;
        const float gf = (float)g, uf = (float)u;
        beta = (double)(2.0f * uf / (gf + copysignf(sqrtf(fmaf(gf, gf, 4.0f * (float)r1 * uf)), gf)));
        const double m = fma(r1, beta, g);
        beta = fma(-fma(m, beta, -u), (double)(1.0f / (float)fma(r1, beta, m)), beta);
        alpha = rho * beta;
        q = alpha * beta;
        on = u * u > (PCA_TOL * PCA_TOL) * (ax * az) && isfinite(q);
      }
      turn[lane] = !on ? 0 : swapped ? 2 : 1;
      al[lane] = alpha;
      be[lane] = beta;
      if (on) {
        dirty[s0] = dirty[s1] = 1;
        ++turns;
      }
    }
    __syncthreads();
    if (team < b && on && turn[team]) {
      if (turn[team] == 2) {
        double* t = x;
        x = z;
        z = t;
      }
      const double av = al[team], bv = be[team];
      for (int i = e0; i <= n; i += PCA_TEAM) {
        const double xv = x[i], zv = z[i];
        x[i] = fma(-av, zv, xv);
        z[i] = fma(bv, xv, zv);
      }
    }
    __syncthreads();
    if (team == b && lane < b && on) {
      const double r = 1.0 / (1.0 + q);
      Ds[s0] *= r;
      Ds[s1] *= r;
      as[s0] = fma(alpha * alpha, az, fma(-2.0 * alpha, u, ax));
      as[s1] = fma(beta * beta, ax, fma(2.0 * beta, u, az));
    }
    __syncwarp();
  }
  if (team == b && turns) atomicAdd(A.rotated, turns);
  __syncthreads();
  // back to memory; a stored column that has grown a lot is scaled down exactly
  if (tid < 2 * b && dirty[tid]) {
    if (as[tid] > 0x1p40) {
      down[tid] = ilogb(as[tid]) / 2;
      as[tid] = scalbn(as[tid], -2 * down[tid]);
      Ds[tid] = scalbn(Ds[tid], 2 * down[tid]);
    }
    A.D[column(tid)] = Ds[tid];
    A.a[column(tid)] = as[tid];
  }
  __syncthreads();
  for (int s = 0; s < 2 * b; ++s) {
    if (!dirty[s] || (!SMEM && !down[s])) continue;
    const double* src = at(s);
    double* dst = A.G + (int64_t)column(s) * A.ld;
    if (down[s]) {
      const double f = scalbn(1.0, -down[s]);
      for (int i = tid; i <= n; i += blockDim.x) dst[i] = f * src[i];
    } else {
      for (int i = 2 * tid; i < A.ld; i += 2 * blockDim.x) *(double2*)(dst + i) = *(const double2*)(src + i);
    }
  }
}

// Columns per block: the sweep's time over b, from what a round and a step cost (us; a
// step is latency-bound at small n, then 1.5 cycles per entry and pair of an SM).  All
// sweeps, b = 1, 2, 3, 4, 5, 7: M = 818 59.8, 47.9, 36.8, 38.8, 41.2, 49.6 ms (the rule
// takes 3: 137 CTAs); M = 144 6.7, 4.3, 4.0, 3.9, 3.9, 4.9 ms
static int pca_block_columns(int n, int ld, int64_t sms, size_t smem_max, bool* fits) {
  int best = 1;
  double t_best = 0.0;
  *fits = false;
  for (int b = 1; b <= PCA_MAX_B; ++b) {
    const size_t smem = sizeof(double) * (2 * (size_t)b * ld + (size_t)b * PCA_TEAM);
    if (smem > smem_max) break;
    *fits = true;
    const int64_t nblk = (n + b - 1) / b, ctas = (nblk + 1) / 2, waves = (ctas + sms - 1) / sms;
    const double t = (double)nblk * (5.0 + b * (2.2 + 0.0016 * n * (double)(b * waves)));
    if (b == 1 || t < t_best) {
      t_best = t;
      best = b;
    }
  }
  return best;
}

// per mode a: lambda_a = |l_a|^2, (S/N)^2_a = (J^T y)_a^2
__global__ void __launch_bounds__(128) k_pca_modes(const double* G, int n, int ld, const double* D, double* lam,
                                                   double* snr2) {
  __shared__ double sh[32];
  const double* g = G + (int64_t)blockIdx.x * ld;
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s = fma(g[i], g[i], s);
  s = block_sum(s, sh);
  if (threadIdx.x == 0) {
    const double d = D[blockIdx.x];
    lam[blockIdx.x] = d * s;
    snr2[blockIdx.x] = d * g[n] * g[n];
  }
}

// rank of key[i stride] (ties by index), ascending or with `desc` descending, by the
// integer order of the bits (a total order, NaN included): a warp per element.  pos[i] =
// rank; inv[rank] = i.
__device__ __forceinline__ long long pca_key(double x, int desc) {
  long long k = __double_as_longlong(x);
  k ^= (long long)((unsigned long long)(k >> 63) >> 1);
  return desc ? ~k : k;
}
__global__ void __launch_bounds__(256) k_pca_rank(int n, const double* key, int64_t stride, int desc, int* pos,
                                                  int* inv) {
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;
  const long long ki = pca_key(key[i * stride], desc);
  int r = 0;
  for (int j = lane; j < n; j += 32) {
    const long long kj = pca_key(key[j * stride], desc);
    r += (kj < ki || (kj == ki && j < i)) ? 1 : 0;
  }
  r = __reduce_add_sync(~0u, r);
  if (lane == 0) {
    if (pos) pos[i] = r;
    if (inv) inv[r] = i;
  }
}

// sorted copies (by the ranks), cumulative (S/N)^2 in both orders (Eq. CumulSN,
// sequential sums as written, one thread each) and the mode counts for 90/95/99% of the
// total S/N (the first mode that reaches it, by all threads)
__global__ void __launch_bounds__(256) k_pca_cumulative(int n, const double* lam, const double* snr2,
                                                        const int* pos_var, const int* pos_info, double* lam_s,
                                                        double* snr2_s, double* cum_var, double* cum_info, int* modes) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    lam_s[pos_var[i]] = lam[i];
    snr2_s[pos_var[i]] = snr2[i];
    cum_var[pos_var[i]] = snr2[i];
    cum_info[pos_info[i]] = snr2[i];
  }
  __shared__ int first[3];
  __shared__ double buf[2][1024];
  if (threadIdx.x < 3) first[threadIdx.x] = n;
  double run = 0.0;
  for (int a0 = 0; a0 < n; a0 += 1024) {
    const int m = min(1024, n - a0);
    __syncthreads();
    for (int a = threadIdx.x; a < m; a += blockDim.x) {
      buf[0][a] = cum_var[a0 + a];
      buf[1][a] = cum_info[a0 + a];
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && threadIdx.x < 64) {
      double* v = buf[threadIdx.x >> 5];
      for (int a = 0; a < m; ++a) v[a] = run += v[a];
    }
    __syncthreads();
    for (int a = threadIdx.x; a < m; a += blockDim.x) {
      cum_var[a0 + a] = buf[0][a];
      cum_info[a0 + a] = buf[1][a];
    }
  }
  __syncthreads();
  const double total = sqrt(cum_info[n - 1]);
  const double fr[3] = {0.90, 0.95, 0.99};
  for (int a = threadIdx.x; a < n; a += blockDim.x) {
    const double c = sqrt(cum_info[a]);
    for (int f = 0; f < 3; ++f)
      if (c >= fr[f] * total) atomicMin(&first[f], a + 1);
  }
  __syncthreads();
  if (threadIdx.x < 3) modes[threadIdx.x] = first[threadIdx.x];
}

extern "C" int cov_pca(cov_handle* h, const double* d_C, int64_t ldc, const double* d_D, double* h_lam,
                       double* h_snr2, double* h_cum_var, double* h_cum_info, cov_pca_info* info, void* stream) {
  if (!h) return COV_ERR_INVALID;
  if (!d_C || !d_D || ldc < h->M) return wl_fail(h, COV_ERR_INVALID, "cov_pca: null input or ldc < M");
  if (h->M > (1 << 20)) return wl_fail(h, COV_ERR_INVALID, "cov_pca: M above 2^20");
  cudaStream_t s = (cudaStream_t)stream;
  using clk = std::chrono::steady_clock;
  auto ms_since = [](clk::time_point t) { return std::chrono::duration<double, std::milli>(clk::now() - t).count(); };
  // 1. the arrays; the rows in order of descending variance; their FP64-accurate Cholesky,
  //    with y = L^-1 D
  auto t0 = clk::now();
  if (h->M < 1) return wl_fail(h, COV_ERR_INVALID, "cov_pca: empty selection");
  const int n = (int)h->M, ld = (n + 2) / 2 * 2;  // even: rows of 16 bytes
  const size_t gbytes = sizeof(double) * (size_t)n * ld;
  const size_t need = sizeof(double) * (size_t)n * ((size_t)n + 9) + sizeof(int) * ((size_t)n * 2 + 4);
  if (need > h->pca_bytes) {
    if (h->pca_buf) {
      cudaFree(h->pca_buf);
      h->allocated -= h->pca_bytes;
      h->pca_buf = nullptr;
      h->pca_bytes = 0;
    }
    if (wl_over_budget(h, need))
      return wl_fail(h, COV_ERR_NOMEM, "hbm_budget exceeded allocating the PCA workspace");
    WL_CHECK(h, cudaMalloc(&h->pca_buf, need));
    h->pca_bytes = need;
    h->allocated += h->pca_bytes;
  }
  double* G = (double*)h->pca_buf;  // n x ld <= n (n + 2), then seven arrays of n
  double *lam = (double*)((char*)h->pca_buf + gbytes), *a = lam + n, *snr2 = a + n, *lam_s = snr2 + n;
  double *snr2_s = lam_s + n, *cum_var = snr2_s + n, *cum_info = cum_var + n, *Dj = lam;
  int* pos_var = (int*)(cum_info + n);
  int* pos_info = pos_var + n;
  int* rotated = pos_info + n;
  int* modes = rotated + 1;
  const unsigned warps = (unsigned)((n + 7) / 8);
  k_pca_rank<<<warps, 256, 0, s>>>(n, d_C, ldc + 1, 1, nullptr, pos_info);
  WL_LAUNCH(h, "k_pca_rank");
  std::vector<double> snr_cum(h->nl);
  int rc;
  if ((rc = wl_snr(h, d_C, ldc, d_D, COV_WHICH_JOINT, snr_cum.data(), s, pos_info))) return rc;
  const double ms_chol = ms_since(t0);
  // 2. the columns of L
  k_pca_build<<<dim3((unsigned)((ld + 31) / 32), (unsigned)((n + 31) / 32)), 256, 0, s>>>(n, ld, h->work, h->work_ld,
                                                                                         pos_info, d_C, ldc, G, Dj);
  WL_LAUNCH(h, "k_pca_build");
  // 3. Jacobi sweeps until a sweep rotates no pair
  auto t1 = clk::now();
  int sweeps = 0, converged = 0;
  if (n > 1) {
    const size_t smem_max = 227 * 1024 - 1024;
    static std::once_flag attr_once[WL_MAX_DEVICES];
    static int attr_rc[WL_MAX_DEVICES];
    if (wl_once_per_device(attr_once, attr_rc, [] {
          return (int)cudaFuncSetAttribute(k_pca_round<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           227 * 1024 - 1024);
        }) != 0)
      return wl_fail(h, COV_ERR_CUDA, "cudaFuncSetAttribute (PCA kernels) failed");
    bool fits = false;
    const int b = pca_block_columns(n, ld, wl_num_sms(), smem_max, &fits);
    const int nblk = ((n + b - 1) / b + 1) / 2 * 2;
    const size_t smem = sizeof(double) * ((fits ? 2 * (size_t)b * ld : 0) + (size_t)b * PCA_TEAM);
    for (sweeps = 1; sweeps <= PCA_MAX_SWEEPS; ++sweeps) {
      WL_CHECK(h, cudaMemsetAsync(rotated, 0, sizeof(int), s));
      k_pca_norms<<<(unsigned)n, 128, 0, s>>>(G, n, ld, Dj, a);
      for (int r = 0; r < std::max(nblk - 1, 1); ++r) {
        PcaRound p{G, Dj, a, n, ld, b, nblk, r, r == 0, rotated};
        if (fits)
          k_pca_round<true><<<(unsigned)(nblk / 2), b * PCA_TEAM + 32, smem, s>>>(p);
        else  // two columns beyond shared memory (M > ~14300): in place
          k_pca_round<false><<<(unsigned)(nblk / 2), b * PCA_TEAM + 32, smem, s>>>(p);
      }
      WL_LAUNCH(h, "k_pca_round");
      int r = 0;
      WL_CHECK(h, cudaMemcpyAsync(&r, rotated, sizeof(int), cudaMemcpyDeviceToHost, s));
      WL_CHECK(h, cudaStreamSynchronize(s));
      if (r == 0) {
        converged = 1;
        break;
      }
    }
    if (sweeps > PCA_MAX_SWEEPS) sweeps = PCA_MAX_SWEEPS;
  } else {
    converged = 1;
  }
  // 4. modes, order, cumulative forms
  k_pca_modes<<<(unsigned)n, 128, 0, s>>>(G, n, ld, Dj, lam, snr2);
  k_pca_rank<<<warps, 256, 0, s>>>(n, lam, 1, 0, pos_var, nullptr);
  k_pca_rank<<<warps, 256, 0, s>>>(n, snr2, 1, 1, pos_info, nullptr);
  k_pca_cumulative<<<1, 256, 0, s>>>(n, lam, snr2, pos_var, pos_info, lam_s, snr2_s, cum_var, cum_info, modes);
  WL_LAUNCH(h, "PCA mode kernels");
  int hm[3] = {0, 0, 0};
  double tot = 0.0;
  if (h_lam) WL_CHECK(h, cudaMemcpyAsync(h_lam, lam_s, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
  if (h_snr2) WL_CHECK(h, cudaMemcpyAsync(h_snr2, snr2_s, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
  if (h_cum_var) WL_CHECK(h, cudaMemcpyAsync(h_cum_var, cum_var, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
  if (h_cum_info) WL_CHECK(h, cudaMemcpyAsync(h_cum_info, cum_info, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
  WL_CHECK(h, cudaMemcpyAsync(hm, modes, sizeof(hm), cudaMemcpyDeviceToHost, s));
  WL_CHECK(h, cudaMemcpyAsync(&tot, cum_info + (n - 1), sizeof(double), cudaMemcpyDeviceToHost, s));
  WL_CHECK(h, cudaStreamSynchronize(s));
  const double ms_jac = ms_since(t1);
  if (info) {
    info->M = n;
    info->sweeps = sweeps;
    info->converged = converged;
    info->total_snr2 = tot;
    info->modes_90 = hm[0];
    info->modes_95 = hm[1];
    info->modes_99 = hm[2];
    info->ms_cholesky = ms_chol;
    info->ms_jacobi = ms_jac;
  }
  if (!converged) return wl_fail(h, COV_ERR_TIMEOUT, "cov_pca: Jacobi did not converge within the sweep limit");
  return COV_OK;
}
