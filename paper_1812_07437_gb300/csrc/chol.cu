// Cumulative signal-to-noise (paper Sec. 5, Eqs. SNprim and eq:SN).
//
// The selected entries (P, B or the joint vector) are reordered by their
// largest ell bin (stable), scaled to a diagonal of 1, C' = S C S and D' = S D,
// and factorised in 64-bit fixed point (chol_fx.cu), which
// carries the data row along as y = L^-1 D'.  Because the leading principal
// block of a Cholesky factor is the factor of the leading principal block,
// (S/N)^2 for every cumulative ell_max is a prefix sum of y^2 over the
// reordered entries.  k_potrf_diag and k_trsm_rows are the FP64 kernels of the
// allocation-free form (noalloc.cu).
#include <algorithm>

#include "common.cuh"

#define NB 64

// in-place Cholesky of the kb x kb diagonal block at (k0, k0); one block of
// 256 threads, thread (tx, ty) owns rows ty + 16 r and columns tx + 16 c
__global__ void k_potrf_diag(OutMap W, int64_t k0, int kb, int* status) {
  __shared__ double L[NB][NB + 1];
  int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      int i = ty + 16 * r, l = tx + 16 * c;
      L[i][l] = (i < kb && l <= i) ? *W.at(k0 + i, k0 + l) : 0.0;
    }
  __shared__ double inv_sh;
  __syncthreads();
  for (int j = 0; j < kb; ++j) {
    if (threadIdx.x == 0) {
      double d = L[j][j];
      if (!(d > 0.0)) {
        atomicExch(status, 1);
        d = 1.0;
      }
      double r = sqrt(d);
      L[j][j] = r;
      inv_sh = 1.0 / r;  // one FP64 division per step, shared by all threads
    }
    __syncthreads();
    double inv = inv_sh;
    if (tx == (j & 15)) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        int i = ty + 16 * r;
        if (i > j && i < kb) L[i][j] *= inv;
      }
    }
    __syncthreads();
    // rank-1 update of the trailing triangle j < l <= i < kb: only the active
    // elements are enumerated, so no FP64 issue slot goes to masked lanes
    int m = kb - j - 1;
    int tot = m * (m + 1) / 2;
    for (int e = threadIdx.x; e < tot; e += blockDim.x) {
      int ii = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
      while (ii * (ii + 1) / 2 > e) --ii;
      while ((ii + 1) * (ii + 2) / 2 <= e) ++ii;
      int ll = e - ii * (ii + 1) / 2;
      int i = j + 1 + ii, l = j + 1 + ll;
      L[i][l] -= L[i][j] * L[l][j];
    }
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      int i = ty + 16 * r, l = tx + 16 * c;
      if (i < kb && l <= i) *W.at(k0 + i, k0 + l) = L[i][l];
    }
}

#define TRSM_ROWS 32
// rows r in [r0, r1): x L11^T = a by forward substitution, one row per lane
// (32 rows per block): every lane runs the whole recurrence of its own row in
// registers, reading L11 from shared memory by broadcast, so no FP64 issue slot
// is spent on masked lanes
__global__ void k_trsm_rows(OutMap W, int64_t k0, int kb, int64_t r0, int64_t r1) {
  __shared__ double L[NB][NB + 1];
  __shared__ double invd[NB];
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    int i = e >> 6, l = e & 63;
    L[i][l] = (i < kb && l <= i) ? *W.at(k0 + i, k0 + l) : 0.0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kb; i += blockDim.x) invd[i] = 1.0 / L[i][i];
  __syncthreads();
  int64_t r = r0 + (int64_t)blockIdx.x * TRSM_ROWS + threadIdx.x;
  if (r >= r1) return;
  double* row = W.at(r, k0);  // kb <= 64 consecutive entries (k0 is a multiple of 64)
  double x[NB];
#pragma unroll
  for (int j = 0; j < NB; ++j) x[j] = (j < kb) ? row[j] : 0.0;
#pragma unroll
  for (int j = 0; j < NB; ++j) {
    if (j < kb) {
      // four independent partial sums break the FP64 dependency chain
      double v0 = x[j], v1 = 0.0, v2 = 0.0, v3 = 0.0;
#pragma unroll
      for (int l = 0; l + 3 < j; l += 4) {
        v0 -= x[l] * L[j][l];
        v1 -= x[l + 1] * L[j][l + 1];
        v2 -= x[l + 2] * L[j][l + 2];
        v3 -= x[l + 3] * L[j][l + 3];
      }
#pragma unroll
      for (int l = j & ~3; l < j; ++l) v0 -= x[l] * L[j][l];
      x[j] = ((v0 + v1) + (v2 + v3)) * invd[j];
    }
  }
#pragma unroll
  for (int j = 0; j < NB; ++j)
    if (j < kb) row[j] = x[j];
}

__global__ void k_snr_prefix(int64_t Ms, OutMap W, const int64_t* cnt, int nl, double* out) {
  __shared__ double sh[32];
  int c = blockIdx.x;
  int64_t n = cnt[c];
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    double y = *W.at(Ms, i);
    s += y * y;
  }
  s = block_sum(s, sh);
  if (threadIdx.x == 0) out[c] = (n > 0) ? sqrt(s) : nan("");
}

// Factorisation of the selection (wl_fx_factor), then (S/N)^2 for every
// cumulative selection as the prefix sums of y^2 up to cnt_d[c] entries, into
// out_d (device, n_ell).  Outside a captured batch step the result is copied to
// h_snr and the status words are checked; inside one (h->deferred) both stay on
// the device and the status words accumulate over the replays.
static int factor_and_prefix(cov_handle* h, OutMap Wm, int64_t Ms, const int* perm, const double* C, int64_t ldc,
                             const double* D, const int64_t* cnt_d, double* out_d, double* h_snr, cudaStream_t s) {
  int rc;
  if ((rc = wl_status_words(h, s))) return rc;
  if (!h->deferred) WL_CHECK(h, cudaMemsetAsync(h->piv_status, 0, 2 * sizeof(int), s));
  if ((rc = wl_fx_factor(h, Wm, Ms, perm, C, ldc, D, s))) return rc;
  int tk = wl_stage_begin(h, ST_SNR_PREFIX, s);
  k_snr_prefix<<<h->nl, 256, 0, s>>>(Ms, Wm, cnt_d, h->nl, out_d);
  WL_LAUNCH(h, "k_snr_prefix");
  wl_stage_end(h, tk, s);
  if (h->deferred) return COV_OK;
  WL_CHECK(h, cudaMemcpyAsync(h_snr, out_d, sizeof(double) * h->nl, cudaMemcpyDeviceToHost, s));
  return wl_snr_status(h, s);
}

int wl_status_words(cov_handle* h, cudaStream_t s) {
  if (h->piv_status) return COV_OK;
  WL_CHECK(h, cudaMalloc(&h->piv_status, 3 * sizeof(int)));
  h->chol_status = h->piv_status + 1;
  h->sl_report = h->piv_status + 2;
  WL_CHECK(h, cudaMemsetAsync(h->piv_status, 0, 3 * sizeof(int), s));
  return COV_OK;
}

// The status words of the factorisations on s, and of the FP64 assemblies before them,
// which do not wait for their kernels themselves (synchronises s)
int wl_snr_status(cov_handle* h, cudaStream_t s) {
  int w[3] = {0, 0, 0};
  WL_CHECK(h, cudaMemcpyAsync(w, h->piv_status, sizeof(w), cudaMemcpyDeviceToHost, s));
  WL_CHECK(h, cudaStreamSynchronize(s));
  if (w[2]) {
    h->ops_terms = -1;  // the trispectrum table that a band prepared may be what is incomplete
    WL_CHECK(h, cudaMemsetAsync(h->sl_report, 0, sizeof(int), s));
    return wl_fail(h, COV_ERR_TIMEOUT, "FP64 contraction of an earlier assembly: a bounded mbarrier wait expired");
  }
  if (w[1]) return wl_fail(h, COV_ERR_TIMEOUT, "Cholesky trailing update: a bounded mbarrier wait expired");
  if (w[0]) return wl_fail(h, COV_ERR_NOT_PD, "Cholesky met a non-positive pivot");
  return COV_OK;
}

static int maxbin_of(const cov_handle* h, int64_t a) {
  return h->rowdesc[8 * a] == 0 ? h->rowdesc[8 * a + 1] : h->rowdesc[8 * a + 3];
}

// Device copies of a selection (slot 0..2: P, B, joint for the dense S/N;
// slot 3: all rows, in their cumulative order, for the packed-tile S/N): the
// reordering permutation and the prefix counts, built once per handle.
static int selection(cov_handle* h, int slot, cudaStream_t s) {
  if (h->sel[slot].ready) return COV_OK;
  std::vector<int> sel;
  for (int64_t a = 0; a < h->M; ++a) {
    int type = h->rowdesc[8 * a];
    if (slot == COV_WHICH_P && type != 0) continue;
    if (slot == COV_WHICH_B && type != 1) continue;
    sel.push_back((int)a);
  }
  if (slot < 3)
    std::stable_sort(sel.begin(), sel.end(), [&](int x, int y) { return maxbin_of(h, x) < maxbin_of(h, y); });
  int64_t Ms = (int64_t)sel.size();
  std::vector<int64_t> cnt(h->nl, 0);
  for (int c = 0; c < h->nl; ++c)
    for (int64_t i = 0; i < Ms; ++i)
      if (maxbin_of(h, sel[i]) <= c) cnt[c] = i + 1;
  auto& z = h->sel[slot];
  if (!z.perm) {
    WL_CHECK(h, cudaMalloc(&z.perm, sizeof(int) * (size_t)std::max<int64_t>(Ms, 1)));
    WL_CHECK(h, cudaMalloc(&z.cnt, sizeof(int64_t) * h->nl));
    WL_CHECK(h, cudaMalloc(&z.out, sizeof(double) * h->nl));
    h->allocated += sizeof(int) * (size_t)std::max<int64_t>(Ms, 1) + sizeof(int64_t) * h->nl + sizeof(double) * h->nl;
  }
  if (Ms) WL_CHECK(h, cudaMemcpyAsync(z.perm, sel.data(), sizeof(int) * Ms, cudaMemcpyHostToDevice, s));
  WL_CHECK(h, cudaMemcpyAsync(z.cnt, cnt.data(), sizeof(int64_t) * h->nl, cudaMemcpyHostToDevice, s));
  WL_CHECK(h, cudaStreamSynchronize(s));  // sel and cnt are host memory read by the copies
  z.Ms = Ms;
  z.ready = true;
  return COV_OK;
}

// What a step with deferred status reads needs first: the selections and status words
int wl_snr_prepare(cov_handle* h, cudaStream_t s) {
  int rc;
  for (int w = 0; w < 3; ++w)
    if ((rc = selection(h, w, s))) return rc;
  return wl_status_words(h, s);
}

// perm: another order of the selection's rows (the factor is then of that order, and the
// prefix sums are of no use)
int wl_snr(cov_handle* h, const double* C, int64_t ldc, const double* D, int which, double* h_snr, cudaStream_t s,
           const int* perm) {
  int rc;
  if ((rc = selection(h, which, s))) return rc;
  const auto& z = h->sel[which];
  const int64_t Ms = z.Ms;
  if (Ms == 0) {
    if (h_snr)
      for (int c = 0; c < h->nl; ++c) h_snr[c] = nan("");
    return COV_OK;
  }
  // rows padded to 8 entries: the trailing update moves pairs of them
  int64_t ldw = (Ms + 1 + 7) / 8 * 8;
  int64_t need = ldw * (Ms + 1);
  if (need > h->work_n) {
    if (h->work) {
      cudaFree(h->work);
      h->allocated -= sizeof(double) * h->work_n;
    }
    h->work = nullptr;
    h->work_n = 0;
    if (wl_over_budget(h, sizeof(double) * need))
      return wl_fail(h, COV_ERR_NOMEM, "hbm_budget exceeded allocating the Cholesky workspace");
    WL_CHECK(h, cudaMalloc(&h->work, sizeof(double) * need));
    h->work_n = need;
    h->allocated += sizeof(double) * need;
  }
  h->work_ld = ldw;
  return factor_and_prefix(h, out_rows(h->work, ldw), Ms, perm ? perm : z.perm, C, ldc, D, z.cnt, z.out, h_snr, s);
}

// In place on the lower-packed tiles (rows in cumulative order)
int wl_snr_tiles(cov_handle* h, double* Ct, const double* D, double* h_snr, cudaStream_t s) {
  int rc;
  if ((rc = selection(h, 3, s))) return rc;
  return factor_and_prefix(h, out_tiles(Ct, 0), h->M, nullptr, nullptr, 0, D, h->sel[3].cnt, h->sel[3].out, h_snr, s);
}
