// Internal declarations shared by the translation units of libwlcov.
// Device helpers are header-inline (no relocatable device code).
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/wlcov.h"

#define WL_PI 3.14159265358979323846
#define WL_EULER_GAMMA 0.57721566490153286061
#define WL_C_OVER_H0 2997.92458      // Mpc/h
#define WL_RHO_CRIT0 2.77536627e11   // (Msun/h)/(Mpc/h)^3
#define WL_DELTA_C 1.686
#define WL_ST_Q 0.707
#define WL_ST_P 0.3
#define WL_DUFFY_A 10.14
#define WL_DUFFY_B (-0.081)
#define WL_DUFFY_C (-1.01)
#define WL_DUFFY_MPIVOT 2.0e12
#define WL_DELTA_VIR 200.0
#define WL_N_GL_CHI 64     // nodes per piece of the source-redshift rules (the bins' norms, W_i)
#define WL_N_ZS 64         // nodes per source-redshift piece of W_i
#define WL_N_RK4 1024      // RK4 steps of the growth ODE
#define WL_A_INIT 1.0e-3
#define WL_BULLOCK_F 0.01        // Bullock et al. median: nu(F m, a_c) = 1, c = K a / a_c
#define WL_BULLOCK_K 4.0
#define WL_NFW_C_INTEGRAL 1.0    // below this concentration u is the quadrature of its defining integral
#define WL_A_COLLAPSE_MAX 100.0  // a_c where F m has not collapsed by then
#define WL_N_K 4096        // nodes of the sigma(R) and sigma_W^2 rules
#define WL_LNK_MIN (-11.512925464970229)  // ln 1e-5
#define WL_LNK_MAX (6.907755278982137)    // ln 1e3
#define WL_FD_H 1.0e-3     // ln k step of the 4th-order differences
#define WL_N_ZI 64         // intervals of the piecewise chi(z) on [0, z_max]
#define WL_N_CH 12         // Chebyshev nodes of 1 / E(z) per interval
#define WL_ZI_STRIDE 32    // doubles per interval: 13 of the integral, 12 of 1 / E, the whole integral
#define WL_ZI_DER 13
#define WL_ZI_TOT 25
#define WL_KT_THREADS 64   // threads (and k nodes) per block of the linear-spectrum table
#define WL_KSPLIT 4        // blocks that share one sum over the k nodes
#define WL_TRI_GEO 42      // per triple: F2 of the three leg pairs, their cosines, F2 of the 12 shifted shapes

// scalars kept on the device (index into h->scal)
enum { SC_CHIMAX = 0, SC_AMP = 1, SC_NOISE = 2, SC_D1 = 3, SC_STATUS = 7, SC_N = 8 };

// cosmology-only factors of the Eisenstein & Hu transfer function
struct EhConst {
  double ks, al, omh, th2;  // 0.43 h s, alpha_Gamma, Omega_m h, (T_cmb / 2.7)^2
};

struct DevCosmo {
  double Om, Ob, h, ns, sigma8, w0, Tcmb;
};

// timed stages (cov_stage_times)
enum {
  ST_TABLES = 0, ST_COUNTS, ST_SPECTRA, ST_ROWS_T, ST_SYRK_T, ST_GATHER, ST_ROWS_A, ST_SYRK_1H, ST_ROWS_S,
  ST_SYRK_SSC, ST_SNR_PACK, ST_SNR_CHOL, ST_SNR_PREFIX, ST_COUNT
};

struct StageEvent {
  int stage;
  cudaEvent_t a, b;
};

// Where a kernel stores element (r, c) of the lower triangle (c <= r).
//  rows : C[(r - row0) * ldc + c]                     (dense row-major band)
//  tiles: 256 x 256 lower tiles, tile (ti, tj) (tj <= ti) stored row-major
//         at tile index ti (ti + 1) / 2 + tj - tile0, 65536 doubles apart
// cuTensorMapEncodeTiled from the driver, looked up once per process
// (thread-safe: the serving scheduler runs requests on several host threads).
PFN_cuTensorMapEncodeTiled_v12000 wl_encode_tiled();
#define WL_TILE_CACHE 16
int wl_ensure(struct cov_handle* h, void** p, size_t bytes, const char* what);  // assemble.cu: allocate once
// Run f once per CUDA device for the calling thread's current device.
#define WL_MAX_DEVICES 64
template <typename F>
inline int wl_once_per_device(std::once_flag (&flags)[WL_MAX_DEVICES], int (&rc)[WL_MAX_DEVICES], F f) {
  int d = 0;
  cudaGetDevice(&d);
  if (d < 0 || d >= WL_MAX_DEVICES) return COV_ERR_INVALID;
  std::call_once(flags[d], [&] { rc[d] = f(); });
  return rc[d];
}

struct OutMap {
  double* C;
  int64_t ldc, row0, tile0;
  int tiled;
  __device__ __forceinline__ double* at(int64_t r, int64_t c) const {
    if (tiled) {
      int64_t ti = r >> 8, tj = c >> 8;
      return C + ((ti * (ti + 1) / 2 + tj - tile0) << 16) + ((r & 255) << 8) + (c & 255);
    }
    return C + (r - row0) * ldc + c;
  }
};
static inline OutMap out_rows(double* C, int64_t ldc, int64_t row0 = 0) { return OutMap{C, ldc, row0, 0, 0}; }
static inline OutMap out_tiles(double* C, int64_t row0) {
  int64_t t0 = row0 >> 8;
  return OutMap{C, 0, row0, t0 * (t0 + 1) / 2, 1};
}

struct cov_handle {
  int device = 0;
  size_t budget = 0, allocated = 0;
  cov_cosmology cosmo{};
  cov_nz nz{};
  cov_bins bins{};
  // plan (host)
  // nm counts the halo-integral nodes: n_mass mass nodes (nmb) times nc
  // concentration nodes, the concentration index fastest (nc = 1 without scatter)
  int nl = 0, nt = 0, nchi = 0, nm = 0, ntri = 0, K = 0, nmb = 0, nc = 1;
  int64_t M = 0, nP = 0, nB = 0;
  int nleg = 0;            // n_ell * n_tomo
  int64_t ntrow = 0;       // rows of the 1-halo trispectrum factor
  int rmax = 0;            // largest lattice radius
  double omega = 0, theta = 0, ell_f = 0;
  std::vector<double> ell_edges, ell, dell;
  std::vector<int64_t> s_lo, s_hi;
  std::vector<int32_t> tris;      // 3 per triple
  std::vector<int32_t> rowdesc;   // 8 per row
  // device: quadrature nodes on [-1, 1]
  double *gl64x = nullptr, *gl64w = nullptr, *glkx = nullptr, *glkw = nullptr, *glcx = nullptr, *glcw = nullptr;
  double *gl16x = nullptr, *gl16w = nullptr;  // 16-point rule of the small-concentration profiles
  // device: tables
  double* scal = nullptr;
  double *chi = nullptr, *wchi = nullptr, *z = nullptr, *D = nullptr;
  double *ell_d = nullptr, *m = nullptr, *om = nullptr, *sig0 = nullptr, *dlns = nullptr;
  double *mb = nullptr, *omb = nullptr;  // [nmb] mass nodes and weights; m, om: [nm] per (mass, c) node
  double *cs = nullptr, *cw = nullptr;   // [nc] ln c offsets from the median and their weights
  double *sigF = nullptr, *ac = nullptr; // [nmb] sigma(F m, 0) and collapse epoch a_c (Bullock median)
  double *f = nullptr, *b1 = nullptr, *b2 = nullptr, *U = nullptr, *Pl = nullptr, *dPl = nullptr;
  double* Psh = nullptr;  // [n_ell][n_chi][4] P_lin at the shifted k of the ln k differences
  double *zedges = nullptr, *norms = nullptr, *W = nullptr, *sigw2 = nullptr;
  // binning- and n(z)-only tables of the builders, made once (wl_quadrature):
  // the sigma rule's k nodes and weights, the source nodes of the fixed pieces
  // between tomographic edges with their n(z) P_i weights, the Duffy mass
  // factors, the Chebyshev matrix of the chi(z) intervals and the triangles' shapes
  double *knode = nullptr, *kwt = nullptr, *kw8 = nullptr, *kws = nullptr;
  double *zsrc = nullptr, *gsel = nullptr, *cmass = nullptr, *chebm = nullptr, *trigeo = nullptr;
  // rebuilt for every cosmology: chi intervals, k^ns T^2 on the k nodes with
  // the partial sigma_8 sums, growth before normalisation, chi and 1 / chi at the
  // source nodes, (1 + z)^C and r_vir, halo integrals [item][n_chi], Limber weights,
  // projected spectra per symmetric tomographic multiset
  double *zint = nullptr, *pk = nullptr, *amp_part = nullptr, *Draw = nullptr, *chis = nullptr, *cz = nullptr;
  double* ksum = nullptr;   // [sum][WL_KSPLIT][3] parts of the sums over the k nodes
  int* kticket = nullptr;   // [sum] parts delivered so far (zero between launches)
  double *rvir = nullptr, *hint = nullptr, *qw = nullptr, *proj = nullptr;
  int64_t *slo_d = nullptr, *shi_d = nullptr, *Nmodes = nullptr, *Ntri = nullptr;
  int32_t* rowtab = nullptr;  // [nl][2][rmax+1]: x_outer, x_inner per row
  int32_t *tris_d = nullptr, *rowdesc_d = nullptr;
  // device: spectra
  double *P3 = nullptr, *RP3 = nullptr, *B3 = nullptr, *RB3 = nullptr, *B1h3 = nullptr;
  double *Ps = nullptr, *B1hp = nullptr, *Bp = nullptr;
  // device: contraction operands and workspaces
  double* A = nullptr;      // [M][K] FP64 1-halo factor rows
  uint16_t *Ahi = nullptr, *Alo = nullptr;  // [M][K] BF16 split rows (tensor-core form)
  double* Ascale = nullptr; // per-row power-of-two scales of the split rows
  double *G2 = nullptr, *G3 = nullptr, *C2 = nullptr, *C3 = nullptr;  // row-builder factor tables
  // per leg-bin signature s (P: ell bin; B: nl + triangle): F[s][n][q] / 2^E[s][n] in FP32,
  // E[s][n], and the FP64 row-block maximum max_q |F[s][n][q]|
  double *invN = nullptr, *omN = nullptr;  // 1 / N(l^b), Omega / N_tri(t)
  // exact BB+PT couplings (COV_COUPLING_EXACT): per ell bin A one column per
  // pair (Y, Z) of other-leg bins, the int64 Gram matrix of their leg counts
  // (lower half) and kappa = G / (N_tri N_tri') (both halves, FP64)
  int coupling = 0;                 // COV_COUPLING_*
  std::vector<int32_t> kcol_h;      // [ntri][3] column of each leg in its bin
  std::vector<int32_t> kn_h;        // [nl] columns of each bin
  std::vector<int64_t> koff_h;      // [nl + 1] offset of each bin's ncol x ncol block
  std::vector<int32_t> kyz_h;       // per bin, per column: Y, Z
  std::vector<int32_t> ktri_h;      // per bin, per column: its triangle
  std::vector<int64_t> kcoff_h;     // [nl + 1] first column of each bin
  double* kap = nullptr;
  unsigned long long* kgram = nullptr;
  int32_t *kcol = nullptr, *kn = nullptr;
  int64_t* koff = nullptr;
  uint64_t* bmask = nullptr;  // ell bins present in each 32-row block (the product terms skip the rest)
  bool bmask_ready = false;
  int4* gblk = nullptr;       // 32 x 32 sub-blocks of the Gaussian-term diagonal blocks, by first row
  uint32_t* plist = nullptr;  // 32 x 32 lower blocks whose row blocks share an ell bin, (ti << 16) | tj
  std::vector<int64_t> plist_start;  // (host) index of row block ti's first listed block; nb + 1 entries
  bool plist_off = false;     // the list does not serve this layout (more than 64 ell bins or 65536 row blocks)
  std::vector<int64_t> gblk_row;  // (host) first row of each sub-block, ascending
  // launch orders of the tensor-core contraction, by tile-row range
  struct TileOrder {
    int kind = -1, group = 0;
    int64_t t0 = -1, t1 = -1, n = 0;
    int64_t rest = 0, rest_tiles = 0;  // pair tiles of the last, partial wave, and their lower 128 x 128 tiles
    int2* p = nullptr;  // a slot of tile_ring
  } tile_cache[WL_TILE_CACHE];
  int2* tile_ring = nullptr;
  size_t tile_ring_cap = 0;  // entries per slot
  int tile_cache_next = 0;
  float* Fsig = nullptr;
  float* FsigT = nullptr;  // the same for the bin pairs of the trispectrum rows
  int* EsigT = nullptr;
  double* MsigT = nullptr;
  int* Esig = nullptr;
  double* Msig = nullptr;
  int* tc_status = nullptr; // status word of the tensor-core contraction
  int* wait_flag = nullptr; // flag of the bounded-wait self-test
  double* Trows = nullptr;  // [ntrow][K]
  double* Tmat = nullptr;   // [ntrow][ntrow] lower
  uint16_t *Thi = nullptr, *Tlo = nullptr;  // split trispectrum rows (tensor-core form)
  double* Tscale = nullptr;
  double* Srows = nullptr;  // [M][nchi]
  // FP64 form on the tensor cores: digit blocks (with their exponents) and row exponents of the factor rows
  // and the trispectrum rows, the latter's descriptors, and their builders' tables
  uint8_t *Asl = nullptr, *Tsl = nullptr;
  int *Aexp = nullptr, *Texp = nullptr;
  int32_t* trd = nullptr;
  double *sl_w = nullptr, *sl_sr = nullptr;
  unsigned long long* sl_part = nullptr;  // exact partial sums of tiles shared by several CTAs, then their tickets
  int sl_rows = 0, sl_tri = 0;            // 0 undecided, 1 digits, -1 FP64 rows (k_gemm_lower)
  bool sl_reserved = false;               // a server's reservation holds the digits
  double* work = nullptr;   // Cholesky workspace (M+1) rows
  int64_t work_n = 0;
  int64_t work_ld = 0;      // its row length (the last dense cov_snr)
  void* pca_buf = nullptr;  // PCA: G, y and the per-mode arrays
  size_t pca_bytes = 0;
  void* chol_scratch = nullptr;  // Cholesky: digit buffers, diagonal factors, data vector, scaling
  size_t chol_scratch_n = 0;
  size_t chol_scratch_cap = 0;   // bytes it should stay within (the server's reservation; 0: no limit)
  cudaStream_t side = nullptr;   // look-ahead stream of the Cholesky panel kernels
  cudaEvent_t ev_cols = nullptr, ev_panel = nullptr;
  // status words, one allocation (wl_status_words): a non-positive pivot seen, an expired wait in a
  // Cholesky update (both sticky inside a batch), an expired wait in an FP64 contraction since the
  // last call that read the words
  int *piv_status = nullptr, *chol_status = nullptr, *sl_report = nullptr;
  bool spectra_ready = false;
  int row_set = 0, row_order = 0;  // COV_ROWS_*, COV_ORDER_*
  cov_cosmology* cosmo_d = nullptr;  // the cosmology the kernels read (device copy of cosmo)
  bool deferred = false;  // inside a captured batch step: no host synchronisation, no host-side copies
  bool chol_lookahead = true;  // Cholesky panel look-ahead on the side stream
  int chol_kernel = 0;         // Cholesky trailing update: 0 persistent CTAs, 1 one CTA per tile
  int tc_kernel = -1;          // contraction kernel: -1 automatic, 0 one CTA per tile, 1 CTA pairs
  int pr_group = 8;            // tile rows per group of the pair-tile launch order
  struct Selection {           // cumulative S/N selections (P, B, joint; all rows in place)
    bool ready = false;
    int64_t Ms = 0;
    int* perm = nullptr;
    int64_t* cnt = nullptr;
    double* out = nullptr;
  } sel[4];
  double *batch_C = nullptr, *batch_D = nullptr;  // covariance and data vector of cov_batch_snr
  cudaStream_t batch_stream = nullptr;             // cov_batch_snr runs (and captures) on this stream
  cudaEvent_t batch_ev = nullptr;
  int ops_terms = -1, ops_precision = -1;  // operands prepared for the band assembly (-1: none)
  bool prof = false;
  std::vector<StageEvent> pending;
  std::vector<cudaEvent_t> pool;
  double stage_ms[ST_COUNT] = {0};
  int64_t stage_calls[ST_COUNT] = {0};
  std::string err;
};

// ---- host helpers (api.cu) -------------------------------------------------
int wl_fail(cov_handle* h, int code, const std::string& msg);
int wl_cuda(cov_handle* h, cudaError_t e, const char* what);
#define WL_CHECK(h, call)                                 \
  do {                                                    \
    cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) return wl_cuda((h), e_, #call); \
  } while (0)
#define WL_LAUNCH(h, what)                                 \
  do {                                                     \
    cudaError_t e_ = cudaGetLastError();                   \
    if (e_ != cudaSuccess) return wl_cuda((h), e_, (what)); \
  } while (0)

// stage timing: the returned index pairs a begin with its end (-1 = off)
int wl_stage_begin(cov_handle* h, int stage, cudaStream_t s);
void wl_stage_end(cov_handle* h, int token, cudaStream_t s);

// ---- stage entry points (one per translation unit) -------------------------
int wl_quadrature(cov_handle* h, cudaStream_t s);  // tables.cu
int wl_tables(cov_handle* h, cudaStream_t s);   // tables.cu
int wl_triangle_shapes(cov_handle* h, cudaStream_t s);  // spectra.cu: once per handle
int wl_counts(cov_handle* h, cudaStream_t s);   // counts.cu
int wl_couplings(cov_handle* h, cudaStream_t s);  // coupling.cu: exact BB+PT couplings (synchronises s)
void wl_coupling_plan(cov_handle* h);             // coupling.cu: columns per bin (host)
size_t wl_coupling_bytes(const cov_handle* h);    // coupling.cu: resident bytes of the exact couplings
int wl_spectra(cov_handle* h, double* d_D, cudaStream_t s);  // spectra.cu
int wl_assemble(cov_handle* h, double* d_C, int64_t ldc, unsigned terms, int precision, cudaStream_t s);
int wl_snr_tiles(cov_handle* h, double* Ct, const double* D, double* h_snr, cudaStream_t s);  // chol.cu
int wl_assemble_band(cov_handle* h, int64_t row0, int64_t nrows, OutMap out, unsigned terms, int precision,
                     cudaStream_t s);
int wl_snr_prepare(cov_handle* h, cudaStream_t s);  // chol.cu
int wl_status_words(cov_handle* h, cudaStream_t s);  // chol.cu
int wl_snr_status(cov_handle* h, cudaStream_t s);    // chol.cu
int wl_snr(cov_handle* h, const double* d_C, int64_t ldc, const double* d_D, int which, double* h_snr,
           cudaStream_t s, const int* perm = nullptr);  // chol.cu
int wl_gemm_lower_fp64(cov_handle* h, const double* A, int64_t lda, const double* B, int64_t ldb, double* C,
                       int64_t ldc, int64_t n, int64_t k, double alpha, double beta, bool lower_only,
                       cudaStream_t s);  // assemble.cu
int wl_syrk_tc(cov_handle* h, int nssc, OutMap out, cudaStream_t s, int64_t row1 = -1);  // syrk_tc.cu
int wl_syrk_tc_part(cov_handle* h, int nssc, OutMap out, int64_t r0, int64_t r1, cudaStream_t s);
int wl_num_sms();  // chol_fx.cu: SMs of the current device
size_t wl_sl_bytes(const cov_handle* h, bool tri);                                       // syrk_sl.cu
size_t wl_sl_fixed_bytes(const cov_handle* h);                                           // syrk_sl.cu
int wl_sl_alloc(cov_handle* h, bool tri, bool* use, cudaStream_t s);                     // syrk_sl.cu
int wl_sl_rows(cov_handle* h, bool tri, int nssc, cudaStream_t s);                       // syrk_sl.cu
int wl_sl_syrk(cov_handle* h, bool tri, int nssc, OutMap out, int64_t row1, cudaStream_t s);  // syrk_sl.cu
int wl_tc_status_reset(cov_handle* h, cudaStream_t s);
int wl_tc_status_check(cov_handle* h, cudaStream_t s);
int wl_split_bytes(int64_t M, int K, size_t* bytes);                      // syrk_tc.cu
int wl_kpad(int K);  // K padded to the contraction's K granularity
int wl_request_bytes(const cov_nz* nz, const cov_bins* bins, int precision, unsigned terms, int64_t* M,
                     size_t* bytes, bool digits = false);  // api.cu: host-only footprint estimate of one request
size_t wl_handle_bytes(const cov_handle* h);
void wl_set_global_error(const std::string& msg);  // api.cu: read by cov_last_error(NULL)
size_t wl_chol_scratch_est(int64_t n);  // api.cu
size_t wl_late_bytes(const cov_handle* h);  // api.cu: bound of later allocations
bool wl_over_budget(cov_handle* h, size_t extra);  // chol_fx.cu
size_t wl_fx_bytes(int64_t n, int w);  // chol_fx.cu: scratch with super-panels of w panels
int wl_fx_factor(cov_handle* h, OutMap W, int64_t Ms, const int* perm, const double* C, int64_t ldc, const double* D,
                 cudaStream_t s);  // chol_fx.cu
int wl_side_stream(cov_handle* h);  // api.cu: the handle's high-priority side stream
int wl_syrk_tc_rows(cov_handle* h, const void* hi, const void* lo, const double* rscale, int64_t rows, int Kp,
                    OutMap out, cudaStream_t s, int64_t row1 = -1);
// ---- device helpers ------------------------------------------------------------
__device__ __forceinline__ DevCosmo dev_cosmo(const cov_cosmology& c) {
  return DevCosmo{c.Om, c.Ob, c.h, c.ns, c.sigma8, c.w0, c.Tcmb};
}

// d(chi H0 / c) / dy at y = ln(1 + z) for flat w0-CDM: e^y / E, E = H / H0
__device__ __forceinline__ double dev_dchi_dy(double y, const cov_cosmology& c) {
  const double a1 = exp(y);
  return a1 * rsqrt(c.Om * a1 * a1 * a1 + (1.0 - c.Om) * exp(3.0 * (1.0 + c.w0) * y));
}

// ---- chi(z) as a piecewise polynomial in y = ln(1 + z) ------------------------
// chi H0 / c = int e^y / E dy.  [0, ln(1 + z_max)] is cut into WL_N_ZI equal
// intervals, each holding the integrated Chebyshev interpolant of the integrand
// (WL_N_CH nodes).  The integrand's singularities lie at |Im y| ~ 1, so the
// interpolant is good to rounding (its coefficients fall by ~1/190 each at
// z_max = 3, by ~1/39 at z_max = 1000), and one evaluation costs ~25 operations
// where the direct 64-node rule on [0, z] costs 64 evaluations of E.
// sum_k b_k T_k(t), t in [-1, 1], by Clenshaw
__device__ __forceinline__ double dev_clenshaw(const double* b, int n, double t) {
  double u1 = 0.0, u2 = 0.0;
  const double t2 = 2.0 * t;
  for (int k = n - 1; k >= 1; --k) {
    const double u0 = fma(t2, u1, b[k] - u2);
    u2 = u1;
    u1 = u0;
  }
  return fma(t, u1, b[0] - u2);
}
// chi H0 / c at y; cum[j]: the integral up to interval j
__device__ __forceinline__ double dev_chi_unit(double y, double ymax, const double* zint, const double* cum) {
  const double s = y / ymax * WL_N_ZI;
  int j = (int)s;
  j = j < 0 ? 0 : (j > WL_N_ZI - 1 ? WL_N_ZI - 1 : j);
  return cum[j] + dev_clenshaw(zint + j * WL_ZI_STRIDE, WL_N_CH + 1, 2.0 * (s - j) - 1.0);
}

// Eisenstein & Hu (1998) no-wiggle transfer function, k in h/Mpc
__device__ __forceinline__ EhConst dev_eh_const(const cov_cosmology& c) {
  double omh2 = c.Om * c.h * c.h, obh2 = c.Ob * c.h * c.h, fb = c.Ob / c.Om;
  double th = c.Tcmb / 2.7;
  double s = 44.5 * log(9.83 / omh2) / sqrt(1.0 + 10.0 * sqrt(obh2 * sqrt(obh2)));
  double al = 1.0 - 0.328 * log(431.0 * omh2) * fb + 0.38 * log(22.3 * omh2) * fb * fb;
  return EhConst{0.43 * c.h * s, al, c.Om * c.h, th * th};
}

__device__ __forceinline__ double dev_eh_T(double k, const EhConst& e) {
  double ks = k * e.ks;
  double ks2 = ks * ks;
  double geff = e.omh * (e.al + (1.0 - e.al) / (1.0 + ks2 * ks2));
  double q = k * e.th2 / geff;
  double L0 = log(2.0 * 2.718281828459045 + 1.8 * q);
  double C0 = 14.2 + 731.0 / (1.0 + 62.5 * q);
  return L0 / (L0 + C0 * q * q);
}

// k^ns T(k)^2: P_lin = amplitude x this x D^2
__device__ __forceinline__ double dev_plin_unit(double k, const EhConst& e, double ns) {
  double T = dev_eh_T(k, e);
  return pow(k, ns) * T * T;
}

// spherical top-hat window W and its derivative dW (Taylor series below
// x = 0.5); one sine, one cosine and one reciprocal serve both
__device__ __forceinline__ void dev_tophat(double x, double* W, double* dW) {
  if (x < 0.5) {
    // coefficients 3 (-1)^n (2n+2)/(2n+3)!, n = 0..7; the derivative's are 2n times these
    const double c[8] = {1.0, -0.1, 1.0 / 280.0, -1.0 / 15120.0, 1.0 / 1330560.0, -1.0 / 172972800.0,
                         1.0 / 31135104000.0, -1.0 / 7410154752000.0};
    double x2 = x * x, acc = 0.0, dcc = 0.0;
#pragma unroll
    for (int n = 6; n >= 0; --n) acc = acc * x2 + c[n];
#pragma unroll
    for (int n = 7; n >= 1; --n) dcc = dcc * x2 + 2.0 * n * c[n];
    *W = acc;
    *dW = dcc * x;
    return;
  }
  double sx, cx;
  sincos(x, &sx, &cx);
  double iv = 1.0 / x, iv3 = 3.0 * (iv * iv) * iv;
  *W = (sx - x * cx) * iv3;
  *dW = ((x * x - 3.0) * sx + 3.0 * x * cx) * (iv3 * iv);
}

// Auxiliary functions of the sine and cosine integrals (Abramowitz & Stegun
// 5.2.6-5.2.7): f(x) = Ci(x) sin x + (pi/2 - Si(x)) cos x,
// g(x) = -Ci(x) cos x + (pi/2 - Si(x)) sin x, for x >= 4.  x f and x^2 g are
// Stieltjes functions of 1/x^2, so rational forms in 1/x^2 converge fast and
// have positive coefficients only (no cancellation): least-squares fits on
// Chebyshev nodes of (0, 1/16] in 50-digit arithmetic, relative error below
// 2e-17 (f, degree 10) and 8e-18 (g, degree 11).
__device__ __forceinline__ void dev_sici_fg(double x, double ix, double* f, double* g) {
  const double fn[11] = {0.99999999999999998378, 928.05420382076693203, 311792.70383167412804,
                         49241850.478246443474,  3978741250.1625408183, 167994398922.03792598,
                         3636504135501.9774993,  37980955670999.667919, 168886251080155.99331,
                         244439194595624.65367,  50540378205319.638131};
  const double fd[11] = {1.0,
                         930.05420382076576918,
                         313628.81223932914864,
                         49847506.801771428012,
                         4071538491.4537409714,
                         175133077250.8030367,
                         3915194333202.1978355,
                         43309300071250.424812,
                         214523982278849.61302,
                         390009839291757.9415,
                         160657256290782.04942};
  const double gn[12] = {0.99999999999999999237, 1275.0091795677156003, 605421.35439380592647,
                         139649577.9133789602,   17136978224.50301275,  1153313898494.0901147,
                         42382981825994.469923,  821420612961746.69728, 7801194798999991.8498,
                         31529642294798734.145,  39893722197823414.851, 4895049205879604.8997};
  const double gd[12] = {1.0,
                         1281.0091795677148263,
                         612987.40947122489641,
                         143178821.26857615156,
                         17928586069.529463862,
                         1246368476448.8059744,
                         48253850554104.998422,
                         1017580800246133.922,
                         11111072139559062.084,
                         57203395181087421.55,
                         116198203079107446.44,
                         61464150475231224.378};
  const double s = ix * ix;
  double a = fn[10], b = fd[10], c = gn[11], d = gd[11];
#pragma unroll
  for (int i = 9; i >= 0; --i) {
    a = fma(a, s, fn[i]);
    b = fma(b, s, fd[i]);
  }
#pragma unroll
  for (int i = 10; i >= 0; --i) {
    c = fma(c, s, gn[i]);
    d = fma(d, s, gd[i]);
  }
  const double r = 1.0 / (b * d);
  *f = ix * a * (d * r);
  *g = s * c * (b * r);
}

// Si(x) / x and (Ci(x) - gamma - ln x) / x^2 for 0 < x <= 4: entire functions
// of x^2, Chebyshev interpolants of degree 11 (errors below 1e-19) written as
// polynomials.
__device__ __forceinline__ void dev_sici_small(double x2, double* p, double* q) {
  const double P[12] = {1.0,
                        -0.055555555555555554183,
                        0.0016666666666666625773,
                        -0.000028344671201809284662,
                        3.0619243581918498966e-7,
                        -2.2774643976507699453e-9,
                        1.2353110412022082067e-11,
                        -5.0981057067843259861e-14,
                        1.6537641118389194423e-16,
                        -4.3243943635141795944e-19,
                        9.2258372308936945248e-22,
                        -1.4510986112315725863e-24};
  const double Q[12] = {-0.25,
                        0.010416666666666666615,
                        -0.00023148148148148132892,
                        3.1001984126982345943e-6,
                        -2.7557319223878443742e-8,
                        1.739729748606424921e-10,
                        -8.1933896262629766677e-13,
                        2.9871720472757203718e-15,
                        -8.6772094614299662671e-18,
                        2.0543184505162214002e-20,
                        -4.0087791977665931461e-23,
                        5.8582225667303094627e-26};
  double a = P[11], b = Q[11];
#pragma unroll
  for (int i = 10; i >= 0; --i) {
    a = fma(a, x2, P[i]);
    b = fma(b, x2, Q[i]);
  }
  *p = a;
  *q = b;
}

// u(k | m, c) for c < 1 from its defining integral in t = r / r_vir:
// int_0^1 w(t) sinc(K t) dt / int_0^1 w(t) dt, w(t) = t / (1 + c t)^2,
// K = k r_vir, both on one composite 16-point Gauss-Legendre rule (x16, w16
// on [-1, 1]) of ceil(K / (2 pi)) panels: no term cancels, so the result is
// good to rounding where the closed form loses ~1/c^2 of its digits.
__device__ __forceinline__ double dev_nfw_u_integral(double K, double c, const double* x16, const double* w16) {
  const int P = K > 2.0 * WL_PI ? (int)ceil(K / (2.0 * WL_PI)) : 1;
  const double hp = 1.0 / P;
  double num = 0.0, den = 0.0;
  for (int p = 0; p < P; ++p)
    for (int i = 0; i < 16; ++i) {
      const double t = (p + 0.5 * (x16[i] + 1.0)) * hp;
      const double ct = 1.0 + c * t;
      const double wt = w16[i] * t / (ct * ct);
      const double Kt = K * t;
      num += wt * sin(Kt) / Kt;
      den += wt;
    }
  return num / den;
}

// Normalised Fourier transform u(k | m, c) of the truncated NFW profile
// (200 x mean-density mass) with K = k r_vir, the concentration c and
// l1 = ln(1 + c), inorm = 1 / (l1 - c / (1 + c)).  For c >= 1, with x = K / c:
//   u inorm^-1 = sin x (Si(x + K) - Si(x)) + cos x (Ci(x + K) - Ci(x)) - sin K / (x + K).
// The angle of the second argument minus that of the first is K, so where
// x + K >= 4 the auxiliary functions leave
//   g(x) + (f(x + K) - 1 / (x + K)) sin K - g(x + K) cos K,
// with g(x) from its definition for x < 4; below, Ci(x + K) - Ci(x) is
// ln(1 + c) plus two entire functions.  c < 1: the defining integral.
__device__ __forceinline__ double dev_nfw_u(double K, double c, double l1, double inorm, const double* x16,
                                            const double* w16) {
  if (c < WL_NFW_C_INTEGRAL) return dev_nfw_u_integral(K, c, x16, w16);
  const double x = K / c, x2 = x + K;
  double sK, cK, num;
  sincos(K, &sK, &cK);
  const double i2 = 1.0 / x2;
  if (x2 >= 4.0) {
    double f2, g2, g1;
    dev_sici_fg(x2, i2, &f2, &g2);
    if (x >= 4.0) {
      double f1;
      dev_sici_fg(x, c / K, &f1, &g1);
    } else {
      double p, q, sx, cx;
      dev_sici_small(x * x, &p, &q);
      sincos(x, &sx, &cx);
      g1 = (0.5 * WL_PI - x * p) * sx - (WL_EULER_GAMMA + log(x) + x * x * q) * cx;
    }
    num = g1 + (f2 - i2) * sK - g2 * cK;
  } else {
    double p1, q1, p2, q2, sx, cx;
    dev_sici_small(x * x, &p1, &q1);
    dev_sici_small(x2 * x2, &p2, &q2);
    sincos(x, &sx, &cx);
    num = sx * (x2 * p2 - x * p1) + cx * (l1 + (x2 * x2 * q2 - x * x * q1)) - sK * i2;
  }
  return num * inorm;
}

// RN(a) 2^ex as an FP64 value for 0 < |a| < 2^63, without branches on the
// value: normalise |a| so that its leading bit is bit 63, keep the 53 leading
// bits rounded to nearest (ties to even), and add the rounded significand
// (2^52 <= r <= 2^53) to the biased exponent field, which carries a rounding
// overflow into the exponent by itself.  Results outside the normal range take
// the FP64 path.
__device__ __forceinline__ double scaled_to_double_rn(long long a, int ex) {
  if (a == 0) return 0.0;
  const unsigned long long sign = (unsigned long long)a & (1ull << 63);
  const unsigned long long u = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
  const int lz = __clzll((long long)u);
  const unsigned long long mn = u << lz;
  const unsigned long long r0 = mn >> 11;
  const unsigned long long rb = (mn >> 10) & 1ull;
  const unsigned long long sticky = ((mn & 0x3FFull) != 0ull) | (r0 & 1ull);
  const unsigned long long r = r0 + (rb & sticky);
  const int e = (63 - lz) + ex + 1023;
  if (e <= 0 || e >= 2046) return ldexp((double)a, ex);
  return __longlong_as_double((long long)(sign | (((unsigned long long)(e - 1) << 52) + r)));
}

// Scale of a covariance row for the fixed-point Cholesky: 1 / sqrt(d) of the variance d,
// rounded down to 24 significant bits less one in the last, so that d s^2 is in (1 - 2^-21, 1)
// and the product of two scales is exact; 0 for d that is no positive finite number
__device__ __forceinline__ double variance_scale(double d) {
  if (!(d > 0.0 && isfinite(d))) return 0.0;
  return __longlong_as_double((__double_as_longlong(1.0 / sqrt(d)) & ~0x1FFFFFFFll) - 0x20000000ll);
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_max(double v) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// block-wide sum for blockDim.x a multiple of 32 (<= 1024); result on all threads
__device__ __forceinline__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  int nw = (blockDim.x + 31) >> 5;
  double t = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
  if (w == 0) t = warp_sum(t);
  if (threadIdx.x == 0) sh[0] = t;
  __syncthreads();
  double r = sh[0];
  __syncthreads();
  return r;
}
