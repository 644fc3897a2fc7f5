// Table builder: background, growth, linear power, halo model, profiles,
// lensing kernels and sigma_W^2 on the device (paper Secs. 2 and 4,
// Appendices A and B).  Every kernel writes FP64 tables laid out chi-major
// (node index outermost, mass index contiguous) so that the row builders read
// them coalesced.
#include "common.cuh"

// Gauss-Legendre nodes/weights on [-1, 1] by Newton iteration on P_n with the
// three-term recurrence; nodes ascending.
__global__ void k_gauss_legendre(int n, double* x, double* w) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double zz = cos(WL_PI * (i + 0.75) / (n + 0.5));
  double pp = 1.0;
  // Newton from the cosine guess: quadratic convergence reaches double
  // precision in a handful of steps; stop at 5e-16 or after 10 steps
  for (int it = 0; it < 10; ++it) {
    double p1 = 1.0, p2 = 0.0;
    for (int j = 1; j <= n; ++j) {
      double p3 = p2;
      p2 = p1;
      p1 = ((2.0 * j - 1.0) * zz * p2 - (j - 1.0) * p3) / j;
    }
    pp = n * (zz * p1 - p2) / (zz * zz - 1.0);
    double z1 = zz;
    zz = z1 - p1 / pp;
    if (fabs(zz - z1) <= 5e-16) break;
  }
  double p1 = 1.0, p2 = 0.0;
  for (int j = 1; j <= n; ++j) {
    double p3 = p2;
    p2 = p1;
    p1 = ((2.0 * j - 1.0) * zz * p2 - (j - 1.0) * p3) / j;
  }
  pp = n * (zz * p1 - p2) / (zz * zz - 1.0);
  x[i] = -zz;
  w[i] = 2.0 / ((1.0 - zz * zz) * pp * pp);
}

// Normalised probabilists' Hermite polynomials h_k = He_k / sqrt(k!) by the
// three-term recurrence h_{k+1} = (x h_k - sqrt(k) h_{k-1}) / sqrt(k+1),
// h_0 = 1, h_1 = x.  Returns h_n(x) and h_{n-1}(x) in *prev (n >= 1).
__device__ double dev_hermite_h(int n, double x, double* prev) {
  double p0 = 1.0, p1 = x;
  for (int k = 1; k < n; ++k) {
    double p2 = (x * p1 - sqrt((double)k) * p0) / sqrt(k + 1.0);
    p0 = p1;
    p1 = p2;
  }
  *prev = p0;
  return p1;
}

#define WL_GH_GRID 1023
// Concentration rule of Eq. LogNormC (one block of 256 threads): Gauss-Hermite
// nodes x_j and weights w_j of the standard normal density (sum w_j = 1),
// written as ln c offsets cs[j] = sigma x_j and weights cw[j].  The roots of
// He_n lie in |x| < sqrt(4n + 2); the grid of WL_GH_GRID intervals on that
// range is finer than their spacing for n <= 32, so each interval holds at
// most one root.  Each root is bisected to the last bit and weighted by
// w = 1 / (n h_{n-1}(x)^2).  n <= 1: one node, offset 0, weight 1.  A rule
// that does not find n roots is written with NaN weights.
__global__ void k_gauss_hermite(int n, double sigma, double* cs, double* cw) {
  __shared__ double root[WL_GH_GRID];
  if (n <= 1) {
    if (threadIdx.x == 0) {
      cs[0] = 0.0;
      cw[0] = 1.0;
    }
    return;
  }
  const double L = sqrt(4.0 * n + 2.0) + 0.5, dx = 2.0 * L / WL_GH_GRID;
  double pr;
  for (int i = threadIdx.x; i < WL_GH_GRID; i += blockDim.x) {
    double xa = -L + i * dx, xb = -L + (i + 1) * dx;
    double va = dev_hermite_h(n, xa, &pr), vb = dev_hermite_h(n, xb, &pr);
    double r = nan("");
    if (va == 0.0) {
      r = xa;  // a root on the left end; one on the right end belongs to the next interval
    } else if (vb != 0.0 && (va < 0.0) != (vb < 0.0)) {
      double lo = xa, hi = xb;
      for (int it = 0; it < 200; ++it) {
        double mid = 0.5 * (lo + hi);
        if (mid <= lo || mid >= hi) break;
        double vm = dev_hermite_h(n, mid, &pr);
        if (vm == 0.0) {
          lo = hi = mid;
          break;
        }
        if ((vm < 0.0) == (va < 0.0))
          lo = mid;
        else
          hi = mid;
      }
      r = 0.5 * (lo + hi);
    }
    root[i] = r;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int found = 0;
    for (int i = 0; i < WL_GH_GRID; ++i) {
      if (root[i] != root[i]) continue;
      if (found < n) {
        double hprev;
        dev_hermite_h(n, root[i], &hprev);
        cs[found] = sigma * root[i];
        cw[found] = 1.0 / (n * hprev * hprev);
      }
      ++found;
    }
    if (found != n)
      for (int j = 0; j < n; ++j) cw[j] = nan("");
  }
}


// ---- growth -------------------------------------------------------------------
// The linear growth ODE in ln a, D'' = -(2 + dlnH) D' + 1.5 Om(a) D, by WL_N_RK4
// Runge-Kutta steps from a = WL_A_INIT (D = D' = a) to a_t.  The ODE is linear,
// so a step is a 2 x 2 matrix that depends on a alone: each of the block's
// threads carries the two unit vectors through its own run of steps, and the
// matrices are multiplied in order by shuffles.  The sequential chain of 1024
// steps (~3 ms on one thread: a dependent FP64 operation takes 64 cycles here)
// becomes 8 steps and 7 products; the steps are those of the sequential rule.
#define GR_THREADS 128
__device__ __forceinline__ void growth_coef(double am, double ad, double om, double ode, double w3, double* A,
                                            double* B) {
  const double em = om * am, ed = ode * ad, inv = 1.0 / (em + ed);
  *A = -(2.0 + 0.5 * (-3.0 * em - w3 * ed) * inv);
  *B = 1.5 * em * inv;
}

struct GrowthMat {
  double d0, p0, d1, p1;  // images of (D, D') = (1, 0) and (0, 1)
};

__device__ __forceinline__ GrowthMat growth_after(const GrowthMat& l, const GrowthMat& e) {  // l after e
  return GrowthMat{fma(l.d0, e.d0, l.d1 * e.p0), fma(l.p0, e.d0, l.p1 * e.p0), fma(l.d0, e.d1, l.d1 * e.p1),
                   fma(l.p0, e.d1, l.p1 * e.p1)};
}

// D and D' at a_t; every one of the GR_THREADS threads of the block calls it and receives the result
__device__ void block_growth(double at, const cov_cosmology& c, double* D, double* Dp) {
  __shared__ GrowthMat sh[GR_THREADS / 32];
  constexpr int PER = WL_N_RK4 / GR_THREADS;
  const double x0 = log(WL_A_INIT), h = (log(at) - x0) / WL_N_RK4;
  const double om = c.Om, ode = 1.0 - c.Om, w3 = 3.0 * (1.0 + c.w0);
  const double qm = exp(-1.5 * h), qd = exp(-0.5 * w3 * h);  // a^-3 and a^(-3(1+w)) over half a step
  const double xs = x0 + h * (double)(threadIdx.x * PER);
  double am = exp(-3.0 * xs), ad = exp(-w3 * xs), A0, B0;
  growth_coef(am, ad, om, ode, w3, &A0, &B0);
  double v[2][2] = {{1.0, 0.0}, {0.0, 1.0}};
  const double hh = 0.5 * h, h6 = h / 6.0;
#pragma unroll 1
  for (int s = 0; s < PER; ++s) {
    double Ah, Bh, A1, B1;
    const double amh = am * qm, adh = ad * qd;
    am = amh * qm;
    ad = adh * qd;
    growth_coef(amh, adh, om, ode, w3, &Ah, &Bh);
    growth_coef(am, ad, om, ode, w3, &A1, &B1);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const double d = v[i][0], p = v[i][1];
      const double k1p = fma(A0, p, B0 * d);
      const double k2d = fma(hh, k1p, p), k2p = fma(Ah, k2d, Bh * fma(hh, p, d));
      const double k3d = fma(hh, k2p, p), k3p = fma(Ah, k3d, Bh * fma(hh, k2d, d));
      const double k4d = fma(h, k3p, p), k4p = fma(A1, k4d, B1 * fma(h, k3d, d));
      v[i][0] = fma(h6, p + 2.0 * (k2d + k3d) + k4d, d);
      v[i][1] = fma(h6, k1p + 2.0 * (k2p + k3p) + k4p, p);
    }
    A0 = A1;
    B0 = B1;
  }
  GrowthMat m{v[0][0], v[0][1], v[1][0], v[1][1]};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {  // lane i holds the steps of lanes i .. i + 2 o - 1 after the round
    GrowthMat l;
    l.d0 = __shfl_down_sync(0xffffffffu, m.d0, o);
    l.p0 = __shfl_down_sync(0xffffffffu, m.p0, o);
    l.d1 = __shfl_down_sync(0xffffffffu, m.d1, o);
    l.p1 = __shfl_down_sync(0xffffffffu, m.p1, o);
    m = growth_after(l, m);
  }
  __syncthreads();  // an earlier call's readers are done
  if (lane == 0) sh[warp] = m;
  __syncthreads();
  double d = WL_A_INIT, p = WL_A_INIT;
#pragma unroll
  for (int w = 0; w < GR_THREADS / 32; ++w) {
    const double nd = fma(sh[w].d0, d, sh[w].d1 * p);
    p = fma(sh[w].p0, d, sh[w].p1 * p);
    d = nd;
  }
  *D = d;
  *Dp = p;
}

// ---- survey: equipopulated edges, bin normalisations, lensing kernels ----
__device__ __forceinline__ double cdf15(double z, double z0) {
  double x = z / z0 * sqrt(z / z0);
  return 1.0 - (1.0 + x) * exp(-x);
}

__device__ __forceinline__ double nz_shape(double z, const cov_nz& nz) {
  const double x = z / nz.z0;  // alpha is 1.5 (checked at cov_init)
  return z * z * exp(-x * sqrt(x));
}

__device__ __forceinline__ double bin_sel(double z, int i, const double* e, int nt, double s0) {
  double lo = e[i], hi = e[i + 1];
  if (s0 == 0.0) {
    bool last = (i == nt - 1);
    return (z >= lo && (last ? z <= hi : z < hi)) ? 1.0 : 0.0;
  }
  double s = sqrt(2.0) * s0 * (1.0 + z);
  return 0.5 * (erf((hi - z) / s) - erf((lo - z) / s));
}

__global__ void k_edges(cov_nz nz, double* e, double* scal) {
  int t = threadIdx.x;
  int nt = nz.n_tomo;
  if (t > nt) return;
  if (t == 0) {
    e[0] = nz.zmin;
    double nbar = nz.n_gal_arcmin2 * (10800.0 / WL_PI) * (10800.0 / WL_PI) / nt;
    scal[SC_NOISE] = nz.sigma_e * nz.sigma_e / nbar;
    return;
  }
  if (t == nt) {
    e[nt] = nz.zmax;
    return;
  }
  double g0 = cdf15(nz.zmin, nz.z0), g1 = cdf15(nz.zmax, nz.z0);
  double target = (double)t / nt, lo = nz.zmin, hi = nz.zmax;
  for (int it = 0; it < 200; ++it) {
    double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if ((cdf15(mid, nz.z0) - g0) / (g1 - g0) < target)
      lo = mid;
    else
      hi = mid;
  }
  e[t] = 0.5 * (lo + hi);
}

// pieces of [a, b] split at the edges strictly inside it; returns the count
__device__ __forceinline__ int make_pieces(double a, double b, const double* e, int nt, double* pts) {
  int np = 0;
  pts[np++] = a;
  for (int i = 0; i <= nt; ++i)
    if (e[i] > a && e[i] < b) pts[np++] = e[i];
  pts[np++] = b;
  return np - 1;
}

__global__ void k_norms(cov_nz nz, const double* e, const double* gx, const double* gw, double* norms) {
  __shared__ double sh[32];
  int i = blockIdx.x, nt = nz.n_tomo;
  double pts[40];
  int np = make_pieces(nz.zmin, nz.zmax, e, nt, pts);
  double s = 0.0;
  for (int p = 0; p < np; ++p) {
    double a = pts[p], b = pts[p + 1], half = 0.5 * (b - a);
    for (int j = threadIdx.x; j < WL_N_ZS; j += blockDim.x) {
      double zz = a + half * (gx[j] + 1.0);
      s += half * gw[j] * nz_shape(zz, nz) * bin_sel(zz, i, e, nt, nz.photoz_sigma0);
    }
  }
  s = block_sum(s, sh);
  if (threadIdx.x == 0) norms[i] = s;
}


// ---- tables that depend on the binning and n(z) only (made once per handle) ----
// Source nodes of the pieces [e_k, e_(k+1)] between neighbouring edges and their
// weights w n(z) P_i(z); the lensing kernels use them for every piece that
// starts at an edge.
__global__ void k_sources(cov_nz nz, const double* e, const double* gx, const double* gw, double* zs, double* gsel) {
  const int k = blockIdx.x, j = threadIdx.x, nt = nz.n_tomo;
  if (j >= WL_N_ZS) return;
  const double half = 0.5 * (e[k + 1] - e[k]), z = e[k] + half * (gx[j] + 1.0);
  const double g = half * gw[j] * nz_shape(z, nz);
  zs[k * WL_N_ZS + j] = z;
  for (int i = 0; i < nt; ++i) gsel[(size_t)(k * WL_N_ZS + j) * nt + i] = g * bin_sel(z, i, e, nt, nz.photoz_sigma0);
}

// k nodes of the sigma(R) and sigma_W^2 rules with their weights, and the
// Chebyshev matrix of the chi intervals
__global__ void k_static_nodes(const double* glkx, const double* glkw, double* kn, double* kwt, double* kw8,
                               double* kws, double* chebm) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < WL_N_CH * WL_N_CH) {  // a_k = sum_i chebm[k][i] f(t_i), t_i = cos(pi (i + 1/2) / n)
    const int k = i / WL_N_CH, n = i % WL_N_CH;
    chebm[i] = (k == 0 ? 1.0 : 2.0) / WL_N_CH * cospi((double)((2 * n + 1) * k) / (2 * WL_N_CH));
  }
  if (i >= WL_N_K) return;
  const double half = 0.5 * (WL_LNK_MAX - WL_LNK_MIN), k = exp(WL_LNK_MIN + half * (glkx[i] + 1.0));
  const double w = half * glkw[i];
  double W, dW;
  dev_tophat(8.0 * k, &W, &dW);
  kn[i] = k;
  kwt[i] = w * k * k * k / (2.0 * WL_PI * WL_PI);
  kw8[i] = kwt[i] * W * W;
  kws[i] = w * k * k;
}

// mass nodes and weights; m, om per (mass, concentration) node, om times the c
// weight; the mass factor of the Duffy median
__global__ void k_mass_nodes(cov_bins b, int nc, const double* cw, double* mb, double* omb, double* m, double* om,
                             double* cmass) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= b.n_mass) return;
  const double dl = log(b.m_max / b.m_min) / (b.n_mass - 1), mq = b.m_min * exp(dl * q);
  double w = dl * mq;
  if (q == 0 || q == b.n_mass - 1) w *= 0.5;
  mb[q] = mq;
  omb[q] = w;
  cmass[q] = WL_DUFFY_A * pow(mq / WL_DUFFY_MPIVOT, WL_DUFFY_B);
  for (int j = 0; j < nc; ++j) {
    m[q * nc + j] = mq;
    om[q * nc + j] = w * cw[j];
  }
}

// ---- per cosmology --------------------------------------------------------------
// First launch: blocks 0 .. WL_N_ZI - 1 build the chi intervals; the others the
// linear spectrum k^ns T^2 on the k nodes and their partial sigma_8 sums.
__global__ void __launch_bounds__(WL_KT_THREADS)
    k_prep(const cov_cosmology* __restrict__ cosmo_p, double ymax, const double* __restrict__ chebm,
           const double* __restrict__ kn, const double* __restrict__ kw8, double* zint, double* pk, double* part) {
  __shared__ double sh[32];
  const cov_cosmology c = *cosmo_p;
  if (blockIdx.x < WL_N_ZI) {
    const int j = blockIdx.x, n = threadIdx.x;
    const double hw = 0.5 * ymax / WL_N_ZI;
    double* o = zint + j * WL_ZI_STRIDE;
    if (n < WL_N_CH) {  // t_n = cos(pi (n + 1/2) / 12) = the k = 1 row of the matrix times 12 / 2
      const double t = chebm[WL_N_CH + n] * (0.5 * WL_N_CH);
      sh[n] = hw * dev_dchi_dy((2 * j + 1 + t) * hw, c);
    }
    __syncwarp();
    double a = 0.0;
    if (n < WL_N_CH)
#pragma unroll
      for (int i = 0; i < WL_N_CH; ++i) a = fma(chebm[n * WL_N_CH + i], sh[i], a);
    if (n < 32) {
      // integral from t = -1: b_k = (a_(k-1) - a_(k+1)) / (2 k), b_1 with 2 a_0; b_0 makes it vanish at -1
      const double lo = __shfl_up_sync(0xffffffffu, a, 1), hi = __shfl_down_sync(0xffffffffu, a, 1);
      double b = 0.0;
      if (n >= 1 && n <= WL_N_CH) b = ((n == 1 ? 2.0 * lo : lo) - (n < WL_N_CH - 1 ? hi : 0.0)) / (2.0 * n);
      const double alt = warp_sum((n & 1) ? b : -b), tot = warp_sum(b);
      if (n <= WL_N_CH) o[n] = n == 0 ? alt : b;
      if (n < WL_N_CH) o[WL_ZI_DER + n] = a;
      if (n == 0) o[WL_ZI_TOT] = alt + tot;
    }
    return;
  }
  const int i = (blockIdx.x - WL_N_ZI) * WL_KT_THREADS + threadIdx.x;
  const EhConst e = dev_eh_const(c);
  const double p = dev_plin_unit(kn[i], e, c.ns);
  pk[i] = p;
  const double s = block_sum(p * kw8[i], sh);
  if (threadIdx.x == 0) part[blockIdx.x - WL_N_ZI] = s;
}

// Integrals up to each chi interval (inclusive scan of the interval totals) in
// shared memory, for a block of at least WL_N_ZI threads; returns chi(z_max) H0 / c
__device__ __forceinline__ double chi_cum(const double* __restrict__ zint, double* cum) {
  const int t = threadIdx.x, lane = t & 31;
  double v = 0.0;
  if (t < WL_N_ZI) {
    v = zint[t * WL_ZI_STRIDE + WL_ZI_TOT];
    for (int o = 1; o < 32; o <<= 1) {
      const double u = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += u;
    }
    cum[t + 1] = v;
  }
  if (t == 0) cum[0] = 0.0;
  __syncthreads();
  if (t >= 32 && t < WL_N_ZI) cum[t + 1] += cum[32];
  __syncthreads();
  return cum[WL_N_ZI];
}

// amplitude of the linear spectrum from the partial sums (every lane of a warp)
__device__ __forceinline__ double plin_amp(const double* __restrict__ part, double sigma8) {
  double s = 0.0;
  for (int i = threadIdx.x & 31; i < WL_N_K / WL_KT_THREADS; i += 32) s += part[i];
  return sigma8 * sigma8 / warp_sum(s);
}

struct NodeArgs {
  const cov_cosmology* cosmo;
  cov_bins b;
  int nchi, nsrc;
  double ymax, theta;
  const double *glcx, *glcw, *zint, *part, *kn, *kwt, *kws, *pk, *mb, *zsrc;
  double *scal, *chi, *wchi, *z, *Draw, *cz, *sig0, *dlns, *sigF, *rvir, *sigw2, *chis;
  double* ksum;
  int* ticket;
};

// The sums over the 4096 k nodes (one per mass and one per line-of-sight node) are
// each cut over WL_KSPLIT blocks, so that few nodes still spread over the SMs (64
// nodes: 128 us for the launch uncut, its longest block 32 k nodes per thread).
// Thread 0 of each block delivers its part; the one that delivers last adds the
// parts in their fixed order into v[0..2] and gets true.
__device__ __forceinline__ bool ksum_last(const NodeArgs& A, int id, int part, double* v) {
  double* p = A.ksum + (size_t)id * WL_KSPLIT * 3;
  for (int i = 0; i < 3; ++i) __stcg(p + part * 3 + i, v[i]);
  __threadfence();
  if (atomicAdd(A.ticket + id, 1) != WL_KSPLIT - 1) return false;
  __threadfence();
  for (int i = 0; i < 3; ++i) {
    v[i] = 0.0;
    for (int k = 0; k < WL_KSPLIT; ++k) v[i] += __ldcg(p + k * 3 + i);
  }
  A.ticket[id] = 0;
  return true;
}

// Second launch, by block: nchi + 1 line-of-sight nodes (the last: the growth to
// a = 1), WL_KSPLIT blocks for each of the nmb mass nodes (sigma,
// d ln sigma / d ln m, r_vir; for the Bullock median also sigma(F m), the variance
// of the collapsing mass) and of the nchi sigma_W^2 (Appendix B, before its D^2),
// and the source nodes' chi.
// All are independent and FP64-bound; together they fill the SMs.
__global__ void __launch_bounds__(GR_THREADS) k_nodes(NodeArgs A) {
  __shared__ double sh[32], cum[WL_N_ZI + 1];
  const cov_cosmology c = *A.cosmo;
  int blk = blockIdx.x;
  if (blk <= A.nchi) {  // line-of-sight nodes: chi_n (Gauss-Legendre on [0, chi_max]), weights, z(chi_n), D(z_n)
    const int n = blk;
    const double um = chi_cum(A.zint, cum);
    double zz = 0.0, ch = 0.0;
    if (n < A.nchi) {
      const double u = 0.5 * um * (A.glcx[n] + 1.0), dy = A.ymax / WL_N_ZI;
      ch = WL_C_OVER_H0 * u;
      int j = 0;
      for (int i = 32; i > 0; i >>= 1)
        if (j + i < WL_N_ZI && cum[j + i] <= u) j += i;
      // Newton on the interval's polynomial (its derivative is the integrand's interpolant)
      const double* o = A.zint + j * WL_ZI_STRIDE;
      double t = 2.0 * (u - cum[j]) / (cum[j + 1] - cum[j]) - 1.0;
      for (int it = 0; it < 8; ++it) {
        const double st = (cum[j] + dev_clenshaw(o, WL_N_CH + 1, t) - u) / dev_clenshaw(o + WL_ZI_DER, WL_N_CH, t);
        t -= st;
        if (fabs(st) < 1e-15) break;
      }
      zz = expm1(dy * (j + 0.5 * (t + 1.0)));
    }
    double D, Dp;
    block_growth(1.0 / (1.0 + zz), c, &D, &Dp);
    if (threadIdx.x == 0) {
      if (n == A.nchi) {
        A.scal[SC_D1] = D;
        A.scal[SC_CHIMAX] = WL_C_OVER_H0 * um;
      } else {
        A.chi[n] = ch;
        A.wchi[n] = 0.5 * (WL_C_OVER_H0 * um) * A.glcw[n];
        A.z[n] = zz;
        A.Draw[n] = D;
        A.cz[n] = pow(1.0 + zz, WL_DUFFY_C);
      }
    }
    return;
  }
  blk -= A.nchi + 1;
  constexpr int SPAN = WL_N_K / WL_KSPLIT;
  const int part = blk % WL_KSPLIT, i0 = part * SPAN;
  blk /= WL_KSPLIT;
  if (blk < A.b.n_mass) {  // one mass node
    const double rho = WL_RHO_CRIT0 * c.Om, mq = A.mb[blk];
    const double R = cbrt(3.0 * mq / (4.0 * WL_PI * rho));
    const bool bullock = A.b.conc_model == COV_CONC_BULLOCK;
    const double RF = cbrt(3.0 * (WL_BULLOCK_F * mq) / (4.0 * WL_PI * rho));
    double s2 = 0.0, ds2 = 0.0, s2F = 0.0;
    for (int i = i0 + threadIdx.x; i < i0 + SPAN; i += GR_THREADS) {
      const double k = A.kn[i], d2 = A.kwt[i] * A.pk[i];
      double W, dW;
      dev_tophat(k * R, &W, &dW);
      s2 = fma(d2, W * W, s2);
      ds2 = fma(2.0 * d2 * k, W * dW, ds2);
      if (bullock) {
        dev_tophat(k * RF, &W, &dW);
        s2F = fma(d2, W * W, s2F);
      }
    }
    double v[3] = {block_sum(s2, sh), block_sum(ds2, sh), bullock ? block_sum(s2F, sh) : 0.0};
    if (threadIdx.x < 32) {
      const double amp = plin_amp(A.part, c.sigma8);
      if (threadIdx.x == 0 && ksum_last(A, blk, part, v)) {
        A.sig0[blk] = sqrt(amp * v[0]);
        A.dlns[blk] = (R / 6.0) * v[1] / v[0];
        if (bullock) A.sigF[blk] = sqrt(amp * v[2]);
        A.rvir[blk] = cbrt(3.0 * mq / (4.0 * WL_PI * WL_DELTA_VIR * rho));
        if (blk == 0) A.scal[SC_AMP] = amp;
      }
    }
    return;
  }
  blk -= A.b.n_mass;
  if (blk < A.nchi) {  // sigma_W^2 of a disk of angular radius Theta
    const double cm = WL_C_OVER_H0 * chi_cum(A.zint, cum);
    const double xs = 0.5 * cm * (A.glcx[blk] + 1.0) * A.theta;
    double s = 0.0;
    for (int i = i0 + threadIdx.x; i < i0 + SPAN; i += GR_THREADS) {
      const double x = A.kn[i] * xs, win = j1(x) / x;
      s = fma(A.kws[i] * A.pk[i], win * win, s);
    }
    double v[3] = {block_sum(s, sh), 0.0, 0.0};
    if (threadIdx.x < 32) {
      const double amp = plin_amp(A.part, c.sigma8);
      if (threadIdx.x == 0 && ksum_last(A, A.b.n_mass + blk, part, v))
        A.sigw2[blk] = 4.0 / (2.0 * WL_PI) * amp * v[0];
    }
    return;
  }
  blk = (blk - A.nchi) * WL_KSPLIT + part;
  // chi at the source nodes
  chi_cum(A.zint, cum);
  const int i = blk * GR_THREADS + threadIdx.x;
  if (i < A.nsrc) A.chis[i] = WL_C_OVER_H0 * dev_chi_unit(log1p(A.zsrc[i]), A.ymax, A.zint, cum);
}

struct HaloArgs {
  const cov_cosmology* cosmo;
  cov_bins b;
  cov_nz nz;
  int nchi, nc, nl;
  double ymax, st_amp;
  const double *scal, *chi, *z, *Draw, *mb, *omb, *sig0, *dlns, *sigF, *zedges, *norms, *gsel, *chis;
  const double *zint, *gx, *gw, *ell;
  double *D, *f, *b1, *b2, *W, *sigw2, *ac, *Pl, *dPl, *Psh;
};

// Collapse epoch of the Bullock et al. median (Sec. 5.4): a_c with
// D(a_c) sigma(F m, 0) = delta_c, D(1) = 1, D the growth rule's value.  Newton in
// ln a (the rule carries D' along) inside a shrinking bracket, bisecting where a
// step would leave it.  a_c = WL_A_COLLAPSE_MAX where D stays below the target
// up to there; the start of the growth rule where D starts above it.
__device__ double block_collapse(const HaloArgs& A, const cov_cosmology& c, int q) {
  const double d1 = A.scal[SC_D1], target = WL_DELTA_C / A.sigF[q] * d1;
  double D, Dp;
  block_growth(WL_A_COLLAPSE_MAX, c, &D, &Dp);
  if (D <= target) return WL_A_COLLAPSE_MAX;
  if (WL_A_INIT >= target) return WL_A_INIT;
  double lo = log(WL_A_INIT), hi = log(WL_A_COLLAPSE_MAX);
  double x = log(target);  // D ~ a in matter domination
  if (!(x > lo && x < hi)) x = 0.5 * (lo + hi);
  for (int it = 0; it < 60; ++it) {
    block_growth(exp(x), c, &D, &Dp);
    if (D >= target)
      hi = x;
    else
      lo = x;
    double nx = x - (D - target) / Dp;
    if (fabs(nx - x) <= 4e-15 * fmax(1.0, fabs(x))) {  // Newton's next step would be below rounding
      x = nx;
      break;
    }
    if (!(nx > lo && nx < hi)) nx = 0.5 * (lo + hi);
    x = nx;
  }
  return exp(x);
}

// Third launch, by block: nmb collapse epochs (Bullock only), nchi lensing kernels,
// nchi halo nodes, and the linear spectra on the Limber grid (8 lanes per point).
__global__ void __launch_bounds__(GR_THREADS) k_halo(HaloArgs A) {
  __shared__ double sh[32], cum[WL_N_ZI + 1], shw[4][32];
  const cov_cosmology c = *A.cosmo;
  int blk = blockIdx.x;
  const int nm = A.b.n_mass, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (A.b.conc_model == COV_CONC_BULLOCK) {
    if (blk < nm) {
      const double a = block_collapse(A, c, blk);
      if (threadIdx.x == 0) A.ac[blk] = a;
      return;
    }
    blk -= nm;
  }
  if (blk < A.nchi) {
    // W_i(chi_n): the piece from z_n to the next edge has its own source nodes;
    // every later piece runs from edge to edge on the shared ones, whose chi,
    // n(z) and bin probabilities do not depend on n.  One source per thread.
    const int n = blk, nt = A.nz.n_tomo;
    const double ch = A.chi[n], zn = A.z[n];
    chi_cum(A.zint, cum);
    double acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.0;
    const bool any = zn < A.nz.zmax;
    int k1 = nt;  // first edge above z_n
    for (int i = nt; i >= 0; --i)
      if (A.zedges[i] > zn) k1 = i;
    if (any) {
      if (threadIdx.x < WL_N_ZS) {
        const double half = 0.5 * (A.zedges[k1] - zn), zs = zn + half * (A.gx[threadIdx.x] + 1.0);
        const double cs = WL_C_OVER_H0 * dev_chi_unit(log1p(zs), A.ymax, A.zint, cum);
        const double geo = half * A.gw[threadIdx.x] * nz_shape(zs, A.nz) * (cs - ch) / cs;
        if (A.nz.photoz_sigma0 == 0.0) {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (i < nt) acc[i] = geo * bin_sel(zs, i, A.zedges, nt, 0.0);
        } else {
          // neighbouring bins share an edge: one error function per edge
          const double is = 1.0 / (sqrt(2.0) * A.nz.photoz_sigma0 * (1.0 + zs));
          double lo = erf((A.zedges[0] - zs) * is);
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (i < nt) {
              const double v = (A.zedges[i + 1] - zs) * is, hi = fabs(v) >= 6.0 ? copysign(1.0, v) : erf(v);
              acc[i] = geo * (0.5 * (hi - lo));
              lo = hi;
            }
        }
      }
      for (int s = k1 * WL_N_ZS + threadIdx.x; s < nt * WL_N_ZS; s += GR_THREADS) {
        const double cs = A.chis[s], geo = (cs - ch) / cs;
        const double* g = A.gsel + (size_t)s * nt;
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (i < nt) acc[i] = fma(geo, g[i], acc[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (i < nt) {
        const double s = warp_sum(acc[i]);
        if (lane == 0) shw[warp][i] = s;
      }
    __syncthreads();
    if (threadIdx.x < nt) {
      const int i = threadIdx.x;
      const double pref = 1.5 * c.Om / (WL_C_OVER_H0 * WL_C_OVER_H0) * (1.0 + zn) * ch;
      const double s = (shw[0][i] + shw[1][i]) + (shw[2][i] + shw[3][i]);
      A.W[i * A.nchi + n] = any ? pref * s / A.norms[i] : 0.0;
    }
    return;
  }
  blk -= A.nchi;
  if (blk < A.nchi) {
    // Sheth-Tormen f_m, PBS biases and the m_min regularisation on the mass rule.
    // The values are written for every concentration node of each mass node
    // ([n][q * nc + j]), so the regularised halos at m_min carry the same
    // concentration scatter as the others.
    const int n = blk, nc = A.nc;
    const double rho = WL_RHO_CRIT0 * c.Om, Dn = A.Draw[n] / A.scal[SC_D1];
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int q = threadIdx.x; q < nm; q += GR_THREADS) {
      const double m = A.mb[q];
      const double nu0 = WL_DELTA_C / (Dn * A.sig0[q]);
      const double nu = nu0 * nu0, inu = 1.0 / nu;
      const double qn = WL_ST_Q * nu, qp = pow(qn, WL_ST_P);
      const double G = A.st_amp * sqrt(qn / (2.0 * WL_PI)) * (1.0 + 1.0 / qp) * exp(-0.5 * qn);
      const double fm = rho / (m * m) * G * (-2.0 * A.dlns[q]);
      const double ip = 1.0 / (1.0 + qp);
      const double a = 0.5 * inu - WL_ST_P * inu * ip - 0.5 * WL_ST_Q;
      const double ap = -0.5 * (inu * inu) + WL_ST_P * (1.0 + (WL_ST_P + 1.0) * qp) * (inu * inu) * (ip * ip);
      const double b1L = -2.0 * nu * a / WL_DELTA_C;
      const double b2L =
          (a * a + ap) * 4.0 * nu * nu / (WL_DELTA_C * WL_DELTA_C) + a * 2.0 * nu / (WL_DELTA_C * WL_DELTA_C);
      const double bb1 = 1.0 + b1L, bb2 = (8.0 / 21.0) * b1L + b2L;
      for (int j = 0; j < nc; ++j) {
        const size_t idx = ((size_t)n * nm + q) * nc + j;
        A.f[idx] = fm;
        A.b1[idx] = bb1;
        A.b2[idx] = bb2;
      }
      const double wq = A.omb[q] * m / rho * fm;
      s0 += wq;
      if (q > 0) {
        s1 += wq * bb1;
        s2 += wq * bb2;
      }
    }
    s0 = block_sum(s0, sh);
    s1 = block_sum(s1, sh);
    s2 = block_sum(s2, sh);
    if (threadIdx.x == 0) {
      const size_t i0 = (size_t)n * nm * nc;
      const double mr0 = A.mb[0] / rho;
      const double alpha0 = (1.0 - s0) / mr0;
      const double ft = A.f[i0] + alpha0 / A.omb[0];
      const double den = A.omb[0] * mr0 * ft;
      const double a1 = (1.0 - s1) / den, a2 = (0.0 - s2) / den;
      for (int j = 0; j < nc; ++j) {
        A.f[i0 + j] = ft;
        A.b1[i0 + j] = a1;
        A.b2[i0 + j] = a2;
      }
      A.D[n] = Dn;
      A.sigw2[n] *= Dn * Dn;
    }
    return;
  }
  blk -= A.nchi;
  // P_lin and dP_lin / d ln k at k = l_b / chi_n: lane s of 8 evaluates k exp(s h), s = 0, -2, -1, 1, 2
  const int id = (blk * GR_THREADS + threadIdx.x) >> 3, s = threadIdx.x & 7;
  const bool in = id < A.nl * A.nchi;
  const int b = in ? id / A.nchi : 0, n = in ? id % A.nchi : 0;
  const double shift[5] = {0.0, -2.0 * WL_FD_H, -WL_FD_H, WL_FD_H, 2.0 * WL_FD_H};
  const double k = A.ell[b] / A.chi[n];
  double v = 0.0;
  if (in && s < 5 && k <= A.b.k_max) {
    const double Dn = A.Draw[n] / A.scal[SC_D1];
    v = A.scal[SC_AMP] * dev_plin_unit(s ? k * exp(shift[s]) : k, dev_eh_const(c), c.ns) * Dn * Dn;
  }
  const int g = lane & ~7;
  const double m2 = __shfl_sync(0xffffffffu, v, g + 1), m1 = __shfl_sync(0xffffffffu, v, g + 2);
  const double f1 = __shfl_sync(0xffffffffu, v, g + 3), f2 = __shfl_sync(0xffffffffu, v, g + 4);
  if (in && s == 0) {
    A.Pl[id] = v;
    A.dPl[id] = (-f2 + 8.0 * f1 - 8.0 * m1 + m2) / (12.0 * WL_FD_H);
  }
  if (in && s >= 1 && s < 5) A.Psh[(size_t)id * 4 + s - 1] = v;
}

// Fourth launch: NFW profiles on the Limber grid at every (mass, concentration)
// node, u(k | m_q, c_bar(m_q, z_n) exp(cs[j])), c_bar the Duffy fit or the Bullock
// median K / ((1 + z) a_c(m_q)).  A thread holds its node's concentration and
// normalisation over `lper` ell bins (they do not depend on k).
__global__ void __launch_bounds__(128)
    k_profiles(cov_bins b, int nl, int nm, int nc, int lper, const double* __restrict__ cs,
               const double* __restrict__ ac, const double* __restrict__ ell, const double* __restrict__ chi,
               const double* __restrict__ z, const double* __restrict__ cz, const double* __restrict__ cmass,
               const double* __restrict__ rvir, const double* gl16x, const double* gl16w, double* U) {
  __shared__ double x16[16], w16[16];
  if (threadIdx.x < 16) {
    x16[threadIdx.x] = gl16x[threadIdx.x];
    w16[threadIdx.x] = gl16w[threadIdx.x];
  }
  __syncthreads();
  const int nchi = b.n_chi, n = blockIdx.x, q = blockIdx.z * 128 + threadIdx.x;
  if (q >= nm) return;
  double c = b.conc_model == COV_CONC_BULLOCK ? WL_BULLOCK_K / ((1.0 + z[n]) * ac[q / nc]) : cmass[q / nc] * cz[n];
  if (nc > 1) c *= exp(cs[q % nc]);
  const double l1 = log(1.0 + c), inorm = 1.0 / (l1 - c / (1.0 + c)), rv = rvir[q / nc], ich = chi[n];
  const int l0 = blockIdx.y * lper, l1_ = l0 + lper < nl ? l0 + lper : nl;
#pragma unroll 1
  for (int l = l0; l < l1_; ++l) {
    const double k = ell[l] / ich;
    U[((size_t)l * nchi + n) * nm + q] = k <= b.k_max ? dev_nfw_u(k * rv, c, l1, inorm, x16, w16) : 0.0;
  }
}

// quadrature nodes and everything else that depends on no cosmology: built once per handle
int wl_quadrature(cov_handle* h, cudaStream_t s) {
  const cov_nz nz = h->nz;
  k_gauss_legendre<<<1, 64, 0, s>>>(WL_N_GL_CHI, h->gl64x, h->gl64w);
  k_gauss_legendre<<<1, 32, 0, s>>>(16, h->gl16x, h->gl16w);
  k_gauss_legendre<<<(WL_N_K + 127) / 128, 128, 0, s>>>(WL_N_K, h->glkx, h->glkw);
  k_gauss_legendre<<<(h->nchi + 127) / 128, 128, 0, s>>>(h->nchi, h->glcx, h->glcw);
  k_gauss_hermite<<<1, 256, 0, s>>>(h->nc, h->bins.sigma_lnc, h->cs, h->cw);
  k_edges<<<1, 64, 0, s>>>(nz, h->zedges, h->scal);
  k_norms<<<h->nt, 64, 0, s>>>(nz, h->zedges, h->gl64x, h->gl64w, h->norms);
  k_sources<<<h->nt, WL_N_ZS, 0, s>>>(nz, h->zedges, h->gl64x, h->gl64w, h->zsrc, h->gsel);
  k_static_nodes<<<WL_N_K / 64, 64, 0, s>>>(h->glkx, h->glkw, h->knode, h->kwt, h->kw8, h->kws, h->chebm);
  k_mass_nodes<<<(h->nmb + 63) / 64, 64, 0, s>>>(h->bins, h->nc, h->cw, h->mb, h->omb, h->m, h->om, h->cmass);
  WL_LAUNCH(h, "quadrature kernels");
  return wl_triangle_shapes(h, s);
}

// Four launches: what depends on what decides the cut (chi intervals and linear
// spectrum; line of sight, sigma(m), sigma_W^2; halos, kernels, P_lin; profiles).
// Each launch holds every independent part of its level as blocks of its own, so
// a small set-up pays four launches and the FP64 latency of the longest part, and
// a large one fills the FP64 pipes (2 per clock and SM here, the bound of them all).
// With one sum per thread block and every factor recomputed where it is used (12
// launches; the transfer function once per mass, node and table, the growth as one
// serial chain, chi(z) by 64 evaluations of E) the stage took 7.02 ms at 1 bin,
// 8 ell bins, N_chi = N_M = 64 and 12.59 ms at 10 bins, 20 ell bins, N_chi = 256,
// N_M = 128; now 0.19 and 0.62 ms.
int wl_tables(cov_handle* h, cudaStream_t s) {
  const cov_cosmology* c = h->cosmo_d;  // read by the kernels: a captured graph replays with new values
  const cov_bins b = h->bins;
  const cov_nz nz = h->nz;
  const int nsrc = h->nt * WL_N_ZS;
  const double ymax = log1p(nz.zmax);
  k_prep<<<WL_N_ZI + WL_N_K / WL_KT_THREADS, WL_KT_THREADS, 0, s>>>(c, ymax, h->chebm, h->knode, h->kw8, h->zint, h->pk,
                                                                   h->amp_part);
  NodeArgs na{c,       b,       h->nchi,  nsrc,    ymax,     h->theta, h->glcx, h->glcw, h->zint, h->amp_part,
              h->knode, h->kwt, h->kws,   h->pk,   h->mb,    h->zsrc,  h->scal, h->chi,  h->wchi, h->z,    h->Draw,
              h->cz,   h->sig0, h->dlns,  h->sigF, h->rvir,  h->sigw2, h->chis, h->ksum, h->kticket};
  k_nodes<<<h->nchi + 1 + WL_KSPLIT * (h->nmb + h->nchi) + (nsrc + GR_THREADS - 1) / GR_THREADS, GR_THREADS, 0, s>>>(na);
  const double sta =
      1.0 / (1.0 + pow(2.0, -WL_ST_P) * tgamma(0.5 - WL_ST_P) / sqrt(WL_PI));  // Sheth-Tormen normalisation
  HaloArgs ha{c,       b,        nz,       h->nchi,  h->nc,   h->nl,   ymax,    sta,     h->scal,
              h->chi,  h->z,     h->Draw,  h->mb,    h->omb,  h->sig0, h->dlns, h->sigF, h->zedges, h->norms,
              h->gsel, h->chis,  h->zint,  h->gl64x, h->gl64w, h->ell_d, h->D,  h->f,    h->b1,
              h->b2,   h->W,     h->sigw2, h->ac,    h->Pl,   h->dPl,  h->Psh};
  const int npl = (h->nl * h->nchi * 8 + GR_THREADS - 1) / GR_THREADS;
  k_halo<<<(b.conc_model == COV_CONC_BULLOCK ? h->nmb : 0) + 2 * h->nchi + npl, GR_THREADS, 0, s>>>(ha);
  // ell bins per thread: one where the grid would leave the SMs short of warps, else four
  const int qb = (h->nm + 127) / 128;
  const int lper = (int64_t)h->nchi * qb * h->nl < 2048 ? 1 : 4;
  k_profiles<<<dim3((unsigned)h->nchi, (unsigned)((h->nl + lper - 1) / lper), (unsigned)qb), 128, 0, s>>>(
      b, h->nl, h->nm, h->nc, lper, h->cs, h->ac, h->ell_d, h->chi, h->z, h->cz, h->cmass, h->rvir, h->gl16x, h->gl16w,
      h->U);
  WL_LAUNCH(h, "table kernels");
  return COV_OK;
}
