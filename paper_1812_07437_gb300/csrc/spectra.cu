// Halo-model 3D polyspectra, responses and their Limber projections (paper
// Sec. 4, Eqs. ImunuHalos, PspHMtot2, B1halo, B2halos, B3halos, PowerHMResp,
// BispHMResp, RespP, RespB; Eq. nProjection), and the row builders of the
// (chi, M) contractions: the 1-halo factor rows A (Eqs. CovPPNG, Ins5P,
// Ins6P), the 1-halo trispectrum rows of the PT term (Eq. CovBB) and the
// super-sample rows (Eq. WLSSCflatskyLimber).
//
// Layout: per-node spectra are [entry][n_chi] (node contiguous); factor rows
// are [row][n_chi * nm] with the halo-integral node index q contiguous,
// matching the chi-major halo tables U[b][n][q], f[n][q].  q runs over the
// mass nodes, or over (mass, concentration) pairs with the concentration
// fastest when the lognormal scatter of Eq. LogNormC is on: every sum over q
// here is then the mass and the concentration integral at once.
#include "common.cuh"

// ---- triangle shapes (once per handle) -------------------------------------------
__device__ __forceinline__ double f2k(double ka, double kb, double mu) {
  return 5.0 / 7.0 + 0.5 * mu * (ka / kb + kb / ka) + 2.0 / 7.0 * mu * mu;
}

// F2 of the leg pairs (0,1), (1,2), (2,0) of a triangle and, optionally, their cosines
__device__ __forceinline__ void pair_f2(const double* k, double* F, int64_t stride, double* mu_out) {
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    const int y = (x + 1) % 3, o = (x + 2) % 3;
    const double mu = (k[o] * k[o] - k[x] * k[x] - k[y] * k[y]) / (2.0 * k[x] * k[y]);
    F[x * stride] = f2k(k[x], k[y], mu);
    if (mu_out) mu_out[x * stride] = mu;
  }
}

// The kernels F2 and the cosines depend on ratios of the legs only, i.e. on the
// triangle's ell bins, neither on chi nor on the cosmology: geo[.][t] holds F2 of
// the three pairs, their cosines, and F2 of the three pairs with leg i scaled by
// exp(s), s = -2h, -h, h, 2h (the ln k differences of the response).
__global__ void k_triangle_shapes(int ntri, const int32_t* tris, const double* ell, double* geo) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ntri) return;
  const double k[3] = {ell[tris[3 * t]], ell[tris[3 * t + 1]], ell[tris[3 * t + 2]]};
  pair_f2(k, geo + t, ntri, geo + 3 * (int64_t)ntri + t);
  const double s[4] = {-2.0 * WL_FD_H, -WL_FD_H, WL_FD_H, 2.0 * WL_FD_H};
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 4; ++j) {
      double kk[3] = {k[0], k[1], k[2]};
      kk[i] *= exp(s[j]);
      pair_f2(kk, geo + (6 + 3 * (int64_t)(4 * i + j)) * ntri + t, ntri, nullptr);
    }
}

int wl_triangle_shapes(cov_handle* h, cudaStream_t s) {
  if (h->ntri > 0)
    k_triangle_shapes<<<(h->ntri + 63) / 64, 64, 0, s>>>(h->ntri, h->tris_d, h->ell_d, h->trigeo);
  WL_LAUNCH(h, "k_triangle_shapes");
  return COV_OK;
}

// ---- halo integrals ---------------------------------------------------------------
// One thread per (node n, item): an item is an ell bin (I_2^0, I_1^1, I_1^2), a
// pair of ell bins (I_2^1, I_2^2) or a closed triple (I_3^0, I_3^1); each is a sum
// over the halo nodes q of products of profiles and weights, staged through shared
// memory in slabs of HI_Q nodes (rows padded so that lanes on different bins do
// not collide).  The pair integrals are shared by every triple that holds the
// pair, and no sum needs a reduction across lanes: ~3 FP64 operations per (triple,
// node, q), which is what bounds the kernel, where a warp per (triple, node) spent
// 14 five-step reductions and a serial tail on one lane (N_l = 20, 298 triples,
// N_chi = 256, N_M = 128: 6.92 ms for the bispectra before, see k_bfinish).
#define HI_Q 32
#define HI_THREADS 128
__global__ void __launch_bounds__(HI_THREADS)
    k_halo_int(const cov_cosmology* __restrict__ cosmo_p, int nl, int ntri, int nchi, int nm,
               const int32_t* __restrict__ tris, const double* __restrict__ m, const double* __restrict__ om,
               const double* __restrict__ f, const double* __restrict__ b1, const double* __restrict__ b2,
               const double* __restrict__ U, double* __restrict__ out) {
  extern __shared__ double hs[];  // U, g2 b1 U, g2 b2 U, g3 U, g3 b1 U: [5][nl][HI_Q + 1], then three weights
  const int n = blockIdx.x, LD = HI_Q + 1, S = nl * LD;
  double* wt = hs + 5 * S;  // g1 b1, g1 b2, g2 (per q)
  const double irho = 1.0 / (WL_RHO_CRIT0 * cosmo_p->Om);
  const int npair = nl * (nl + 1) / 2, nitem = nl + npair + ntri;
  const int it = blockIdx.y * HI_THREADS + threadIdx.x;
  int a = 0, b = 0, c = 0, kind = -1;
  if (it < nl) {
    kind = 0;
    a = it;
  } else if (it < nl + npair) {
    kind = 1;
    int r = it - nl;
    while (r >= nl - a) {
      r -= nl - a;
      ++a;
    }
    b = a + r;
  } else if (it < nitem) {
    kind = 2;
    const int32_t* t = tris + 3 * (it - nl - npair);
    a = t[0];
    b = t[1];
    c = t[2];
  }
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  for (int q0 = 0; q0 < nm; q0 += HI_Q) {
    const int nq = nm - q0 < HI_Q ? nm - q0 : HI_Q;
    __syncthreads();
    for (int e = threadIdx.x; e < nl * HI_Q; e += HI_THREADS) {
      const int l = e / HI_Q, j = e % HI_Q, q = q0 + j;
      double u = 0.0, w2 = 0.0, w3 = 0.0, bb1 = 0.0, bb2 = 0.0, w1 = 0.0;
      if (j < nq) {
        const double mr = m[q] * irho;
        u = U[((size_t)l * nchi + n) * nm + q];
        bb1 = b1[(size_t)n * nm + q];
        bb2 = b2[(size_t)n * nm + q];
        w1 = om[q] * f[(size_t)n * nm + q] * mr;
        w2 = w1 * mr;
        w3 = w2 * mr;
      }
      double* p = hs + l * LD + j;
      p[0] = u;
      p[S] = w2 * bb1 * u;
      p[2 * S] = w2 * bb2 * u;
      const double v = w3 * u;
      p[3 * S] = v;
      p[4 * S] = v * bb1;
      if (l == 0) {
        wt[j] = w1 * bb1;
        wt[HI_Q + j] = w1 * bb2;
        wt[2 * HI_Q + j] = w2;
      }
    }
    __syncthreads();
    if (kind == 0) {
      const double* u = hs + a * LD;
      for (int j = 0; j < nq; ++j) {
        const double x = u[j];
        s0 = fma(wt[2 * HI_Q + j] * x, x, s0);
        s1 = fma(wt[j], x, s1);
        s2 = fma(wt[HI_Q + j], x, s2);
      }
    } else if (kind == 1) {
      const double *u = hs + a * LD, *v1 = hs + S + b * LD, *v2 = hs + 2 * S + b * LD;
      for (int j = 0; j < nq; ++j) {
        s0 = fma(u[j], v1[j], s0);
        s1 = fma(u[j], v2[j], s1);
      }
    } else if (kind == 2) {
      const double *ua = hs + a * LD, *ub = hs + b * LD, *v0 = hs + 3 * S + c * LD, *v1 = hs + 4 * S + c * LD;
      for (int j = 0; j < nq; ++j) {
        const double x = ua[j] * ub[j];
        s0 = fma(x, v0[j], s0);
        s1 = fma(x, v1[j], s1);
      }
    }
  }
  // [item row][n]: 3 rows per bin, 2 per pair, 2 per triple
  if (kind == 0) {
    double* o = out + (size_t)(3 * a) * nchi + n;
    o[0] = s0;
    o[nchi] = s1;
    o[2 * (size_t)nchi] = s2;
  } else if (kind > 0) {
    const size_t row = 3 * (size_t)nl + 2 * (size_t)(it - nl);
    out[row * nchi + n] = s0;
    out[(row + 1) * nchi + n] = s1;
  }
}

// ---- 3D spectra, responses and Limber weights -------------------------------------
__device__ __forceinline__ double tree2(const double* F, double P0, double P1, double P2) {
  return 2.0 * (F[0] * P0 * P1 + F[1] * P1 * P2 + F[2] * P2 * P0);
}

struct FinishArgs {
  int nl, ntri, nchi, nt;
  double kmax;
  const int32_t* tris;
  const double *ell, *chi, *wchi, *W, *hint, *geo, *Pl, *dPl, *Psh;
  double *P3, *RP3, *B3, *RB3, *B1h3, *qw;
};

// One thread per (bin, node): P^HM and its response (Eqs. PspHMtot2, PowerHMResp);
// per (triple, node): B^HM, its response and the 1-halo B (Eqs. BspHMtot,
// BispHMResp, RespB) from the halo integrals and the triangle's stored shapes
// (~150 FP64 operations; the shapes' divisions and exponentials are not repeated
// per node); per (symmetric tomographic pair or triple, node): the Limber weight
// w_n chi^(2-2n) prod W.  The k_max rule zeroes everything beyond k_max.
__global__ void __launch_bounds__(128) k_bfinish(FinishArgs g) {
  const int nchi = g.nchi, nl = g.nl;
  int64_t id = (int64_t)blockIdx.x * 128 + threadIdx.x;
  const int64_t nP = (int64_t)nl * nchi, nB = (int64_t)g.ntri * nchi;
  auto leg = [&](int l, int row, int n) { return g.hint[(size_t)(3 * l + row) * nchi + n]; };
  auto pair = [&](int a, int b, int row, int n) {
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const int r = lo * nl - lo * (lo - 1) / 2 + (hi - lo);
    return g.hint[(size_t)(3 * nl + 2 * r + row) * nchi + n];
  };
  if (id < nP) {
    const int l = (int)(id / nchi), n = (int)(id % nchi);
    const bool valid = g.ell[l] / g.chi[n] <= g.kmax;
    const double pl = g.Pl[id], rlin = 47.0 / 21.0 * pl - g.dPl[id] / 3.0, i11 = leg(l, 1, n);
    g.P3[id] = valid ? leg(l, 0, n) + i11 * i11 * pl : 0.0;
    g.RP3[id] = valid ? i11 * i11 * rlin + pair(l, l, 0, n) : 0.0;
    return;
  }
  id -= nP;
  if (id < nB) {
    const int t = (int)(id / nchi), n = (int)(id % nchi);
    const int l[3] = {g.tris[3 * t], g.tris[3 * t + 1], g.tris[3 * t + 2]};
    bool valid = true;
    double P[3], rl[3], I1[3], I2[3], J1[3], J2[3], F[3], mu[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      valid = valid && g.ell[l[x]] / g.chi[n] <= g.kmax;
      P[x] = g.Pl[(size_t)l[x] * nchi + n];
      rl[x] = 47.0 / 21.0 * P[x] - g.dPl[(size_t)l[x] * nchi + n] / 3.0;
      I1[x] = leg(l[x], 1, n);
      I2[x] = leg(l[x], 2, n);
      J1[x] = pair(l[(x + 1) % 3], l[(x + 2) % 3], 0, n);  // I_2^1 of the two other legs
      J2[x] = pair(l[(x + 1) % 3], l[(x + 2) % 3], 1, n);
      F[x] = g.geo[(size_t)x * g.ntri + t];
      mu[x] = g.geo[(size_t)(3 + x) * g.ntri + t];
    }
    if (!valid) {
      g.B3[id] = 0.0;
      g.RB3[id] = 0.0;
      g.B1h3[id] = 0.0;
      return;
    }
    const size_t row = 3 * (size_t)nl + (size_t)nl * (nl + 1) + 2 * (size_t)t;
    const double i30 = g.hint[row * nchi + n], i31 = g.hint[(row + 1) * nchi + n];
    const double bpt = tree2(F, P[0], P[1], P[2]), i111 = I1[0] * I1[1] * I1[2];
    double B = i30 + i111 * bpt, r = i31, bg2 = 0.0;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const int y = (x + 1) % 3, o = (x + 2) % 3;
      const double pp = P[x] * P[y], m2 = mu[x] * mu[x];  // the pair (x, y), opposite leg o
      B += I1[x] * J1[x] * P[x];
      B += I1[x] * I1[y] * pp * (I2[o] + 4.0 / 7.0 * (m2 - 1.0 / 3.0) * (1.0 - I1[o]));
      r += I1[x] * (J2[x] * P[x] + J1[x] * rl[x]);
      bg2 += 2.0 * (m2 - 1.0) * pp;
    }
    g.B3[id] = B;
    g.B1h3[id] = i30;
    // 4th-order ln k differences of the tree level, each leg in turn
    double dsum = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double* ps = g.Psh + ((size_t)l[i] * nchi + n) * 4;  // s = -2h, -h, +h, +2h
      double v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double* ge = g.geo + (size_t)(6 + 3 * (4 * i + j)) * g.ntri + t;
        const double Fs[3] = {ge[0], ge[g.ntri], ge[2 * (size_t)g.ntri]}, p = ps[j];
        v[j] = tree2(Fs, i == 0 ? p : P[0], i == 1 ? p : P[1], i == 2 ? p : P[2]);
      }
      dsum += (-v[3] + 8.0 * v[2] - 8.0 * v[1] + v[0]) * (1.0 / (12.0 * WL_FD_H));
    }
    g.RB3[id] = r + i111 * (433.0 / 126.0 * bpt + 5.0 / 126.0 * bg2 - dsum / 3.0);
    return;
  }
  id -= nB;
  const int nt = g.nt, n2 = nt * (nt + 1) / 2, n3 = n2 * (nt + 2) / 3;
  if (id >= (int64_t)(n2 + n3) * nchi) return;
  int u = (int)(id / nchi);
  const int n = (int)(id % nchi);
  const double c2 = g.chi[n] * g.chi[n];
  double w = g.wchi[n] / c2;
  int i = 0;
  if (u < n2) {
    while (u >= nt - i) {
      u -= nt - i;
      ++i;
    }
    w *= g.W[i * nchi + n] * g.W[(i + u) * nchi + n];
  } else {
    u -= n2;
    while (u >= (nt - i) * (nt - i + 1) / 2) {
      u -= (nt - i) * (nt - i + 1) / 2;
      ++i;
    }
    int j = i;
    while (u >= nt - j) {
      u -= nt - j;
      ++j;
    }
    w *= g.W[i * nchi + n] * g.W[j * nchi + n] * g.W[(j + u) * nchi + n] / c2;
  }
  g.qw[id] = w;
}

// ---- Limber projection --------------------------------------------------------------
// index of the sorted multiset i <= j <= k among the n_t (n_t + 1) (n_t + 2) / 6
__device__ __forceinline__ int sym3(int i, int j, int k, int nt) {
  int t;
  if (i > j) t = i, i = j, j = t;
  if (j > k) t = j, j = k, k = t;
  if (i > j) t = i, i = j, j = t;
  const int r = nt - i, d = j - i;  // multisets that start below i, then pairs of the rest that start below j
  return (nt * (nt + 1) * (nt + 2) - r * (r + 1) * (r + 2)) / 6 + d * r - d * (d - 1) / 2 + (k - j);
}
__device__ __forceinline__ int sym2(int i, int j, int nt) {
  const int a = i < j ? i : j, b = i < j ? j : i;
  return a * nt - a * (a - 1) / 2 + (b - a);
}

struct ProjectArgs {
  int nl, ntri, nt, nchi;
  const double *P3, *B3, *B1h3, *qw, *scal;
  double *proj, *Ps, *B1hp;
};

// out[row][u] = sum_n S[row][n] Q[u][n].  The projection kernel is symmetric in
// the tomographic bins, so only the sorted multisets u are summed (220 of 1000
// triples at ten bins) and written out to every permutation: the 1-halo
// bispectra straight into B1h[t][i][j][k], P^s with its noise into Ps[l][i][j],
// P and B of the data vector as proj[l][u], proj[t][u] (read by k_datavec).
// 16 x 16 outputs per block, slabs of 32 nodes through shared memory.
// grid.z: 0 P, 1 B1h, 2 B (of the data vector).
__global__ void __launch_bounds__(256) k_project(ProjectArgs g) {
  __shared__ double Ss[16][33], Qs[16][33];
  const int nt = g.nt, n2 = nt * (nt + 1) / 2, n3 = n2 * (nt + 2) / 3, z = blockIdx.z;
  const int rows = z == 0 ? g.nl : g.ntri, nu = z == 0 ? n2 : n3;
  const int r0 = blockIdx.x * 16, u0 = blockIdx.y * 16;
  if (r0 >= rows || u0 >= nu) return;
  const double* S = z == 0 ? g.P3 : (z == 1 ? g.B1h3 : g.B3);
  const double* Q = z == 0 ? g.qw : g.qw + (size_t)n2 * g.nchi;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc = 0.0;
  for (int c0 = 0; c0 < g.nchi; c0 += 32) {
    for (int e = threadIdx.x; e < 512; e += 256) {
      const int r = e >> 5, n = e & 31;
      const bool in = c0 + n < g.nchi;
      Ss[r][n] = (in && r0 + r < rows) ? S[(size_t)(r0 + r) * g.nchi + c0 + n] : 0.0;
      Qs[r][n] = (in && u0 + r < nu) ? Q[(size_t)(u0 + r) * g.nchi + c0 + n] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int n = 0; n < 32; ++n) acc = fma(Ss[ty][n], Qs[tx][n], acc);
    __syncthreads();
  }
  const int r = r0 + ty;
  int u = u0 + tx;
  if (r >= rows || u >= nu) return;
  if (z == 0) {
    g.proj[(size_t)r * n2 + u] = acc;
    int i = 0;
    while (u >= nt - i) {
      u -= nt - i;
      ++i;
    }
    const int j = i + u;
    double* o = g.Ps + (size_t)r * nt * nt;
    const double v = acc + (i == j ? g.scal[SC_NOISE] : 0.0);
    o[i * nt + j] = v;
    o[j * nt + i] = v;
  } else if (z == 2) {
    g.proj[(size_t)g.nl * n2 + (size_t)r * n3 + u] = acc;
  } else {
    int i = 0;
    while (u >= (nt - i) * (nt - i + 1) / 2) {
      u -= (nt - i) * (nt - i + 1) / 2;
      ++i;
    }
    int j = i;
    while (u >= nt - j) {
      u -= nt - j;
      ++j;
    }
    const int k = j + u;
    double* o = g.B1hp + (size_t)r * nt * nt * nt;
    o[(i * nt + j) * nt + k] = acc;
    o[(i * nt + k) * nt + j] = acc;
    o[(j * nt + i) * nt + k] = acc;
    o[(j * nt + k) * nt + i] = acc;
    o[(k * nt + i) * nt + j] = acc;
    o[(k * nt + j) * nt + i] = acc;
  }
}

// data vector D (no noise): row -> its projected spectrum
__global__ void k_datavec(int64_t M, int nl, int nt, const int32_t* __restrict__ rd, const double* __restrict__ proj,
                          double* Dv) {
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= M) return;
  const int4 x = ((const int4*)rd)[2 * a], y = ((const int4*)rd)[2 * a + 1];  // type, bins | tomos, triangle
  const int n2 = nt * (nt + 1) / 2, n3 = n2 * (nt + 2) / 3;
  Dv[a] = x.x == 0 ? proj[(size_t)x.y * n2 + sym2(y.x, y.y, nt)]
                   : proj[(size_t)nl * n2 + (size_t)y.w * n3 + sym3(y.x, y.y, y.z, nt)];
}

// 1-halo factor rows A[a][(n,q)] = sqrt(w_n omega_q f_nq / Omega) chi^(1-2mu)
// prod W (m_q/rho)^mu prod U; grid (row blocks of K), coalesced along K.
__global__ void k_rows_a(int64_t M, int nchi, int nm, double inv_omega, const cov_cosmology* __restrict__ cosmo_p,
                         const int32_t* rd,
                         const double* chi, const double* wchi, const double* W, const double* m, const double* om,
                         const double* f, const double* U, double* A) {
  const double rho = WL_RHO_CRIT0 * cosmo_p->Om;
  int64_t a = blockIdx.x;
  int K = nchi * nm;
  int kk = blockIdx.y * blockDim.x + threadIdx.x;
  if (a >= M || kk >= K) return;
  int n = kk / nm, q = kk % nm;
  const int32_t* r = rd + 8 * a;
  int mu = (r[0] == 0) ? 2 : 3;
  double mr = m[q] / rho;
  double v = sqrt(wchi[n] * om[q] * f[kk] * inv_omega);
  double ch = chi[n];
  v *= (mu == 2) ? 1.0 / (ch * ch * ch) : 1.0 / (ch * ch * ch * ch * ch);
  v *= (mu == 2) ? mr * mr : mr * mr * mr;
  v *= W[r[4] * nchi + n] * W[r[5] * nchi + n];
  v *= U[((size_t)r[1] * nchi + n) * nm + q] * U[((size_t)r[2] * nchi + n) * nm + q];
  if (mu == 3) v *= W[r[6] * nchi + n] * U[((size_t)r[3] * nchi + n) * nm + q];
  A[a * K + kk] = v;
}

// trispectrum rows for leg pairs (L1 <= L2), L = bin * nt + tomo
__global__ void k_rows_t(int nleg, int nt, int nchi, int nm, const cov_cosmology* __restrict__ cosmo_p,
                         const double* chi, const double* wchi,
                         const double* W, const double* m, const double* om, const double* f, const double* U,
                         double* Tr) {
  const double rho = WL_RHO_CRIT0 * cosmo_p->Om;
  int64_t r = blockIdx.x;
  int K = nchi * nm;
  int kk = blockIdx.y * blockDim.x + threadIdx.x;
  if (kk >= K) return;
  // invert the pair index r = L1 * (2 nleg - L1 + 1)/2 + (L2 - L1)
  int L1 = 0;
  int64_t base = 0;
  while (base + (nleg - L1) <= r) {
    base += nleg - L1;
    ++L1;
  }
  int L2 = L1 + (int)(r - base);
  int b1 = L1 / nt, t1 = L1 % nt, b2 = L2 / nt, t2 = L2 % nt;
  int n = kk / nm, q = kk % nm;
  double mr = m[q] / rho, ch = chi[n];
  double v = sqrt(wchi[n] * om[q] * f[kk]) / (ch * ch * ch) * mr * mr;
  v *= W[t1 * nchi + n] * W[t2 * nchi + n];
  v *= U[((size_t)b1 * nchi + n) * nm + q] * U[((size_t)b2 * nchi + n) * nm + q];
  Tr[r * K + kk] = v;
}

// super-sample rows S[a][n] = sqrt(w_n sigma_W^2) chi^(2-2mu) prod W R_a
__global__ void k_rows_s(int64_t M, int nchi, const int32_t* rd, const double* chi, const double* wchi,
                         const double* W, const double* sigw2, const double* RP3, const double* RB3, double* S) {
  int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= M * nchi) return;
  int64_t a = id / nchi;
  int n = (int)(id % nchi);
  const int32_t* r = rd + 8 * a;
  double ch = chi[n], v = sqrt(wchi[n] * sigw2[n]);
  if (r[0] == 0) {
    v *= W[r[4] * nchi + n] * W[r[5] * nchi + n] / (ch * ch) * RP3[r[1] * nchi + n];
  } else {
    double c2 = ch * ch;
    v *= W[r[4] * nchi + n] * W[r[5] * nchi + n] * W[r[6] * nchi + n] / (c2 * c2) * RB3[r[7] * nchi + n];
  }
  S[id] = v;
}

// Halo integrals, spectra at the nodes, projections, data vector: 10.37 -> 0.30 ms
// at 10 bins, 20 ell bins, N_chi = 256, N_M = 128 (M = 181350), 0.56 -> 0.05 ms at
// 1 bin, 8 ell bins, N_chi = N_M = 64, against a warp per (triple, node) with a
// serial tail and one full sum over the nodes per row and tomographic triple.
int wl_spectra(cov_handle* h, double* d_D, cudaStream_t s) {
  const int nl = h->nl, nchi = h->nchi, nm = h->nm, nt = h->nt, ntri = h->ntri;
  const size_t smem = sizeof(double) * (5 * (size_t)nl * (HI_Q + 1) + 3 * HI_Q);  // <= 86 KB for 64 ell bins
  static std::once_flag attr_once[WL_MAX_DEVICES];
  static int attr_rc[WL_MAX_DEVICES];
  if (wl_once_per_device(attr_once, attr_rc, [] {
        return (int)cudaFuncSetAttribute(k_halo_int, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(sizeof(double) * (5 * 64 * (HI_Q + 1) + 3 * HI_Q)));
      }) != 0)
    return wl_fail(h, COV_ERR_CUDA, "cudaFuncSetAttribute(k_halo_int) failed");
  const int nitem = nl + nl * (nl + 1) / 2 + ntri;
  k_halo_int<<<dim3((unsigned)nchi, (unsigned)((nitem + HI_THREADS - 1) / HI_THREADS)), HI_THREADS, smem, s>>>(
      h->cosmo_d, nl, ntri, nchi, nm, h->tris_d, h->m, h->om, h->f, h->b1, h->b2, h->U, h->hint);
  const int n2 = nt * (nt + 1) / 2, n3 = n2 * (nt + 2) / 3;
  FinishArgs f{nl,      ntri,     nchi,      nt,    h->bins.k_max, h->tris_d, h->ell_d, h->chi, h->wchi, h->W, h->hint,
               h->trigeo, h->Pl, h->dPl, h->Psh, h->P3, h->RP3, h->B3, h->RB3, h->B1h3, h->qw};
  const int64_t nf = (int64_t)(nl + ntri + n2 + n3) * nchi;
  k_bfinish<<<(unsigned)((nf + 127) / 128), 128, 0, s>>>(f);
  ProjectArgs p{nl, ntri, nt, nchi, h->P3, h->B3, h->B1h3, h->qw, h->scal, h->proj, h->Ps, h->B1hp};
  const int rmax = std::max(nl, ntri), umax = ntri ? n3 : n2;
  k_project<<<dim3((unsigned)((rmax + 15) / 16), (unsigned)((std::max(umax, n2) + 15) / 16), ntri ? (d_D ? 3 : 2) : 1),
              256, 0, s>>>(p);
  if (d_D)
    k_datavec<<<(unsigned)((h->M + 255) / 256), 256, 0, s>>>(h->M, nl, nt, h->rowdesc_d, h->proj, d_D);
  WL_LAUNCH(h, "spectra kernels");
  h->spectra_ready = true;
  return COV_OK;
}

int wl_rows_a(cov_handle* h, cudaStream_t s) {
  dim3 g((unsigned)h->M, (h->K + 255) / 256);
  k_rows_a<<<g, 256, 0, s>>>(h->M, h->nchi, h->nm, 1.0 / h->omega, h->cosmo_d, h->rowdesc_d, h->chi, h->wchi, h->W,
                             h->m,
                             h->om, h->f, h->U, h->A);
  WL_LAUNCH(h, "k_rows_a");
  return COV_OK;
}

int wl_rows_t(cov_handle* h, cudaStream_t s) {
  dim3 g((unsigned)h->ntrow, (h->K + 255) / 256);
  k_rows_t<<<g, 256, 0, s>>>(h->nleg, h->nt, h->nchi, h->nm, h->cosmo_d, h->chi, h->wchi, h->W, h->m, h->om, h->f, h->U,
                             h->Trows);
  WL_LAUNCH(h, "k_rows_t");
  return COV_OK;
}

int wl_rows_s(cov_handle* h, cudaStream_t s) {
  int64_t n = h->M * h->nchi;
  k_rows_s<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(h->M, h->nchi, h->rowdesc_d, h->chi, h->wchi, h->W, h->sigw2,
                                                       h->RP3, h->RB3, h->Srows);
  WL_LAUNCH(h, "k_rows_s");
  return COV_OK;
}
