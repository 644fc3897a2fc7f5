"""The workloads on which this framework's speed is measured.

A case is one call (or the short chain of calls) that a user's program makes
per cosmology, through `paper_1812_07437_gb300.handle.Handle`:

* ``predict``  a new cosmology: every table, the spectra and the data vector
  (an MCMC or emulator loop that needs no covariance);
* ``assemble`` the dense covariance of a handle whose spectra are in hand, in
  the FP64 form (the default) or the split-BF16 tensor-core form;
* ``bands``    a new cosmology up to the covariance as lower-packed tiles (the
  streaming form, what the benchmark times);
* ``snr``      the cumulative signal-to-noise of a covariance in hand;
* ``stream``   the covariance assembled on packed tiles and its cumulative
  signal-to-noise in place (data vectors too large for a second copy);
* ``fisher``   a batch of cosmologies of one survey set-up;
* ``pca``      the principal components of a covariance in hand.

Sizes are those of the package's workloads and tests: 1 to 10 tomographic bins,
5 to 24 ell bins, 16 to 256 line-of-sight nodes, 12 to 128 masses, with and
without photometric scatter, Duffy and Bullock concentrations, with and without
concentration scatter.
"""
import math

import numpy as np
import torch

from paper_1812_07437_gb300 import native as N
from paper_1812_07437_gb300 import workloads
from paper_1812_07437_gb300.handle import Handle, packed_tiles

WHICH = {"P": N.COV_WHICH_P, "B": N.COV_WHICH_B, "joint": N.COV_WHICH_JOINT}
PRECISION = {"fp64": N.COV_FP64, "split": N.COV_SPLIT_BF16}


def _case(name, op, setup="euclid", n_tomo=1, n_ell=8, ell_min=10.0, ell_max=5000.0, n_chi=128, n_mass=96, n_conc=0,
          photoz=0.05, precision="fp64", terms=N.COV_TERMS_ALL, which="joint", batch=0):
    c = dict(op=op, setup=setup, n_tomo=n_tomo, n_ell=n_ell, ell_min=ell_min, ell_max=ell_max, n_chi=n_chi,
             n_mass=n_mass, n_conc=n_conc, photoz=photoz, precision=precision, terms=terms, which=which, batch=batch)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one bin, 8 ell bins (the cfg1_1bin set-up), one cosmology of a chain
        _case("predict_1bin", "predict", n_tomo=1, n_ell=8, ell_min=20.0, ell_max=3000.0, n_chi=64, n_mass=64, photoz=0.0),
        # the 10-bin survey of the benchmark (M = 181350): prediction only
        _case("predict_10bin", "predict", n_tomo=10, n_ell=20, n_chi=256, n_mass=128),
        # the paper's own 2-bin set-up (M = 818), which only the FP64 form serves (no photometric scatter)
        _case("cov_fp64_2bin", "assemble", setup="paper", n_tomo=2, n_ell=14, photoz=0.0),
        # the 5-bin survey (cfg2_5bin, M = 6375) in the default, FP64 form
        _case("cov_fp64_5bin", "assemble", n_tomo=5, n_ell=12),
        # the smallest covariance (cfg1_1bin), Gaussian and 1-halo terms, tensor-core form
        _case("cov_split_1bin", "assemble", n_tomo=1, n_ell=8, ell_min=20.0, ell_max=3000.0, n_chi=64, n_mass=64, photoz=0.0,
              precision="split", terms=N.COV_TERM_G | N.COV_TERM_1H),
        # the 5-bin survey in the tensor-core form
        _case("cov_split_5bin", "assemble", n_tomo=5, n_ell=12, precision="split"),
        # the benchmark's step at 4 bins (cfg3_4bin, M = 12944): tables, spectra, every term, packed tiles
        _case("step_split_4bin", "bands", n_tomo=4, n_ell=20, n_chi=256, n_mass=128, precision="split"),
        # cumulative S/N of the paper's 2-bin joint vector
        _case("snr_2bin", "snr", setup="paper", n_tomo=2, n_ell=14, photoz=0.0),
        # cumulative S/N of the 5-bin survey's joint vector
        _case("snr_5bin", "snr", n_tomo=5, n_ell=12),
        # 20 ell bins, 5 tomographic bins (cfg3_5bin, M = 24400): assembly and S/N in place on the tiles
        _case("stream_5bin", "stream", n_tomo=5, n_ell=20, n_chi=256, n_mass=128, precision="split"),
        # Fisher steps of a 3-bin survey (16 ell bins, M = 3064): the batched call over four cosmologies
        _case("fisher_3bin", "fisher", n_tomo=3, n_ell=16, n_chi=256, n_mass=128, precision="split", batch=4),
        # principal components of the paper's 2-bin set-up
        _case("pca_2bin", "pca", setup="paper", n_tomo=2, n_ell=14, photoz=0.0),
    ]


def _workload(case):
    paper = case["setup"] == "paper"
    wl = workloads.get("paper_2bin_full" if paper else "cfg2_5bin")
    wl["nz"].update(n_tomo=case["n_tomo"], photoz_sigma0=case["photoz"])
    wl["bins"].update(n_ell=case["n_ell"], ell_min=case["ell_min"], ell_max=case["ell_max"], n_chi=case["n_chi"],
                      n_mass=case["n_mass"], n_conc=case["n_conc"], sigma_lnc=workloads.SIGMA_LNC)
    return wl


def _cosmologies(case, seed):
    """Seeded cosmologies within 3% of the set-up's own."""
    rng = np.random.default_rng([int(seed), 18120743])
    base = _workload(case)["cosmology"]
    out = []
    for _ in range(max(1, case["batch"])):
        out.append({k: v if k == "Tcmb" else v * (1.0 + rng.uniform(-0.03, 0.03)) for k, v in base.items()})
    return out


def _layout(case):
    """(ell centres, closed triples, number of rows) of the data vector."""
    r, n = case["ell_max"] / case["ell_min"], case["n_ell"]
    e = [case["ell_min"] * r ** (i / n) for i in range(n + 1)]
    ell = [0.5 * (e[i] + e[i + 1]) for i in range(n)]
    tri = [(a, b, c) for c in range(n) for a in range(c + 1) for b in range(a, c + 1) if ell[c] <= ell[a] + ell[b]]
    t = case["n_tomo"]
    rows = n * t * (t + 1) // 2
    for a, b, c in tri:
        rows += t * (t + 1) * (t + 2) // 6 if a == b == c else t * t * (t + 1) // 2 if a == b or b == c else t ** 3
    return ell, tri, rows


def work(case):
    """Inputs are a few numbers; what counts is the arithmetic and one write of the result."""
    ell, tri, M = _layout(case)
    K = case["n_chi"] * case["n_mass"] * max(case["n_conc"], 1)
    nl, nt, op = case["n_ell"], case["n_tomo"], case["op"]
    low = 8.0 * M * (M + 1) / 2
    # profiles (~100 operations each), the halo integrals per triple and node, the Limber sums per row
    predict = 100.0 * nl * K + 24.0 * len(tri) * K + 4.0 * M * case["n_chi"]
    legs = nl * nt * (nl * nt + 1) / 2
    contraction = K * (float(M) * M + (legs * legs if case["terms"] & N.COV_TERM_BBPT else 0.0))
    factor = M ** 3 / 3.0
    if op == "predict":
        return {"bytes": 8.0 * M, "flops": predict}
    if op == "assemble":
        return {"bytes": low, "flops": contraction}
    if op == "bands":
        return {"bytes": low, "flops": predict + contraction}
    if op == "snr":
        return {"bytes": low, "flops": factor}
    if op == "stream":
        return {"bytes": low, "flops": contraction + factor}
    if op == "fisher":
        return {"bytes": case["batch"] * 8.0 * M, "flops": case["batch"] * (predict + contraction + factor)}
    return {"bytes": low, "flops": factor + 9.0 * M ** 3}  # pca: the factor and an eigen-decomposition


def draw(rng):
    """One more case: the operation, then sizes over its range (redrawn until it costs no more than the listed ones)."""
    op = rng.choice(["predict", "assemble", "assemble", "bands", "snr", "stream", "fisher", "pca"])
    # most rows, and most FP64 contraction work, that the operation's listed cases have
    rows = dict(predict=181350, assemble=6375, bands=12944, snr=6375, stream=24400, fisher=3064, pca=818)[op]
    while True:
        # (the tensor-core form's S/N needs the Euclid-like set-up: its covariance stays positive definite there)
        setup = "paper" if op == "pca" else "euclid" if op in ("stream", "fisher") else rng.choice(["euclid", "euclid", "paper"])
        precision = "split" if op in ("bands", "stream", "fisher") else rng.choice(["fp64", "split"])
        c = _case(None, op, setup=setup, n_tomo=rng.randint(1, 10 if op == "predict" else 2 if op == "pca" else 5),
                  n_ell=rng.randint(5, 20), ell_min=10.0 + 20.0 * rng.random(), ell_max=round(3000.0 + 2000.0 * rng.random()),
                  n_chi=round(math.exp(rng.uniform(math.log(16), math.log(256)))),
                  n_mass=round(math.exp(rng.uniform(math.log(12), math.log(128)))),
                  n_conc=rng.choice([0, 0, 0, 4]), photoz=0.0 if setup == "paper" and precision == "fp64" else 0.05,
                  precision=precision, which=rng.choice(["P", "B", "joint", "joint"]) if op == "snr" else "joint",
                  batch=rng.randint(2, 4) if op == "fisher" else 0)
        if op in ("snr", "pca"):  # the covariance in hand is assembled in FP64, whichever form the call has
            c["precision"] = "fp64"
        M, K = _layout(c)[2], c["n_chi"] * c["n_mass"] * max(c["n_conc"], 1)
        most = 12288 if op in ("assemble", "snr", "pca") else 32768
        if M <= rows and K <= most:
            return c


# ---------------------------------------------------------------- state and one pass
def prepare(case, seed):
    cosmos = _cosmologies(case, seed)
    wl = _workload(case)
    wl["cosmology"] = dict(cosmos[0])
    op, dev = case["op"], torch.device("cuda")
    h = Handle(wl, order=N.COV_ORDER_CUMULATIVE if op == "stream" else N.COV_ORDER_NATURAL)
    st = dict(op=op, h=h, cosmos=cosmos, precision=PRECISION[case["precision"]], terms=case["terms"])
    st["D"] = torch.zeros(h.M, dtype=torch.float64, device=dev)
    if op in ("assemble", "stream", "snr", "pca"):
        h.spectra(st["D"])
    if op in ("assemble", "snr", "pca"):
        st["C"] = torch.zeros(h.M, h.M, dtype=torch.float64, device=dev)
    if op == "bands":
        st["tiles"] = torch.zeros(packed_tiles(h.M) * 65536, dtype=torch.float64, device=dev)
    if op == "stream":  # with room for the row that carries the data vector
        st["tiles"] = torch.zeros(packed_tiles(h.M + 1) * 65536, dtype=torch.float64, device=dev)
    if op in ("snr", "pca"):
        h.assemble(st["C"], case["terms"], N.COV_FP64)
        st["which"] = WHICH[case["which"]]
    return st


def run(st):
    op, h, D = st["op"], st["h"], st["D"]
    if op == "predict":
        h.update(st["cosmos"][0])
        h.spectra(D)
        return {"D": D}
    if op == "assemble":
        h.assemble(st["C"], st["terms"], st["precision"])
        return {"C": st["C"]}
    if op == "bands":
        h.update(st["cosmos"][0])
        h.spectra(D)
        h.assemble_band(0, h.M, st["tiles"], terms=st["terms"], precision=st["precision"])
        return {"D": D, "tiles": st["tiles"]}
    if op == "snr":
        return {"snr": h.snr(st["C"], D, st["which"])}
    if op == "stream":
        h.assemble_band(0, h.M, st["tiles"], terms=st["terms"], precision=st["precision"])
        return {"snr": h.snr_tiles(st["tiles"], D)}
    if op == "fisher":
        snr, Ds, _ = h.batch_snr(st["cosmos"], terms=st["terms"], precision=st["precision"], with_D=True)
        return {"snr": snr, "D": Ds}
    r = h.pca(st["C"], D)
    return {k: r[k] for k in ("lam", "snr2", "cum_var", "cum_info", "total_snr2")}


# ---------------------------------------------------------------- the same quantities, plainly, in 64 bits
C_H0, RHO0, DELTA_C = 2997.92458, 2.77536627e11, 1.686


def _leggauss(n):
    """Nodes and weights on [-1, 1], ascending (Newton on the three-term recurrence, all nodes at once)."""
    x = np.cos(np.pi * (np.arange(n) + 0.75) / (n + 0.5))
    for _ in range(8):
        p0, p1 = np.ones(n), x.copy()
        for j in range(2, n + 1):
            p0, p1 = p1, ((2 * j - 1) * x * p1 - (j - 1) * p0) / j
        dp = n * (x * p1 - p0) / (x * x - 1.0)
        x = x - p1 / dp
    return -x, 2.0 / ((1.0 - x * x) * dp * dp)


def _E(z, c):
    return np.sqrt(c["Om"] * (1 + z) ** 3 + (1 - c["Om"]) * (1 + z) ** (3 * (1 + c["w0"])))


def _growth(a, c):
    """Growing solution of the linear growth equation from a = 1e-3, 1024 Runge-Kutta steps in ln a."""
    om, w = c["Om"], c["w0"]
    x0 = math.log(1e-3)
    h = (np.log(a) - x0) / 1024

    def rhs(x, d, p):
        em, ed = om * np.exp(-3 * x), (1 - om) * np.exp(-3 * (1 + w) * x)
        e2 = em + ed
        return p, -(2 + 0.5 * (-3 * em - 3 * (1 + w) * ed) / e2) * p + 1.5 * em / e2 * d

    x, d, p = np.full_like(h, x0), np.full_like(h, 1e-3), np.full_like(h, 1e-3)
    for _ in range(1024):
        a1, b1 = rhs(x, d, p)
        a2, b2 = rhs(x + h / 2, d + h / 2 * a1, p + h / 2 * b1)
        a3, b3 = rhs(x + h / 2, d + h / 2 * a2, p + h / 2 * b2)
        a4, b4 = rhs(x + h, d + h * a3, p + h * b3)
        x, d, p = x + h, d + h / 6 * (a1 + 2 * a2 + 2 * a3 + a4), p + h / 6 * (b1 + 2 * b2 + 2 * b3 + b4)
    return d


def _transfer(k, c):
    """Eisenstein and Hu (1998) transfer function without wiggles."""
    om, ob, fb, th = c["Om"] * c["h"] ** 2, c["Ob"] * c["h"] ** 2, c["Ob"] / c["Om"], c["Tcmb"] / 2.7
    s = 44.5 * math.log(9.83 / om) / math.sqrt(1 + 10 * ob ** 0.75)
    al = 1 - 0.328 * math.log(431 * om) * fb + 0.38 * math.log(22.3 * om) * fb * fb
    q = k * th * th / (c["Om"] * c["h"] * (al + (1 - al) / (1 + (0.43 * k * c["h"] * s) ** 4)))
    L = np.log(2 * math.e + 1.8 * q)
    return L / (L + (14.2 + 731 / (1 + 62.5 * q)) * q * q)


def _window(x):
    """Top-hat window and its derivative."""
    xs, xl = np.minimum(x, 0.5), np.maximum(x, 0.5)
    co = [3.0 * (-1) ** n * (2 * n + 2) / math.factorial(2 * n + 3) for n in range(9)]
    W = sum(co[n] * xs ** (2 * n) for n in range(9))
    dW = sum(2 * n * co[n] * xs ** (2 * n - 1) for n in range(1, 9))
    sx, cx = np.sin(xl), np.cos(xl)
    return (np.where(x < 0.5, W, 3 * (sx - xl * cx) / xl ** 3),
            np.where(x < 0.5, dW, 3 * ((xl * xl - 3) * sx + 3 * xl * cx) / xl ** 4))


def _collapse(sigma, c):
    """Scale factor at which the growth reaches DELTA_C / sigma (at most 100), by narrowing a bracket in ln a 33-fold."""
    d1 = _growth(np.array([1.0]), c)[0]
    t = DELTA_C / sigma
    lo, hi = np.full_like(t, math.log(1e-3)), np.full_like(t, math.log(100.0))
    never = _growth(np.array([100.0]), c)[0] / d1 <= t
    at = np.arange(34) / 33.0
    for _ in range(10):
        x = lo[:, None] + (hi - lo)[:, None] * at
        above = _growth(np.exp(x.ravel()), c).reshape(x.shape) / d1 >= t[:, None]
        above[:, -1] = True
        f = np.maximum(np.argmax(above, axis=1), 1)
        lo, hi = np.take_along_axis(x, f[:, None] - 1, 1)[:, 0], np.take_along_axis(x, f[:, None], 1)[:, 0]
    return np.where(never, 100.0, np.exp(0.5 * (lo + hi)))


def _j1(x):
    """J_1 (its integral over half a turn by the trapezoid rule up to x = 30, exact to rounding there)."""
    small = torch.zeros_like(x)
    xs = torch.clamp(x, max=30.0)
    for i in range(100):
        th = math.pi * (i + 0.5) / 100
        small += torch.cos(th - xs * math.sin(th)) / 100
    return torch.where(x < 30.0, small, torch.special.bessel_j1(x))


def _counts(edges, f_sky, tri, dev):
    """Lattice modes per bin, and lattice triangles per bin triple as a cyclic triple correlation (no wrap-around)."""
    lf = 2 * math.pi / math.sqrt(4 * math.pi * f_sky)
    n = len(edges) - 1
    lo = [math.ceil((e / lf) ** 2) for e in edges[:-1]]
    hi = lo[1:] + [math.floor((edges[-1] / lf) ** 2) + 1]
    R = math.isqrt(max(hi) - 1)
    L = 1 << 5
    L = -(-(3 * R + 2) // L) * L
    g = torch.arange(L, device=dev)
    g = torch.where(g > L // 2, g - L, g)
    r2 = g[:, None] ** 2 + g[None, :] ** 2
    r2 = torch.where((g.abs()[:, None] <= R) & (g.abs()[None, :] <= R), r2, torch.full_like(r2, -1))
    Nm, F = [], []
    for b in range(n):
        ind = (r2 >= lo[b]) & (r2 < hi[b])
        Nm.append(int(ind.sum()))
        F.append(torch.fft.rfft2(ind.double()).real.reshape(-1))
    del r2
    wt = torch.full((L, L // 2 + 1), 2.0, dtype=torch.float64, device=dev)
    wt[:, 0] = 1.0
    wt[:, -1] = 1.0
    wt = wt.reshape(-1) / float(L * L)
    F = torch.stack(F)
    Nt = np.zeros(len(tri))
    for c in range(n):
        G = ((F * (F[c] * wt)) @ F.T).cpu().numpy()
        for t, (a, b, cc) in enumerate(tri):
            if cc == c:
                Nt[t] = round(G[a, b])
    return np.array(Nm, dtype=np.float64), Nt


def _model(case, c, dev):
    """Tables and spectra of one cosmology: a dict of 64-bit arrays on `dev`."""
    wl = _workload(case)
    b, nz = wl["bins"], wl["nz"]
    ell, tri, _ = _layout(case)
    nl, nt, nchi, nm = case["n_ell"], case["n_tomo"], case["n_chi"], case["n_mass"]
    ell = np.array(ell)
    x64, w64 = _leggauss(64)

    def chi_of(z):
        zz = 0.5 * z[..., None] * (x64 + 1)
        return C_H0 * 0.5 * z * np.sum(w64 / _E(zz, c), axis=-1)

    # line of sight
    xc, wc = _leggauss(nchi)
    cm = chi_of(np.array([nz["zmax"]]))[0]
    chi, wchi = 0.5 * cm * (xc + 1), 0.5 * cm * wc
    z = chi / C_H0
    for _ in range(40):
        z = z - (chi_of(z) - chi) / C_H0 * _E(z, c)
    D = _growth(np.append(1 / (1 + z), 1.0), c)
    D = D[:-1] / D[-1]
    # linear power, halo abundance and biases
    xk, wk = _leggauss(4096)
    half = 0.5 * math.log(1e8)
    lk, wk = math.log(1e-5) + half * (xk + 1), half * wk
    k4 = np.exp(lk)
    d2 = k4 ** (3 + c["ns"]) * _transfer(k4, c) ** 2 / (2 * math.pi ** 2)
    amp = c["sigma8"] ** 2 / np.sum(wk * d2 * _window(8.0 * k4)[0] ** 2)
    d2 = amp * d2
    rho = RHO0 * c["Om"]
    dl = math.log(b["m_max"] / b["m_min"]) / (nm - 1)
    m = b["m_min"] * np.exp(dl * np.arange(nm))
    om = dl * m
    om[0] *= 0.5
    om[-1] *= 0.5
    R = np.cbrt(3 * m / (4 * math.pi * rho))
    sig, dls, sigF = np.empty(nm), np.empty(nm), np.empty(nm)
    for q in range(nm):
        W, dW = _window(k4 * R[q])
        s2 = np.sum(wk * d2 * W * W)
        sig[q], dls[q] = math.sqrt(s2), R[q] / 6 * np.sum(wk * d2 * 2 * W * dW * k4) / s2
        sigF[q] = math.sqrt(np.sum(wk * d2 * _window(k4 * R[q] * 0.01 ** (1 / 3))[0] ** 2))
    A = 1 / (1 + 2 ** -0.3 * math.gamma(0.2) / math.sqrt(math.pi))
    nu = (DELTA_C / (D[:, None] * sig)) ** 2
    qn = 0.707 * nu
    qp = qn ** 0.3
    f = rho / m ** 2 * A * np.sqrt(qn / (2 * math.pi)) * (1 + 1 / qp) * np.exp(-0.5 * qn) * (-2 * dls)
    a1 = 0.5 / nu - 0.3 / (nu * (1 + qp)) - 0.5 * 0.707
    a2 = -0.5 / nu ** 2 + 0.3 * (1 + 1.3 * qp) / (nu ** 2 * (1 + qp) ** 2)
    bL1 = -2 * nu * a1 / DELTA_C
    bL2 = (a1 * a1 + a2) * 4 * nu ** 2 / DELTA_C ** 2 + a1 * 2 * nu / DELTA_C ** 2
    b1, b2 = 1 + bL1, 8 / 21 * bL1 + bL2
    mr = m / rho
    f[:, 0] += (1 - np.sum(om * mr * f, axis=1)) / mr[0] / om[0]
    den = om[0] * mr[0] * f[:, 0]
    b1[:, 0] = (1 - np.sum((om * mr * f * b1)[:, 1:], axis=1)) / den
    b2[:, 0] = -np.sum((om * mr * f * b2)[:, 1:], axis=1) / den
    # concentrations and profiles: u = int w(t) sinc(K t) dt / int w(t) dt, w = t / (1 + c t)^2, on panels
    if b["conc_model"] if "conc_model" in b else 0:
        conc = 4.0 / ((1 + z)[:, None] * _collapse(sigF, c))
    else:
        conc = 10.14 * (m / 2e12) ** -0.081 * (1 + z)[:, None] ** -1.01
    if case["n_conc"] > 1:
        xh, wh = np.polynomial.hermite_e.hermegauss(case["n_conc"])
        off, wcn = np.exp(xh * b["sigma_lnc"]), wh / math.sqrt(2 * math.pi)
    else:
        off, wcn = np.ones(1), np.ones(1)
    conc = (conc[:, :, None] * off).reshape(nchi, -1)
    nc = len(off)
    mq, omq = np.repeat(m, nc), (om[:, None] * wcn).ravel()
    f, b1, b2 = (np.repeat(v, nc, axis=1) for v in (f, b1, b2))
    rv = np.cbrt(3 * mq / (4 * math.pi * 200.0 * rho))
    T = lambda v: torch.as_tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)  # noqa: E731
    x16, w16 = _leggauss(16)
    U = torch.zeros(nl, nchi, nm * nc, dtype=torch.float64, device=dev)
    ct, kr = T(conc), T(rv)
    kk = ell[:, None] / chi
    ok = kk <= b["k_max"]
    for i in range(nl):
        for n0 in range(0, nchi, 32):
            n1 = min(nchi, n0 + 32)
            if not ok[i, n0:n1].any():
                continue
            K = T(np.where(ok[i, n0:n1], kk[i, n0:n1], 1e-3))[:, None] * kr
            P = int(math.ceil(max(float(K.max()) / (2 * math.pi), float(ct[n0:n1].max()), 1.0)))
            num, den2 = torch.zeros_like(K), torch.zeros_like(K)
            for p in range(P):
                for xx, ww in zip(x16, w16):
                    t = (p + 0.5 * (xx + 1)) / P
                    w = ww * t / (1 + ct[n0:n1] * t) ** 2
                    num += w * torch.sin(K * t) / (K * t)
                    den2 += w
            U[i, n0:n1] = num / den2 * T(ok[i, n0:n1].astype(float))[:, None]
    # lensing kernels
    zmin, zmax, z0, s0 = nz["zmin"], nz["zmax"], nz["z0"], nz["photoz_sigma0"]
    cdf = lambda v: 1 - (1 + (v / z0) ** 1.5) * math.exp(-((v / z0) ** 1.5))  # noqa: E731
    ed = [zmin]
    for t in range(1, nt):
        lo, hi = zmin, zmax
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if (cdf(mid) - cdf(zmin)) / (cdf(zmax) - cdf(zmin)) < t / nt:
                lo = mid
            else:
                hi = mid
        ed.append(0.5 * (lo + hi))
    ed.append(zmax)

    def erf(v):
        return torch.special.erf(torch.as_tensor(v, dtype=torch.float64)).numpy()

    def sel(v, i):
        if s0 == 0:
            return ((v >= ed[i]) & ((v <= ed[i + 1]) if i == nt - 1 else (v < ed[i + 1]))).astype(float)
        s = math.sqrt(2) * s0 * (1 + v)
        return 0.5 * (erf((ed[i + 1] - v) / s) - erf((ed[i] - v) / s))

    def nodes(a):
        pts = [a] + [e for e in ed if a < e < zmax] + [zmax]
        hw = [0.5 * (q - p) for p, q in zip(pts, pts[1:])]
        return (np.concatenate([p + h * (x64 + 1) for p, h in zip(pts, hw)]), np.concatenate([h * w64 for h in hw]))

    shape = lambda v: v * v * np.exp(-((v / z0) ** 1.5))  # noqa: E731
    v, w = nodes(zmin)
    norm = [np.sum(w * shape(v) * sel(v, i)) for i in range(nt)]
    Wk = np.zeros((nt, nchi))
    for n in range(nchi):
        if z[n] < zmax:
            v, w = nodes(z[n])
            cs = chi_of(v)
            geo = w * shape(v) * (cs - chi[n]) / cs * 1.5 * c["Om"] / C_H0 ** 2 * (1 + z[n]) * chi[n]
            for i in range(nt):
                Wk[i, n] = np.sum(geo * sel(v, i)) / norm[i]
    # survey variance on the disc, linear spectra on the Limber grid
    theta = math.acos(1 - 2 * b["f_sky"])
    pl0 = T(amp * k4 ** c["ns"] * _transfer(k4, c) ** 2 * wk * k4 * k4)
    xx = T(k4) * T(chi)[:, None] * theta
    sw = 4 / (2 * math.pi) * ((_j1(xx) / xx) ** 2 * pl0).sum(1) * T(D) ** 2

    def plin(k):
        return np.where(ok, amp * k ** c["ns"] * _transfer(k, c) ** 2 * D ** 2, 0.0)

    Pl = T(plin(kk))
    sh = {s: T(plin(kk * math.exp(s * 1e-3))) for s in (-2, -1, 1, 2)}
    dPl = (-sh[2] + 8 * sh[1] - 8 * sh[-1] + sh[-2]) / (12 * 1e-3)
    okt = T(ok.astype(float))
    # spectra and responses at the nodes
    g1 = T(omq * f * (mq / rho))
    mrt, f1, f2 = T(mq / rho), T(b1), T(b2)
    i11 = (g1 * f1 * U).sum(-1)
    i12 = (g1 * f2 * U).sum(-1)
    rl = 47 / 21 * Pl - dPl / 3
    P3 = ((g1 * mrt * U * U).sum(-1) + i11 ** 2 * Pl) * okt
    RP3 = (i11 ** 2 * rl + (g1 * mrt * f1 * U * U).sum(-1)) * okt
    i21 = torch.einsum("nq,anq,bnq->abn", g1 * mrt * f1, U, U)
    i22 = torch.einsum("nq,anq,bnq->abn", g1 * mrt * f2, U, U)
    kt = T(kk)

    def tree(k, p):
        s = 0.0
        for x in range(3):
            y, o = (x + 1) % 3, (x + 2) % 3
            mu = (k[o] ** 2 - k[x] ** 2 - k[y] ** 2) / (2 * k[x] * k[y])
            s = s + 2 * (5 / 7 + 0.5 * mu * (k[x] / k[y] + k[y] / k[x]) + 2 / 7 * mu * mu) * p[x] * p[y]
        return s

    B3, RB3, B1h = [], [], []
    for leg in tri:
        k, p, r = [kt[a] for a in leg], [Pl[a] for a in leg], [rl[a] for a in leg]
        I, J = [i11[a] for a in leg], [i12[a] for a in leg]
        g3 = g1 * mrt * mrt * U[leg[0]] * U[leg[1]] * U[leg[2]]
        i30, bt = g3.sum(-1), tree(k, p)
        III = I[0] * I[1] * I[2]
        Bv, Rv, bg = i30 + III * bt, (g3 * f1).sum(-1), 0.0
        for x in range(3):
            y, o = (x + 1) % 3, (x + 2) % 3
            mu = (k[o] ** 2 - k[x] ** 2 - k[y] ** 2) / (2 * k[x] * k[y])
            Bv = Bv + I[x] * i21[leg[y], leg[o]] * p[x]
            Bv = Bv + I[x] * I[y] * p[x] * p[y] * (J[o] + 4 / 7 * (mu * mu - 1 / 3) * (1 - I[o]))
            Rv = Rv + I[x] * i22[leg[y], leg[o]] * p[x] + I[x] * i21[leg[y], leg[o]] * r[x]
            bg = bg + 2 * (mu * mu - 1) * p[x] * p[y]
        ds = 0.0
        for x in range(3):
            for s, co in ((2, -1), (1, 8), (-1, -8), (-2, 1)):
                k2, p2 = list(k), list(p)
                k2[x], p2[x] = k[x] * math.exp(s * 1e-3), sh[s][leg[x]]
                ds = ds + co * tree(k2, p2) / (12 * 1e-3)
        Rv = Rv + III * (433 / 126 * bt + 5 / 126 * bg - ds / 3)
        v = okt[leg[0]] * okt[leg[1]] * okt[leg[2]]
        B3.append(Bv * v)
        RB3.append(Rv * v)
        B1h.append(i30 * v)
    z3 = torch.zeros(0, nchi, dtype=torch.float64, device=dev)
    st = lambda v: torch.stack(v) if v else z3  # noqa: E731
    W, ch, wc = T(Wk), T(chi), T(wchi)
    noise = nz["sigma_e"] ** 2 / (nz["n_gal_arcmin2"] * (10800 / math.pi) ** 2 / nt)
    Ps = torch.einsum("in,jn,ln->lij", W, W, P3 * wc / ch ** 2) + noise * torch.eye(nt, dtype=torch.float64, device=dev)
    Bh = torch.einsum("in,jn,kn,tn->tijk", W, W, W, st(B1h) * wc / ch ** 4) if tri else None
    return dict(ell=ell, tri=tri, nl=nl, nt=nt, chi=ch, wchi=wc, W=W, U=U, f=T(f), om=T(omq), mr=mrt, sw=sw, P3=P3,
                RP3=RP3, B3=st(B3), RB3=st(RB3), Ps=Ps, Bh=Bh, bins=b)


def _rows(mod, cumulative):
    """Per row: type, three bins, three tomographic bins, triangle (int64), in the order of the data vector."""
    nt, P, B = mod["nt"], [], []
    for l in range(mod["nl"]):
        P += [(0, l, l, l, i, j, 0, 0) for i in range(nt) for j in range(i, nt)]
    for t, (a, b, c) in enumerate(mod["tri"]):
        for i in range(nt):
            for j in range(i if a == b else 0, nt):
                B += [(1, a, b, c, i, j, k, t) for k in range(j if b == c else 0, nt)]
    rows = P + B
    if cumulative:
        rows.sort(key=lambda r: (r[3], r[0]))
    return np.array(rows, dtype=np.int64)


def _data(mod, rd):
    W, ch, wc = mod["W"], mod["chi"], mod["wchi"]
    out = torch.zeros(len(rd), dtype=torch.float64, device=W.device)
    for a0 in range(0, len(rd), 8192):
        r = torch.as_tensor(rd[a0:a0 + 8192], device=W.device)
        w = W[r[:, 4]] * W[r[:, 5]]
        p = (w * mod["P3"][r[:, 1]] * wc / ch ** 2).sum(1)
        if mod["tri"]:
            q = (w * W[r[:, 6]] * mod["B3"][r[:, 7]] * wc / ch ** 4).sum(1)
            p = torch.where(r[:, 0] == 0, p, q)
        out[a0:a0 + 8192] = p
    return out


def _covariance(mod, rd, terms, counts):
    """The covariance (lower triangle filled), plainly in 64 bits."""
    dev, W, ch, wc, U = mod["W"].device, mod["W"], mod["chi"], mod["wchi"], mod["U"]
    Nm, Nt = (torch.as_tensor(v, device=dev) for v in counts)
    nt, nl, M = mod["nt"], mod["nl"], len(rd)
    omega = 4 * math.pi * mod["bins"]["f_sky"]
    R = torch.as_tensor(rd, device=dev)
    isB = R[:, 0] == 1
    base = torch.sqrt(wc[:, None] * mod["om"] * mod["f"]) * mod["mr"] ** 2
    C = torch.zeros(M, M, dtype=torch.float64, device=dev)

    def add_product(F, scale):  # lower blocks of F F^T
        for i in range(0, len(F), 2048):
            for j in range(0, i + 1, 2048):
                C[i:i + 2048, j:j + 2048] += scale * (F[i:i + 2048] @ F[j:j + 2048].T)

    if terms & N.COV_TERM_1H:
        F = torch.empty(M, base.numel(), dtype=torch.float64, device=dev)
        for a0 in range(0, M, 512):
            r, bb = R[a0:a0 + 512], isB[a0:a0 + 512]
            w = W[r[:, 4]] * W[r[:, 5]] / ch ** 3
            w = torch.where(bb[:, None], w * W[r[:, 6]] / ch ** 2, w)
            v = base * U[r[:, 1]] * U[r[:, 2]] * w[:, :, None]
            v = torch.where(bb[:, None, None], v * mod["mr"] * U[r[:, 3]], v)
            F[a0:a0 + 512] = v.reshape(len(r), -1)
        add_product(F, 1 / omega)
        del F
    if terms & N.COV_TERM_SSC:
        w = W[R[:, 4]] * W[R[:, 5]] * torch.sqrt(wc * mod["sw"]) / ch ** 2
        S = w * mod["RP3"][R[:, 1]]
        if mod["tri"]:
            S = torch.where(isB[:, None], w * W[R[:, 6]] / ch ** 2 * mod["RB3"][R[:, 7]], S)
        add_product(S, 1.0)
    if terms & N.COV_TERM_BBPT and mod["tri"]:  # projected 1-halo trispectrum of leg pairs
        V = (W / ch ** 1.5)[:, :, None]
        leg = (U[:, None] * V[None]).reshape(nl * nt, -1)
        i, j = torch.triu_indices(nl * nt, nl * nt, device=dev)
        Tr = torch.empty(len(i), base.numel(), dtype=torch.float64, device=dev)
        for a0 in range(0, len(i), 512):
            Tr[a0:a0 + 512] = leg[i[a0:a0 + 512]] * leg[j[a0:a0 + 512]] * base.reshape(-1)
        Tm = Tr @ Tr.T
        del Tr
        pid = torch.zeros(nl * nt, nl * nt, dtype=torch.int64, device=dev)
        pid[i, j] = torch.arange(len(i), device=dev)
        pid[j, i] = pid[i, j]
    perms = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))
    Ps, Bh = mod["Ps"], mod["Bh"]
    for a0 in range(0, M, 256):
        A, Bc = R[a0:a0 + 256, None, :], R[None, :a0 + 256, :]
        both0, both1 = (A[..., 0] == 0) & (Bc[..., 0] == 0), (A[..., 0] == 1) & (Bc[..., 0] == 1)
        ba, ta, tb = A[..., 1:4], A[..., 4:7], Bc[..., 4:7]
        bb = Bc[..., 1:4]
        v = torch.zeros(A.shape[0], Bc.shape[1], dtype=torch.float64, device=dev)
        if terms & N.COV_TERM_G:
            l = ba[..., 0]
            pp = Ps[l, ta[..., 0], tb[..., 0]] * Ps[l, ta[..., 1], tb[..., 1]] + Ps[l, ta[..., 0], tb[..., 1]] * Ps[l, ta[..., 1], tb[..., 0]]
            v += torch.where(both0 & (l == bb[..., 0]), pp / Nm[l], 0.0)
            if mod["tri"]:
                same = both1 & (A[..., 7] == Bc[..., 7])
                for s in perms:
                    hit = same & (ba[..., 0] == ba[..., s[0]]) & (ba[..., 1] == ba[..., s[1]]) & (ba[..., 2] == ba[..., s[2]])
                    p3 = Ps[ba[..., 0], ta[..., 0], tb[..., s[0]]] * Ps[ba[..., 1], ta[..., 1], tb[..., s[1]]] * Ps[ba[..., 2], ta[..., 2], tb[..., s[2]]]
                    v += torch.where(hit, p3 * omega / Nt[A[..., 7]], 0.0)
        if terms & N.COV_TERM_BBPT and mod["tri"]:
            for x in range(3):
                for y in range(3):
                    x1, x2, y1, y2 = (x + 1) % 3, (x + 2) % 3, (y + 1) % 3, (y + 2) % 3
                    ii, jj = torch.nonzero(both1 & (ba[..., x] == bb[..., y]), as_tuple=True)
                    a, q = R[a0 + ii], R[jj]
                    l = a[:, 1 + x]
                    r1 = pid[a[:, 1 + x1] * nt + a[:, 4 + x1], a[:, 1 + x2] * nt + a[:, 4 + x2]]
                    r2 = pid[q[:, 1 + y1] * nt + q[:, 4 + y1], q[:, 1 + y2] * nt + q[:, 4 + y2]]
                    t = Bh[a[:, 7], q[:, 4 + y], a[:, 4 + x1], a[:, 4 + x2]] * Bh[q[:, 7], a[:, 4 + x], q[:, 4 + y1], q[:, 4 + y2]]
                    v[ii, jj] += (t + Ps[l, a[:, 4 + x], q[:, 4 + y]] * Tm[r1, r2]) / Nm[l]
        if terms & N.COV_TERM_PB and mod["tri"]:
            for first in (True, False):
                Pr, Br = (A, Bc) if first else (Bc, A)
                mixed = (Pr[..., 0] == 0) & (Br[..., 0] == 1)
                l, i, j, t = Pr[..., 1], Pr[..., 4], Pr[..., 5], Br[..., 7]
                for y in range(3):
                    ty, t1, t2 = Br[..., 4 + y], Br[..., 4 + (y + 1) % 3], Br[..., 4 + (y + 2) % 3]
                    e = Ps[l, i, ty] * Bh[t, j, t1, t2] + Ps[l, j, ty] * Bh[t, i, t1, t2]
                    v += torch.where(mixed & (Br[..., 1 + y] == l), e / Nm[l], 0.0)
        C[a0:a0 + 256, :a0 + 256] += v
    return torch.tril(C)


def _cumulative_snr(C, D, rd, which, nl):
    """sqrt(D^T C^-1 D) of the selected rows up to each largest bin."""
    keep = np.ones(len(rd), bool) if which == "joint" else rd[:, 0] == (0 if which == "P" else 1)
    sel = np.nonzero(keep)[0]
    sel = sel[np.argsort(rd[sel, 3], kind="stable")]
    if not len(sel):
        return np.full(nl, np.nan)
    s = torch.as_tensor(sel, device=C.device)
    full = C + torch.tril(C, -1).T
    c = full[s][:, s]
    d = torch.sqrt(torch.diagonal(c))
    L = torch.linalg.cholesky(c / d[:, None] / d)
    y2 = torch.linalg.solve_triangular(L, (D[s] / d)[:, None], upper=False)[:, 0] ** 2
    cum = np.append(0.0, torch.cumsum(y2, 0).cpu().numpy())
    n = np.array([np.sum(rd[sel, 3] <= b) for b in range(nl)])
    return np.where(n > 0, np.sqrt(cum[n]), np.nan)


def exact(case, seed):
    """What run() returns, from plain 64-bit sums."""
    op = case["op"]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if op == "stream":  # the largest factorisation: too long in plain 64 bits
        return None
    mods = [_model(case, c, dev) for c in _cosmologies(case, seed)]
    rd = _rows(mods[0], op == "stream")
    D = [_data(m, rd) for m in mods]
    if op == "predict":
        return {"D": D[0]}
    b, (_, tri, _) = mods[0]["bins"], _layout(case)
    r = b["ell_max"] / b["ell_min"]
    edges = [b["ell_min"] * r ** (i / b["n_ell"]) for i in range(b["n_ell"] + 1)]
    counts = _counts(edges, b["f_sky"], tri, dev)
    if op == "fisher":
        out = []
        for m, d in zip(mods, D):
            C = _covariance(m, rd, case["terms"], counts)
            out.append([_cumulative_snr(C, d, rd, w, case["n_ell"]) for w in ("P", "B", "joint")])
        return {"snr": np.array(out), "D": torch.stack(D).cpu().numpy()}
    C = _covariance(mods[0], rd, case["terms"], counts)
    if op == "assemble":
        return {"C": C}
    if op == "bands":
        M, nt = len(rd), (len(rd) + 255) // 256
        tiles = torch.zeros(packed_tiles(M), 256, 256, dtype=torch.float64, device=dev)
        for i in range(nt):
            for j in range(i + 1):
                blk = C[256 * i:256 * i + 256, 256 * j:256 * j + 256]
                tiles[i * (i + 1) // 2 + j, :blk.shape[0], :blk.shape[1]] = blk
        return {"D": D[0], "tiles": tiles.reshape(-1)}
    if op == "snr":
        return {"snr": _cumulative_snr(C, D[0], rd, case["which"], case["n_ell"])}
    # pca: eigenvalues (graded over many decades: the sum of squares is theirs to pin) and the total
    lam = torch.linalg.eigvalsh(C + torch.tril(C, -1).T)
    tot = _cumulative_snr(C, D[0], rd, "joint", case["n_ell"])[-1] ** 2
    return {"lam": lam.cpu().numpy(), "snr2": None, "cum_var": None, "cum_info": None, "total_snr2": float(tot)}
