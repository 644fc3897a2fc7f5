"""FP64 form by digits, element by element: every covariance element to FP64 accuracy relative to the sum of its own
terms' magnitudes (not only to sqrt(C_aa C_bb)), however little its two rows overlap; against 64-bit-mantissa sums of the
library's own tables, and for the terms that use the trispectrum table against the FP64 rows' form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402

U = 2.0**-53
# A factor row's entry is a product of ~12 rounded factors (a cube root, two divisions, seven tables), once per side: 24 U
# if all errors agree.  The contraction: the digits drop products below 2^-56 of a K block's row norms (32 of them) and
# round the entries to 2^-56 of the norm; where the two rows of a block of several nodes overlap by a twentieth or more
# that is below 20 U.
TOL = 44 * U

# tomographic bins, ell bins, range, N_chi, N_M, N_conc, photo-z: rows with little overlap (narrow bins, wide ell range),
# K blocks across several nodes (N_M of 5 and 12), within one (64), between (24, 33), K below and above 4096, and more
# than 2048 K blocks
CASES = [(5, 8, 2.0, 2e4, 64, 64, 0, 0.0), (10, 4, 10.0, 2e4, 33, 12, 0, 0.0), (4, 6, 2.0, 2e4, 16, 24, 8, 0.0),
         (2, 9, 10.0, 5000.0, 24, 5, 0, 0.05), (3, 7, 10.0, 2e4, 31, 33, 0, 0.0), (2, 6, 10.0, 5000.0, 128, 40, 0, 0.0),
         (2, 6, 2.0, 2e4, 1100, 64, 0, 0.0)]


def _wl(nt, nl, lo, hi, nchi, nm, nc, photoz):
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=nt, photoz_sigma0=photoz)
    wl["bins"].update(n_ell=nl, n_chi=nchi, n_mass=nm, n_conc=nc, sigma_lnc=0.3, ell_min=lo, ell_max=hi)
    return wl


def _form(wl, terms, budget):
    from paper_1812_07437_gb300.handle import Handle
    h = Handle(wl, hbm_budget=budget)
    h.spectra()
    C = torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda")
    h.assemble(C, terms, N.COV_FP64)
    torch.cuda.synchronize()
    return h, C.cpu().numpy()


def _rows(h, wl, pick):
    """Factor rows and super-sample rows of the picked data-vector rows, from the library's tables, in long double."""
    ld = np.longdouble
    nchi = int(wl["bins"]["n_chi"])
    T = {k: h.table(k).astype(ld) for k in ("chi", "wchi", "mass", "conc_weights", "f", "U", "W", "sigw2", "RP3", "RB3")}
    nm = len(T["mass"])
    nmb, nc = nm // len(T["conc_weights"]), len(T["conc_weights"])
    rho = ld(2.77536627e11) * ld(wl["cosmology"]["Om"])
    mb = T["mass"].reshape(nmb, nc)[:, 0]
    dl = np.log(ld(wl["bins"]["m_max"]) / ld(wl["bins"]["m_min"])) / (nmb - 1)
    om = dl * mb
    om[0] *= ld(0.5)
    om[-1] *= ld(0.5)
    om = (om[:, None] * T["conc_weights"][None, :]).reshape(-1)
    Uk, W, f = T["U"].reshape(-1, nchi, nm), T["W"].reshape(-1, nchi), T["f"].reshape(nchi, nm)
    omega = ld(4.0 * np.pi * wl["bins"]["f_sky"])
    base = np.sqrt(T["wchi"][:, None] * om[None, :] * f / omega)
    mr = T["mass"] / rho
    RP3, RB3 = T["RP3"].reshape(-1, nchi), T["RB3"].reshape(-1, nchi)
    out, ssc = [], []
    for r in h.row_desc()[pick]:
        w = W[r[4]] * W[r[5]]
        s = np.sqrt(T["wchi"] * T["sigw2"])
        if r[0] == 0:
            v = base * mr**2 * Uk[r[1]] * Uk[r[2]] * (w / T["chi"]**3)[:, None]
            s = s * w / T["chi"]**2 * RP3[r[1]]
        else:
            w = w * W[r[6]]
            v = base * mr**3 * Uk[r[1]] * Uk[r[2]] * Uk[r[3]] * (w / T["chi"]**5)[:, None]
            s = s * w / T["chi"]**4 * RB3[r[7]]
        out.append(v.reshape(-1))
        ssc.append(s)
    return np.array(out), np.array(ssc)


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("ssc", [False, True])
def test_elements_of_the_contraction(case, ssc):
    wl = _wl(*case)
    h, C = _form(wl, N.COV_TERM_1H | (N.COV_TERM_SSC if ssc else 0), 0)
    rng = np.random.default_rng(5)
    nP = h.n_P
    pick = np.unique(np.concatenate([rng.integers(0, nP, 40), rng.integers(nP, h.M, 80), [0, nP - 1, h.M - 1]]))
    A, S = _rows(h, wl, pick)
    if ssc:
        A = np.concatenate([A, S], axis=1)
    ref, mag = A @ A.T, np.abs(A) @ np.abs(A).T
    got = C[np.ix_(pick, pick)]
    i, j = np.tril_indices(len(pick))
    d = np.sqrt(np.diag(mag))
    assert np.min((mag / np.outer(d, d))[i, j]) < 0.2  # some rows do overlap little
    err = (np.abs(got - ref) / mag)[i, j].astype(np.float64)
    assert np.max(err) <= TOL, (np.max(err) / U, np.sqrt(np.mean(err**2)) / U)
    h.close()


@pytest.mark.parametrize("case", CASES[:4])
def test_elements_with_the_trispectrum_table(case):
    wl = _wl(*case)
    h, a = _form(wl, N.COV_TERM_BBPT, 0)
    M, nchi = h.M, case[4]
    K, legs = nchi * case[5] * max(1, case[6]), case[0] * case[1]
    tr = legs * (legs + 1) // 2
    h.close()
    rows = 8 * (M * K + M * nchi + tr * K + tr * tr) + (24 << 20)  # room for the FP64 rows, not for the digits' sums
    h, b = _form(wl, N.COV_TERM_BBPT, rows)
    h.close()
    i, j = np.tril_indices(M)
    a, b = a[i, j], b[i, j]
    # the FP64 rows' own chain rounds K positive terms, 44 U for the rows and what the digits leave out
    assert np.all(np.abs(a - b) <= (TOL + np.sqrt(K) * 8 * U) * np.abs(b))
