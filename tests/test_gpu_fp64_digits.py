"""FP64 form of the contraction by exact digit sums (csrc/syrk_sl.cu): at the edges of its blocks (128 rows, 32 K,
8 tile rows per launch group, parts of a K range, N_M below and across a K block, concentration scatter, super-sample
columns), against the FP64 CUDA-core product of the same rows and against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _wl(nt, nl, nchi, nm, n_conc=0, photoz=0.05):
    from paper_1812_07437_gb300 import workloads
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=nt, photoz_sigma0=photoz)
    wl["bins"].update(n_ell=nl, n_chi=nchi, n_mass=nm, n_conc=n_conc, sigma_lnc=0.18, ell_min=30.0, ell_max=2000.0)
    return wl


def _lower(h, terms, precision, band):
    import torch
    from paper_1812_07437_gb300 import native as N
    C = torch.full((h.M, h.M), 7.0, dtype=torch.float64, device="cuda")
    if band:
        step = 256 * max(1, h.M // 512)
        for r0 in range(0, h.M, step):
            n = min(step, h.M - r0)
            h.assemble_band(r0, n, C[r0:r0 + n], N.COV_LAYOUT_ROWS, terms, precision)
    else:
        h.assemble(C, terms, precision)
    torch.cuda.synchronize()
    c = C.cpu().numpy()
    assert np.all(np.triu(c, 1)[np.triu_indices(h.M, 1)] == 7.0)  # nothing above the diagonal is written
    return np.tril(c) + np.tril(c, -1).T


CASES = [(1, 3, 4, 5, 0), (1, 8, 16, 12, 0), (2, 5, 11, 33, 0), (2, 6, 16, 32, 3), (3, 6, 9, 31, 0), (4, 6, 24, 16, 0),
         (5, 7, 33, 24, 0)]


@pytest.mark.parametrize("case", CASES)
@pytest.mark.parametrize("band", [False, True])
def test_against_the_oracle(case, band):
    pytest.importorskip("torch")
    from oracle.pipeline import OracleRun
    from paper_1812_07437_gb300 import native as N
    from paper_1812_07437_gb300.handle import Handle
    nt, nl, nchi, nm, nc = case
    if nt == 5 and band:
        pytest.skip("the dense call covers this size")
    wl = _wl(nt, nl, nchi, nm, nc)
    h = Handle(wl)
    h.spectra()
    got = _lower(h, N.COV_TERMS_ALL, N.COV_FP64, band)
    if nt <= 3:
        ref = OracleRun(wl).cov.full()
    else:  # a budget without room for the digits leaves the FP64 rows and the CUDA-core product
        ref = _cuda_core(wl)
    d = np.sqrt(np.diag(ref))
    # both sides round every sum of ~K positive terms: 1e-10 as for every other FP64 parity test
    assert np.max(np.abs(got - ref) / np.outer(d, d)) < 1e-10
    h.close()


def _cuda_core(wl, terms=None):
    """The FP64 form under an hbm_budget that holds its FP64 rows but not the digits."""
    from paper_1812_07437_gb300 import native as N
    from paper_1812_07437_gb300.handle import Handle
    h = Handle(wl, hbm_budget=1 << 40)
    M, K, nchi = h.M, int(wl["bins"]["n_chi"]) * int(wl["bins"]["n_mass"]) * max(1, int(wl["bins"].get("n_conc", 0))), int(
        wl["bins"]["n_chi"])
    h.close()
    legs = int(wl["bins"]["n_ell"]) * int(wl["nz"]["n_tomo"])
    tr = legs * (legs + 1) // 2
    rows = 8 * (M * K + M * nchi + tr * K + tr * tr) + (24 << 20)  # the digits' shared sums alone take 40 MB
    h = Handle(wl, hbm_budget=rows)
    h.spectra()
    c = _lower(h, N.COV_TERMS_ALL if terms is None else terms, N.COV_FP64, False)
    h.close()
    return c


@pytest.mark.parametrize("terms", [1, 2, 4, 6, 16, 18, 20, 31])
def test_term_sets_match_the_cuda_core_form(terms):
    pytest.importorskip("torch")
    from paper_1812_07437_gb300 import native as N
    from paper_1812_07437_gb300.handle import Handle
    wl = _wl(3, 7, 20, 17)
    h = Handle(wl)
    h.spectra()
    got = _lower(h, terms, N.COV_FP64, False)
    ref = _cuda_core(wl, terms)
    d = np.sqrt(np.diag(_cuda_core(wl)))
    # the digits' error is below 1e-14 of sqrt(C_aa C_bb), the FMA chain's below K 2^-53 = 4e-14
    assert np.max(np.abs(got - ref) / np.outer(d, d)) < 1e-13
    if terms == 2:  # the second assembly reuses every buffer, bit for bit
        assert np.array_equal(got, _lower(h, terms, N.COV_FP64, False))
    h.close()


def test_larger_than_one_launch_group():
    """M = 3064 rows (24 tile rows, three launch groups) against a plain FP64 product of the library's own tables."""
    torch = pytest.importorskip("torch")
    from paper_1812_07437_gb300 import native as N
    from paper_1812_07437_gb300.handle import Handle
    wl = _wl(3, 16, 40, 24)
    wl["bins"].update(ell_min=10.0, ell_max=5000.0)
    h = Handle(wl)
    h.spectra()
    got = _lower(h, N.COV_TERM_1H, N.COV_FP64, False)
    rd = h.row_desc()
    nchi, nm = 40, 24
    T = {k: torch.as_tensor(h.table(k)) for k in ("chi", "wchi", "mass", "f", "U", "W")}
    m = T["mass"]
    rho = 2.77536627e11 * wl["cosmology"]["Om"]
    dl = np.log(1e16 / 1e10) / (nm - 1)
    om = dl * m
    om[0] *= 0.5
    om[-1] *= 0.5
    U, W, f = T["U"].reshape(16, nchi, nm), T["W"].reshape(3, nchi), T["f"].reshape(nchi, nm)
    omega = 4 * np.pi * wl["bins"]["f_sky"]
    base = torch.sqrt(T["wchi"][:, None] * om * f / omega) * (m / rho) ** 2
    R = torch.as_tensor(rd.astype(np.int64))
    isB = R[:, 0] == 1
    w = W[R[:, 4]] * W[R[:, 5]] / T["chi"] ** 3
    w = torch.where(isB[:, None], w * W[R[:, 6].clamp(min=0)] / T["chi"] ** 2, w)
    v = base * U[R[:, 1]] * U[R[:, 2]] * w[:, :, None]
    v = torch.where(isB[:, None, None], v * (m / rho) * U[R[:, 3]], v).reshape(len(rd), -1)
    ref = (v @ v.T).numpy()
    d = np.sqrt(np.diag(ref))
    assert np.max(np.abs(got - ref) / np.outer(d, d)) < 1e-12
    h.close()
