"""Non-finite factor rows in the FP64 form: what a cosmology without a finite spectrum, halo integrals that overflow or a
failed quadrature rule put into the rows has to arrive in the covariance as NaN (or infinity), with the digits as with
FP64 rows, and finite rows beside them keep their values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


def _wl(**bins):
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=2, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=6, n_chi=17, n_mass=24, ell_min=30.0, ell_max=2000.0, **bins)
    return wl


def _assemble(wl, cosmology, terms, digits):
    """The lower triangle; digits False: a budget that holds the FP64 rows but not the digits' shared sums."""
    from paper_1812_07437_gb300.handle import Handle
    h = Handle(wl, hbm_budget=0 if digits else 48 << 20)
    h.update(cosmology)
    h.spectra()
    C = torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda")
    h.assemble(C, terms, N.COV_FP64)
    torch.cuda.synchronize()
    c = C.cpu().numpy()[np.tril_indices(h.M)]
    h.close()
    return c


@pytest.mark.parametrize("bad", [dict(w0=float("nan")), dict(ns=float("nan")), dict(sigma8=float("inf")),
                                 dict(h=float("inf"))])
@pytest.mark.parametrize("terms", [N.COV_TERM_1H, N.COV_TERM_1H | N.COV_TERM_SSC, N.COV_TERM_BBPT, N.COV_TERMS_ALL])
def test_non_finite_cosmology(bad, terms):
    wl = _wl()
    cosmo = dict(wl["cosmology"], **bad)
    ref = _assemble(wl, cosmo, terms, False)
    got = _assemble(wl, cosmo, terms, True)
    if "sigma8" not in bad:
        assert not np.any(np.isfinite(ref)) or terms == N.COV_TERM_BBPT
    assert np.array_equal(np.isfinite(ref), np.isfinite(got))
    fin = np.isfinite(ref)
    assert np.allclose(got[fin], ref[fin], rtol=1e-12, atol=0.0)


def test_good_cosmology_after_a_bad_one():
    from paper_1812_07437_gb300.handle import Handle
    wl = _wl()
    h = Handle(wl)
    C = torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda")
    out = []
    for c in (wl["cosmology"], dict(wl["cosmology"], ns=float("nan")), wl["cosmology"]):
        h.update(c)
        h.spectra()
        h.assemble(C, N.COV_TERMS_ALL, N.COV_FP64)
        torch.cuda.synchronize()
        out.append(C.cpu().numpy()[np.tril_indices(h.M)])
    assert np.all(np.isfinite(out[0])) and np.array_equal(out[0], out[2])
    assert not np.any(np.isfinite(out[1]))
    h.close()
