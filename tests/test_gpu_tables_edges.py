"""Tables, spectra and data vector at the sizes where the builders' blocks are ragged: fewer nodes than a warp, one
node past a slab, one ell bin (no mixed triangles), many tomographic bins, concentration scatter with the Bullock
median, and a survey deep enough that the chi intervals are wide."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = {
    "one_ell": dict(nt=1, nl=1, nchi=2, nm=2),
    "past_slab": dict(nt=2, nl=3, nchi=33, nm=33),
    "many_bins": dict(nt=13, nl=4, nchi=17, nm=31),
    "conc": dict(nt=2, nl=5, nchi=9, nm=11, n_conc=3, conc_model=1),
    "deep": dict(nt=3, nl=4, nchi=20, nm=16, zmax=12.0, photoz=0.0),
    "no_scatter_edge": dict(nt=4, nl=6, nchi=40, nm=12, photoz=0.0, zmin=0.3),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_ragged_tables(name):
    torch = pytest.importorskip("torch")
    from oracle.pipeline import OracleRun
    from paper_1812_07437_gb300 import workloads
    from paper_1812_07437_gb300.handle import Handle
    k = dict(CASES[name])
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=k["nt"], photoz_sigma0=k.get("photoz", 0.05), zmin=k.get("zmin", 0.0), zmax=k.get("zmax", 3.0))
    wl["bins"].update(n_ell=k["nl"], n_chi=k["nchi"], n_mass=k["nm"], n_conc=k.get("n_conc", 0), sigma_lnc=0.18,
                      conc_model=k.get("conc_model", 0))
    h = Handle(wl)
    D = torch.zeros(h.M, dtype=torch.float64, device="cuda")
    for _ in range(2):  # the second pass reuses every buffer
        h.update(wl["cosmology"])
        h.spectra(D)
    r = OracleRun(wl)
    # every quantity is a short FP64 sum of the same terms: 1e-10 as for the other parity tests
    got = {"z": (h.table("z"), r.T.z), "growth": (h.table("growth"), r.T.D), "W": (h.table("W"), r.T.W.ravel()),
           "sigw2": (h.table("sigw2"), r.T.sigW2), "D": (D.cpu().numpy(), r.D)}
    for what, (a, b) in got.items():
        a, b = np.ravel(a), np.ravel(b)
        assert np.max(np.abs(a - b)) <= 1e-10 * np.max(np.abs(b)), what
    Ps = h.table("Ps").reshape(k["nl"], k["nt"], k["nt"])
    assert np.max(np.abs(Ps / r.S.Ps - 1)) < 1e-10
    h.close()
