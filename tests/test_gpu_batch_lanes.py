"""Factorisations of a batched step side by side (csrc/batch.cu): the same numbers as the separate calls, bit for bit,
from the size where the second workspace is taken, and as one after the other under a memory budget; an empty
selection; a matrix that is not positive definite."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


def _wl(nt, nl):
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=nt, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=nl, n_chi=12, n_mass=10, ell_min=30.0, ell_max=2000.0)
    return wl


@pytest.mark.parametrize("nt,nl,rows", [(2, 8, N.COV_ROWS_JOINT), (3, 9, N.COV_ROWS_JOINT), (4, 9, N.COV_ROWS_JOINT),
                                        (5, 60, N.COV_ROWS_P), (3, 10, N.COV_ROWS_B)])
@pytest.mark.parametrize("budget", [0, 32 << 30])
def test_batch_equals_separate_calls(nt, nl, rows, budget):
    from paper_1812_07437_gb300.handle import Handle
    wl = _wl(nt, nl)
    cosmos = [dict(wl["cosmology"], sigma8=wl["cosmology"]["sigma8"] * f) for f in (1.0, 1.02, 0.97)]
    h = Handle(wl, rows=rows, hbm_budget=budget)
    got, D, _ = h.batch_snr(cosmos, precision=N.COV_FP64, with_D=True)
    again, _, _ = h.batch_snr(cosmos[:1], precision=N.COV_FP64, with_D=True)
    h.close()
    h = Handle(wl, rows=rows)
    Dk = torch.zeros(h.M, dtype=torch.float64, device="cuda")
    C = torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda")
    for k, c in enumerate(cosmos):
        h.update(c)
        h.spectra(Dk)
        h.assemble(C, N.COV_TERMS_ALL, N.COV_FP64)
        assert np.array_equal(Dk.cpu().numpy(), D[k])
        for w in (N.COV_WHICH_P, N.COV_WHICH_B, N.COV_WHICH_JOINT):
            ref = h.snr(C, Dk, w)
            if not np.all(np.isnan(ref)) or k == 0:
                assert np.array_equal(ref, got[k][w], equal_nan=True), (k, w)
    assert np.array_equal(got[0], again[0], equal_nan=True)
    h.close()


# rows of all cosmologies from which the second workspace is taken, and the largest matrix for it (csrc/batch.cu)
LANE_MIN_ROWS, LANE_MAX_ROWS = 2048, 8192


@pytest.mark.parametrize("nt,nl,precision", [(3, 9, N.COV_FP64), (4, 9, N.COV_SPLIT_BF16)])
def test_a_failed_factorisation_beside_another(nt, nl, precision):
    """Without the terms that give power spectra a variance every factorisation of the step fails; the handle then gives
    what it gave before, bit for bit."""
    from paper_1812_07437_gb300.handle import Handle
    wl = _wl(nt, nl)
    cosmos = [dict(wl["cosmology"], sigma8=wl["cosmology"]["sigma8"] * f) for f in (1.0, 1.02, 0.97)]
    h = Handle(wl)
    assert (h.M - h.n_P) * len(cosmos) >= LANE_MIN_ROWS and h.M - h.n_P <= LANE_MAX_ROWS
    ref, D, _ = h.batch_snr(cosmos, precision=precision, with_D=True)
    for terms in (N.COV_TERM_PB, N.COV_TERM_BBPT | N.COV_TERM_PB):
        with pytest.raises(N.CovError) as e:
            h.batch_snr(cosmos, terms=terms, precision=precision)
        assert e.value.code == N.COV_ERR_NOT_PD
    got, D2, _ = h.batch_snr(cosmos, precision=precision, with_D=True)
    assert np.array_equal(ref, got, equal_nan=True) and np.array_equal(D, D2)
    h.close()
