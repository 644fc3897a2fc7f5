"""Split-form contraction by 128 x 128 tiles (csrc/syrk_tc.cu: small matrices and the last partial wave): the sums of
the one-CTA 256 x 256 kernel bit for bit, at the edges of the 16-column steps, of the tiles and of the wave."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402

# (tomographic bins, ell bins, rows): M = 1, 15, 16, 17, 63, 126, 129, 192, 255, 258, 384; joint: small, one partial
# wave, whole waves and a rest
SIZES = [(1, n, N.COV_ROWS_P) for n in (1, 15, 16, 17, 63)] + [
    (2, 42, N.COV_ROWS_P), (2, 43, N.COV_ROWS_P), (2, 64, N.COV_ROWS_P), (5, 17, N.COV_ROWS_P), (3, 43, N.COV_ROWS_P),
    (3, 64, N.COV_ROWS_P), (1, 8, N.COV_ROWS_JOINT), (2, 8, N.COV_ROWS_JOINT), (4, 9, N.COV_ROWS_JOINT),
    (5, 8, N.COV_ROWS_JOINT), (5, 12, N.COV_ROWS_JOINT), (4, 14, N.COV_ROWS_JOINT)]


@pytest.mark.parametrize("nt,nl,rows", SIZES)
@pytest.mark.parametrize("nchi,nm", [(7, 5), (16, 24)])
def test_same_sums_as_one_cta_per_tile(nt, nl, rows, nchi, nm):
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=nt)
    wl["bins"].update(n_ell=nl, ell_min=30.0, ell_max=2000.0, n_chi=nchi, n_mass=nm)
    out = []
    for tc in (N.COV_TC_AUTO, N.COV_TC_SINGLE):
        h = Handle(wl, rows=rows, tc_kernel=tc)
        h.spectra()
        C = torch.full((h.M, h.M), 3.0, dtype=torch.float64, device="cuda")
        h.assemble(C, N.COV_TERMS_ALL, N.COV_SPLIT_BF16)
        torch.cuda.synchronize()
        out.append(C)
        h.close()
    assert torch.equal(out[0], out[1])
    assert bool((torch.triu(out[0], 1) == torch.triu(torch.full_like(C, 3.0), 1)).all())
