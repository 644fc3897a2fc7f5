"""Split-form rows (csrc/syrk_tc.cu): signature tables and row split at the edges of their chunks (N_M around 8, 32 and
128 and beyond, K' of any parity), against the FP64 form of the same terms."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


@pytest.mark.parametrize("nchi,nm", [(2, 2), (5, 3), (9, 8), (7, 31), (6, 33), (33, 40), (4, 127), (4, 128), (5, 129),
                                     (3, 136), (3, 300)])
@pytest.mark.parametrize("nt,nl", [(1, 3), (2, 8), (3, 5)])
def test_rows_against_the_fp64_form(nt, nl, nchi, nm):
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=nt, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=nl, ell_min=30.0, ell_max=2000.0, n_chi=nchi, n_mass=nm)
    h = Handle(wl)
    h.spectra()
    C = [torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda") for _ in range(2)]
    h.assemble(C[0], N.COV_TERMS_ALL, N.COV_FP64)
    h.assemble(C[1], N.COV_TERMS_ALL, N.COV_SPLIT_BF16)
    torch.cuda.synchronize()
    d = torch.sqrt(torch.diagonal(C[0]))
    err = float((torch.tril(C[0] - C[1]).abs() / torch.outer(d, d)).max())
    # hi + lo carries 2^-17 of an entry (twice per product), the dropped lo lo 2^-16, the table and weight 2^-24 each;
    # FP32 accumulation of K' = N_chi (N_M + 1) terms
    assert err <= 4 * 2.0**-17 + 2 * 2.0**-16 + nchi * (nm + 1) * 3 * 2.0**-24
    h.close()
