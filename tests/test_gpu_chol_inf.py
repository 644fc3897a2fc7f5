"""A covariance with an infinite variance is refused by the factorisations (COV_ERR_NOT_PD), as one with a NaN is."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


@pytest.mark.parametrize("where", [0, 3, -1])
@pytest.mark.parametrize("call", ["snr", "pca", "tiles"])
def test_infinite_variance(where, call):
    from paper_1812_07437_gb300.handle import Handle, packed_tiles
    h = Handle(workloads.get("tiny_2bin"), order=N.COV_ORDER_CUMULATIVE)
    M = h.M
    where %= M
    D = torch.zeros(M, dtype=torch.float64, device="cuda")
    h.spectra(D)
    if call == "tiles":
        C = torch.zeros(packed_tiles(M + 1) * 65536, dtype=torch.float64, device="cuda")
        h.assemble_band(0, M, C, N.COV_LAYOUT_TILES, N.COV_TERMS_ALL, N.COV_FP64)
        t = where // 256
        C[(t * (t + 1) // 2 + t) * 65536 + (where % 256) * 257] = float("inf")
    else:
        C = torch.zeros((M, M), dtype=torch.float64, device="cuda")
        h.assemble(C, N.COV_TERMS_ALL, N.COV_FP64)
        C[where, where] = float("inf")
    with pytest.raises(N.CovError) as e:
        {"snr": lambda: h.snr(C, D, N.COV_WHICH_JOINT), "pca": lambda: h.pca(C, D),
         "tiles": lambda: h.snr_tiles(C, D)}[call]()
    assert e.value.code == N.COV_ERR_NOT_PD
    h.close()
