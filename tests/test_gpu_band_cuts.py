"""A large band of the split form is assembled in sub-bands with the products on a side stream, a small one in turn:
the same rows in one large call and in small calls agree bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


@pytest.mark.parametrize("order", [N.COV_ORDER_NATURAL, N.COV_ORDER_CUMULATIVE])
def test_cut_and_uncut_bands_agree(order):
    from paper_1812_07437_gb300.handle import Handle, packed_tiles
    h = Handle(workloads.get("cfg3_10bin"), order=order)
    h.spectra()
    tb = (h.M + 255) // 256
    t0 = tb - 30  # 30 tile rows of ~700 tiles: above 64 waves of the device for each of two sub-bands
    out = []
    for cuts in ((t0, tb), (t0, t0 + 1, t0 + 9, t0 + 20, tb)):
        C = torch.zeros((packed_tiles(h.M) - packed_tiles(256 * t0)) * 65536, dtype=torch.float64, device="cuda")
        for a, b in zip(cuts[:-1], cuts[1:]):
            lo = (packed_tiles(256 * a) - packed_tiles(256 * t0)) * 65536
            h.assemble_band(256 * a, min(256 * b, h.M) - 256 * a, C[lo:], N.COV_LAYOUT_TILES, N.COV_TERMS_ALL,
                            N.COV_SPLIT_BF16)
        torch.cuda.synchronize()
        out.append(C)
    assert float(out[0].abs().max()) > 0.0
    assert torch.equal(out[0], out[1])
    h.close()
