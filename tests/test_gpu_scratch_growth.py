"""The Cholesky scratch that a handle ends up with does not depend on what it factorised before, and growing it does not
need the old and the new buffer at the same time."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


def _wl():
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=3, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=16, n_chi=12, n_mass=10, ell_min=10.0, ell_max=5000.0)
    return wl


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _run(wl, first):
    """(S/N of a batch, device bytes the handle holds after it); `first`: selections factorised before the batch."""
    from paper_1812_07437_gb300.handle import Handle
    cosmos = [dict(wl["cosmology"], sigma8=wl["cosmology"]["sigma8"] * f) for f in (1.0, 1.02)]
    M = 3064
    C = torch.zeros((M, M), dtype=torch.float64, device="cuda")
    D = torch.zeros(M, dtype=torch.float64, device="cuda")
    f0 = _free()
    h = Handle(wl)
    assert h.M == M
    h.spectra(D)
    h.assemble(C, N.COV_TERMS_ALL, N.COV_SPLIT_BF16)
    for w in first:
        h.snr(C, D, w)
    snr, _, _ = h.batch_snr(cosmos, precision=N.COV_SPLIT_BF16)
    held = f0 - _free()
    h.close()
    return snr, held


def test_batch_after_a_small_factorisation():
    wl = _wl()
    _run(wl, [])  # modules, streams and graphs of the first use are not the handle's
    ref, fresh = _run(wl, [N.COV_WHICH_JOINT])
    got, held = _run(wl, [N.COV_WHICH_P])
    assert np.array_equal(ref, got, equal_nan=True)
    # scratch of 3064 rows: 2 x 24 row blocks x 8 K blocks x 56 KB = 22 MB in super-panels of four panels, 5.5 MB with one;
    # device memory comes in pieces of 2 MB
    assert abs(held - fresh) <= 8 << 20, (held, fresh)
