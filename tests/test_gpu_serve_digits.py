"""A served FP64 request whose reservation was made with the digit rows in it uses them, also where the rest of the
device is taken: the bytes that it holds are those of the same request on an empty device."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _serve(wl, room):
    """(S/N, bytes held, footprint); `room`: bytes of the device left to the server (0: all)."""
    from paper_1812_07437_gb300.server import Server
    s = Server(n_slots=1, precision=N.COV_FP64, hbm_budget=room if room else 8 << 30)
    fill = torch.empty(_free() - room, dtype=torch.uint8, device="cuda") if room else None
    f0 = _free()
    i = s.submit(wl)
    info, snr = s.wait(i, timeout=300.0)
    assert info["state"] == N.COV_REQ_DONE, s.error(i)
    held = f0 - _free()
    s.close()
    del fill
    torch.cuda.empty_cache()
    return np.array(snr), held, info["footprint"]


def test_reserved_digits_are_used():
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=3, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=16, ell_min=10.0, ell_max=5000.0, n_chi=64, n_mass=64)
    _serve(wl, 0)  # streams and modules of the first use
    ref, held, footprint = _serve(wl, 0)
    got, held_small, again = _serve(wl, footprint + (96 << 20))
    assert again == footprint
    # M = 3064, 1176 trispectrum rows, K = 4096: 260 MB of digits and 40 MB of shared sums against 140 MB of FP64 rows;
    # narrower Cholesky scratch beside them 16 MB
    assert abs(held - held_small) <= 32 << 20, (held, held_small)
    assert np.array_equal(ref, got, equal_nan=True)
