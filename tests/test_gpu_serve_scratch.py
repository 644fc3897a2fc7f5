"""Cholesky scratch of a large served request: the wide form where the budget holds it, the narrow one where it does
not; the same S/N bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


def test_wide_and_narrow_scratch():
    from paper_1812_07437_gb300.server import Server
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=5, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=18, ell_min=30.0, ell_max=2000.0, n_chi=16, n_mass=16)
    got = []
    for _ in range(2):  # the default budget, then one of just the estimate
        s = Server(n_slots=1, precision=N.COV_SPLIT_BF16, hbm_budget=got[0][2] if got else 0)
        base = s.footprint(wl)[1]
        i = s.submit(wl)
        info, snr = s.wait(i, timeout=300.0)
        assert info["state"] == N.COV_REQ_DONE, s.error(i)
        got.append((info["footprint"], np.array(snr), base))
        assert info["footprint"] >= base and info["M"] > 24500
        s.close()
    assert got[0][0] > got[0][2] and got[1][0] == got[1][2]
    assert np.array_equal(got[0][1], got[1][1], equal_nan=True)
