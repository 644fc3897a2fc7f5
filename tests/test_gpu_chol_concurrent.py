"""Factorisations on several streams at once give, bit for bit, what one alone gives: the warps of a panel's thread block, and
the thread blocks of a launch, then run in any order and at any distance from each other, with other launches' blocks between
them.  Exact equality: the order of every sum is fixed by the kernels."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


# rows: under one super-panel of four panels; tens of panels, with the next super-panel's chain on the side stream
@pytest.mark.parametrize("n_ell,reps", [(8, 1000), (24, 500)])
def test_same_result_beside_other_streams(n_ell, reps):
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=2, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=n_ell, n_chi=32, n_mass=24, ell_min=10.0, ell_max=5000.0)
    hs = [Handle(wl) for _ in range(5)]
    M = hs[0].M
    D = torch.zeros(M, dtype=torch.float64, device="cuda")
    C = torch.zeros((M, M), dtype=torch.float64, device="cuda")
    hs[0].spectra(D)
    hs[0].assemble(C)
    want = [hs[0].snr(C, D, w) for w in (N.COV_WHICH_P, N.COV_WHICH_B, N.COV_WHICH_JOINT)]
    assert all(np.isfinite(x).any() for x in want)
    torch.cuda.synchronize()
    bad, start, done = [], threading.Barrier(len(hs)), threading.Event()

    def assemble():  # other kernels' thread blocks on the SMs, as in a serving mix
        s = torch.cuda.Stream()
        D2, C2 = torch.zeros_like(D), torch.zeros_like(C)
        torch.cuda.synchronize()
        start.wait()
        while not done.is_set():
            try:
                hs[4].spectra(D2, stream=s)
                hs[4].assemble(C2, precision=N.COV_SPLIT_BF16, stream=s)
                s.synchronize()
            except Exception as e:
                bad.append(("assembly", str(e)))
                return

    def run(k):
        s = torch.cuda.Stream()
        start.wait()
        for r in range(reps):
            w = (k + r) % 3
            try:
                got = hs[k].snr(C, D, w, stream=s)
            except Exception as e:
                bad.append((k, r, w, str(e)))
                continue
            if not np.array_equal(got, want[w], equal_nan=True):
                bad.append((k, r, w, float(np.nanmax(np.abs(got / want[w] - 1)))))

    ts = [threading.Thread(target=run, args=(k,)) for k in range(4)]
    other = threading.Thread(target=assemble)
    for t in ts + [other]:
        t.start()
    for t in ts:
        t.join()
    done.set()
    other.join()
    for h in hs:
        h.close()
    assert not bad, (len(bad), bad[:5])
