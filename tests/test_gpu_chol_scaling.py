"""The Cholesky's scaling rounds nothing: variances of pairs of strongly correlated rows given the pair's other row, for
variances over many decades, against exact fractions, to what the factorisation itself rounds."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402

EPS = 2.0**-20


@pytest.mark.parametrize("decades", [0.0, 2.0, 12.0, 100.0])
def test_correlated_pairs(decades):
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=2, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=10, n_chi=8, n_mass=6, ell_min=10.0, ell_max=5000.0)
    h = Handle(wl, order=N.COV_ORDER_CUMULATIVE)
    M = h.M
    rng = np.random.default_rng(17)
    d = 10.0 ** rng.uniform(-decades, decades, M) * rng.uniform(1.0, 4.0, M)
    C = torch.diag(torch.as_tensor(d))
    pairs = []
    for k0 in range(0, M - 64, 64):  # both rows of a pair in one panel of 64 columns
        i, j = np.sort(rng.choice(64, 2, replace=False)) + k0
        C[j, i] = C[i, j] = float(np.sqrt(d[i]) * np.sqrt(d[j]) * (1.0 - EPS))
        pairs.append((i, j))
    C = C.cuda()
    worst = 0.0
    for i, j in pairs:
        D = torch.zeros(M, dtype=torch.float64, device="cuda")
        D[j] = float(np.sqrt(d[j]))
        got = Fraction(float(h.snr(C, D, N.COV_WHICH_JOINT)[-1])) ** 2
        a, b, c = (Fraction(float(C[x, y])) for x, y in ((i, i), (j, i), (j, j)))
        want = Fraction(float(D[j])) ** 2 * a / (a * c - b * b)
        worst = max(worst, abs(float(got / want) - 1.0))
    # the pivot c' (1 - rho^2), 1 - rho^2 = 2^-19, from l = b' / sqrt(a'): the reciprocal square root to 2^-54, l to 2^-58,
    # c' in [1/4, 1): 2^19 (2^-53 + 2^-56) of the pivot; 2^-50 for the FP64 rounding of y, its square and the root
    assert worst <= 2.0**19 * (2.0**-53 + 2.0**-56) + 2.0**-50, np.log2(worst)
    h.close()
