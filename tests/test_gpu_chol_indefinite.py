"""Covariances that are far from positive definite are refused (COV_ERR_NOT_PD) wherever the rows that make them so lie:
inside a 64-column panel, over several panels of a super-panel, over several super-panels; a row whose squared factor
entries add up to many times its variance (the fixed-point entries are integers modulo 2^64, a multiple of four variances),
and one just beyond it.  And matrices as close to the limit on the other side are accepted."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


@pytest.fixture(scope="module")
def handle():
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=2, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=14, n_chi=8, n_mass=6, ell_min=10.0, ell_max=5000.0)
    h = Handle(wl, order=N.COV_ORDER_CUMULATIVE)
    assert h.M > 700
    yield h
    h.close()


def _arrow(M, row, cols, total, scale):
    """Unit correlations but for row `row`, whose entries in `cols` have the sum of squares `total`; the variances are
    `scale`."""
    C = torch.eye(M, dtype=torch.float64)
    v = np.sqrt(total / len(cols))
    assert v < 1.0
    for k, c in enumerate(cols):
        C[row, c] = C[c, row] = v if k % 2 else -v
    s = torch.sqrt(torch.as_tensor(scale, dtype=torch.float64))
    return (C * s[:, None] * s[None, :]).cuda()


# (row, first column, number of columns): one panel, two, a super-panel of four, several, and the last rows
WHERE = [(60, 3, 50), (100, 40, 60), (255, 0, 255), (500, 20, 400), (640, 300, 300), (-1, 0, 600)]


def _run(h, C, call):
    from paper_1812_07437_gb300.handle import packed_tiles
    M = h.M
    D = torch.ones(M, dtype=torch.float64, device="cuda")
    if call == "snr":
        return h.snr(C, D, N.COV_WHICH_JOINT)
    if call == "pca":
        return h.pca(C, D)["lam"]
    t = (M + 1 + 255) // 256
    Ct = torch.zeros(packed_tiles(M + 1) * 65536, dtype=torch.float64, device="cuda")
    P = torch.zeros((t * 256, t * 256), dtype=torch.float64, device="cuda")
    P[:M, :M] = C
    for ti in range(t):
        for tj in range(ti + 1):
            k = ti * (ti + 1) // 2 + tj
            Ct[k * 65536:(k + 1) * 65536] = P[256 * ti:256 * ti + 256, 256 * tj:256 * tj + 256].reshape(-1)
    return h.snr_tiles(Ct, D)


@pytest.mark.parametrize("where", WHERE)
@pytest.mark.parametrize("total", [1.01, 2.9, 3.3, 4.1, 4.6, 5.5, 8.4, 12.7, 40.3])
@pytest.mark.parametrize("call", ["snr", "tiles"])
def test_refused(handle, where, total, call):
    row, c0, n = where
    M = handle.M
    rng = np.random.default_rng(3)
    C = _arrow(M, row % M, list(range(c0, c0 + n)), total, np.exp(rng.uniform(-30, 30, M)))
    with pytest.raises(N.CovError) as e:
        _run(handle, C, call)
    assert e.value.code == N.COV_ERR_NOT_PD


@pytest.mark.parametrize("where", WHERE)
@pytest.mark.parametrize("call", ["snr", "tiles", "pca"])
def test_accepted(handle, where, call):
    row, c0, n = where
    M = handle.M
    C = _arrow(M, row % M, list(range(c0, c0 + n)), 0.999, np.ones(M))
    got = _run(handle, C, call)
    if call == "pca":  # eigenvalues 1 and 1 +- sqrt(0.999)
        assert abs(got[0] / (1.0 - np.sqrt(0.999)) - 1.0) < 1e-11 and abs(got[-1] - 1.0 - np.sqrt(0.999)) < 1e-13
    else:
        assert np.isfinite(got[-1])


def test_pca_refuses(handle):
    C = _arrow(handle.M, 300, list(range(20, 250)), 4.4, np.ones(handle.M))
    with pytest.raises(N.CovError) as e:
        _run(handle, C, "pca")
    assert e.value.code == N.COV_ERR_NOT_PD
