"""Blocked one-sided Jacobi (csrc/pca.cu): block edges (odd and ragged sizes, fewer columns than one block pair), rows
given in any order of variance, clustered eigenvalues, and columns beyond shared memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.pca import jacobi_eigh  # noqa: E402
from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402

DEV = "cuda:0"


def _handle(nt, nl, rows):
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=nt)
    wl["bins"].update(n_ell=nl, ell_min=30.0, ell_max=2000.0)
    return Handle(wl, rows=rows)


@pytest.mark.parametrize("nt,nl", [(1, 1), (1, 2), (1, 3), (1, 13), (1, 14), (1, 15), (1, 29), (1, 64), (2, 43)])
@pytest.mark.parametrize("kind", ["graded", "cluster"])
def test_against_the_sequential_solver(nt, nl, kind):
    h = _handle(nt, nl, N.COV_ROWS_P)
    M = h.M
    g = np.random.default_rng(M)
    if kind == "graded":
        X = g.standard_normal((M, 3 * M)) + 0.4
        s = 10.0 ** g.uniform(-11, 0, M)
    else:  # equal variances, equal correlations: one large eigenvalue and M - 1 equal ones
        X = np.linalg.cholesky(np.full((M, M), 0.5) + 0.5 * np.eye(M))
        s = np.full(M, 3e-7)
    R = X @ X.T
    d = np.sqrt(np.diag(R))
    R /= np.outer(d, d)
    C = R * np.outer(s, s)
    D = s * (0.2 + g.random(M))
    got = h.pca(torch.as_tensor(C, device=DEV), torch.as_tensor(D, device=DEV))
    lam, V, _ = jacobi_eigh(C)
    ev = np.linalg.eigvalsh(R)
    eps, cond = 2.0**-53, ev[-1] / ev[0]
    # Cholesky of the unit-diagonal matrix (cond x M units) and up to ten sweeps of M rotations of four roundings, twice
    tol = (2 * cond * (M + 16) + 80 * M) * eps
    assert got["converged"] == 1
    np.testing.assert_allclose(got["lam"], lam, rtol=tol, atol=0)
    tot = float(D @ np.linalg.solve(R * np.outer(s, s), D)) if M < 2 else float(
        (D / s) @ np.linalg.solve(R, D / s))
    assert got["total_snr2"] == pytest.approx(tot, rel=tol, abs=0)
    np.testing.assert_allclose(got["cum_info"], np.cumsum(np.sort(got["snr2"])[::-1]), rtol=M * eps, atol=0)
    np.testing.assert_allclose(got["cum_var"], np.cumsum(got["snr2"]), rtol=M * eps, atol=0)
    if kind == "graded":  # distinct eigenvalues: the modes themselves
        ref = (V.T @ D) ** 2 / lam if V.shape[0] == M else None
        gap = np.min(np.abs(np.diff(lam)) / lam[1:]) if M > 1 else 1.0
        assert np.max(np.abs(got["snr2"] - ref)) <= 4 * tol / min(gap, 1.0) * tot
    f = got["cum_info"]
    for fr, key in ((0.90, "modes_90"), (0.95, "modes_95"), (0.99, "modes_99")):
        assert got[key] == 1 + int(np.argmax(np.sqrt(f) >= fr * np.sqrt(f[-1])))
    h.close()


def test_columns_beyond_shared_memory():
    """M > 14500: the columns are rotated in place.  Disjoint correlated pairs, far apart: eigenvalues known."""
    h = _handle(5, 15, N.COV_ROWS_JOINT)
    M = h.M
    assert M > 14500
    g = np.random.default_rng(5)
    s = 10.0 ** g.uniform(-8, 0, M)
    p = g.permutation(M)[:2000].reshape(1000, 2)
    r = g.uniform(-0.9, 0.9, 1000)
    C = torch.diag(torch.as_tensor(s * s, device=DEV))
    i, j = (torch.as_tensor(p[:, k], device=DEV) for k in (0, 1))
    v = torch.as_tensor(r * s[p[:, 0]] * s[p[:, 1]], device=DEV)
    C[i, j] = v
    C[j, i] = v
    D = s * (0.2 + g.random(M))
    got = h.pca(C, torch.as_tensor(D, device=DEV))
    a, b = s[p[:, 0]].astype(np.longdouble) ** 2, s[p[:, 1]].astype(np.longdouble) ** 2
    c = r.astype(np.longdouble) * np.sqrt(a * b)
    big = (a + b) / 2 + np.sqrt(((a - b) / 2) ** 2 + c * c)
    lam = s.astype(np.longdouble) ** 2
    lam[p[:, 0]], lam[p[:, 1]] = big, (a * b - c * c) / big
    eps, cond = 2.0**-53, 1.9 / 0.1
    # pairs only: rows of two entries, one rotation; entries and product each a few roundings, by cond of a pair
    tol = 32 * cond * eps
    np.testing.assert_allclose(got["lam"], np.sort(lam).astype(float), rtol=tol, atol=0)
    R1 = (D / s) ** 2
    R1[p.reshape(-1)] = 0.0
    x, z = (D / s)[p[:, 0]], (D / s)[p[:, 1]]
    tot = R1.sum() + ((x * x - 2 * r * x * z + z * z) / (1 - r * r)).sum()
    assert got["total_snr2"] == pytest.approx(tot, rel=M * eps, abs=0)
    h.close()
