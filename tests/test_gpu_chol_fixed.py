"""Fixed-point Cholesky (csrc/chol_fx.cu) at the edges of its panels (64 columns), tiles (128 x 64), super-panels
(256 or 512 columns) and of the look-ahead, on correlation matrices with rows of very different scale."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402

DEV = "cuda:0"


def _handle(nt, nl, rows):
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=nt)
    wl["bins"].update(n_ell=nl, ell_min=30.0, ell_max=2000.0)
    return Handle(wl, rows=rows)


def _problem(M, smooth, seed):
    """A covariance (scales over 14 decades), its correlation matrix and a data vector."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    if smooth:
        x = torch.arange(M, dtype=torch.float64, device=DEV)
        R = torch.exp(-(x[:, None] - x[None, :]).abs() / 12.0)
    else:
        G = torch.randn(M, 2 * M, generator=g, dtype=torch.float64, device=DEV) + 0.5
        R = G @ G.T
    s = torch.rsqrt(torch.diagonal(R))
    R = R * s[:, None] * s[None, :]
    d = 10.0 ** (14.0 * torch.rand(M, generator=g, dtype=torch.float64, device=DEV) - 12.0)
    D = d * (0.1 + torch.rand(M, generator=g, dtype=torch.float64, device=DEV))
    return R * d[:, None] * d[None, :], R, D


def _reference(h, C, D):
    rd = h.row_desc()
    mb = np.where(rd[:, 0] == 0, rd[:, 1], rd[:, 3])
    p = torch.as_tensor(np.argsort(mb, kind="stable"), device=DEV)
    Cs = C[p][:, p]
    s = torch.rsqrt(torch.diagonal(Cs))
    L = torch.linalg.cholesky(Cs * s[:, None] * s[None, :])
    y = torch.linalg.solve_triangular(L, (D[p] * s)[:, None], upper=False)[:, 0].cpu().numpy()
    cum = np.cumsum(y * y)
    return np.array([np.sqrt(cum[np.searchsorted(mb[p.cpu().numpy()], c, side="right") - 1]) for c in range(h.n_ell)])


# (tomographic bins, ell bins): M = 1, 2, 31, 63, 64, 66, 126, 129, 192, 252, 255, 258, 320, 384
SMALL = [(1, 1), (1, 2), (1, 31), (1, 63), (1, 64), (2, 22), (2, 42), (2, 43), (2, 64), (3, 42), (5, 17), (3, 43), (4, 32),
         (3, 64)]


def _check(h, smooth):
    M = h.M
    C, R, D = _problem(M, smooth, M)
    got = h.snr(C, D, N.COV_WHICH_P if h.n_B == 0 or M == h.n_P else N.COV_WHICH_JOINT)
    ref = _reference(h, C, D)
    lam = torch.linalg.eigvalsh(R)
    cond = float(lam[-1] / lam[0])
    # any backward stable Cholesky of the unit-diagonal matrix: |d(y^T y)| / (y^T y) <= cond x M 2^-53 (scaling: a few
    # units more), on both sides; the root halves it
    tol = cond * (M + 16) * 2.0**-53
    assert np.max(np.abs(got / ref - 1.0)) <= tol, (M, cond)


@pytest.mark.parametrize("nt,nl", SMALL)
def test_panel_and_tile_edges(nt, nl):
    h = _handle(nt, nl, N.COV_ROWS_P)
    _check(h, False)
    _check(h, True)
    h.close()


# joint row sets: without and with the look-ahead, super-panels of four and of eight panels
@pytest.mark.parametrize("nt,nl", [(3, 5), (4, 9), (5, 10), (5, 14)])
def test_super_panels_and_look_ahead(nt, nl):
    h = _handle(nt, nl, N.COV_ROWS_JOINT)
    _check(h, True)
    h.close()


@pytest.mark.parametrize("nt,nl", [(1, 64), (2, 43), (3, 43)])
def test_not_positive_definite(nt, nl):
    h = _handle(nt, nl, N.COV_ROWS_P)
    M = h.M
    C, _, D = _problem(M, False, 3 * M)
    good = h.snr(C, D, N.COV_WHICH_P)
    d = torch.sqrt(torch.diagonal(C))

    def bad(edit):
        B = C.clone()
        edit(B)
        with pytest.raises(N.CovError) as e:
            h.snr(B, D, N.COV_WHICH_P)
        assert e.value.code == N.COV_ERR_NOT_PD

    def triple(B):  # correlations 0.9, 0.9, -0.9 of three rows: every entry below 1, indefinite
        for i, j, r in ((M // 2, 0, 0.9), (M - 1, 0, 0.9), (M - 1, M // 2, -0.9)):
            B[i, j] = B[j, i] = r * d[i] * d[j]

    bad(triple)
    bad(lambda B: B.__setitem__((M - 1, M - 1), 0.0))
    bad(lambda B: B.__setitem__((M // 2, M // 2), float("nan")))
    bad(lambda B: B.__setitem__((M - 1, 0), float("nan")))
    bad(lambda B: B.__setitem__((M - 1, 1), float("inf")))
    bad(lambda B: B.__setitem__((M - 1, 0), float(2.0 * d[M - 1] * d[0])))
    assert np.array_equal(h.snr(C, D, N.COV_WHICH_P), good)
    h.close()


def test_packed_tiles_off_16_bytes():
    """COV_CHOL_TILE takes tiles that are only 8-byte aligned, with the same numbers; COV_CHOL_AUTO refuses them."""
    from paper_1812_07437_gb300.handle import Handle, packed_tiles
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=3, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=6, ell_min=30.0, ell_max=2000.0)
    out = []
    for off, kernel in ((0, N.COV_CHOL_TILE), (1, N.COV_CHOL_TILE), (1, N.COV_CHOL_AUTO)):
        h = Handle(wl, order=N.COV_ORDER_CUMULATIVE, chol_kernel=kernel)
        D = torch.zeros(h.M, dtype=torch.float64, device=DEV)
        h.spectra(D)
        Ct = torch.zeros(packed_tiles(h.M + 1) * 65536 + 1, dtype=torch.float64, device=DEV)[off:]
        h.assemble_band(0, h.M, Ct, N.COV_LAYOUT_TILES, N.COV_TERMS_ALL, N.COV_FP64)
        if kernel == N.COV_CHOL_TILE:
            out.append(h.snr_tiles(Ct, D))
        else:
            with pytest.raises(N.CovError) as e:
                h.snr_tiles(Ct, D)
            assert e.value.code == N.COV_ERR_CUDA
        h.close()
    assert np.array_equal(out[0], out[1], equal_nan=True)


def test_scratch_under_a_budget():
    """A budget that holds either the wide scratch or a later workspace: the scratch goes, the call is served."""
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("mid_3bin")
    free = Handle(wl)
    M = free.M
    C, _, D = _problem(M, False, 11)
    ref = free.snr(C, D, N.COV_WHICH_JOINT)
    lam = free.pca(C, D)["lam"]
    free.close()
    # what cov_init takes is found as the least accepted budget, in steps of 1 MB
    for mb in range(1, 4096):
        try:
            h = Handle(wl, hbm_budget=mb << 20)
            break
        except N.CovError as e:
            assert e.code == N.COV_ERR_NOMEM
    h.close()
    work, pca = (M + 8) * (M + 1) * 8, M * (M + 9) * 8 + 8 * M + 64
    h = Handle(wl, hbm_budget=(mb << 20) + work + pca + (1 << 20))
    assert np.array_equal(h.snr(C, D, N.COV_WHICH_JOINT), ref, equal_nan=True)
    np.testing.assert_array_equal(h.pca(C, D)["lam"], lam)
    assert np.array_equal(h.snr(C, D, N.COV_WHICH_JOINT), ref, equal_nan=True)
    h.close()
