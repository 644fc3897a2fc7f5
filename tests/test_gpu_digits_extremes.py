"""The digit contraction (csrc/syrk_sl.cu) on rows that no cosmology gives: every digit at its largest magnitude and of
either sign, K blocks at the limit of their norm, block exponents far apart; bit for bit against the same integers in
Python.  A helper built against the library's private header puts the digits in place of a handle's factor rows and runs
the contraction on them."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402

POKE = r"""
#include "common.cuh"
extern "C" int put(cov_handle* h, const void* rows, size_t bytes, const int* rexp) {
  int e = (int)cudaMemcpy(h->Asl, rows, bytes, cudaMemcpyHostToDevice);
  return e ? e : (int)cudaMemcpy(h->Aexp, rexp, sizeof(int) * h->M, cudaMemcpyHostToDevice);
}
extern "C" int contract(cov_handle* h, double* C) {
  const int rc = wl_tc_status_reset(h, 0);
  return rc ? rc : wl_sl_syrk(h, false, 0, out_rows(C, h->M), h->M, 0);
}
"""


@pytest.fixture(scope="module")
def poke(tmp_path_factory):
    from paper_1812_07437_gb300 import build
    d = tmp_path_factory.mktemp("poke")
    src, lib = str(d / "poke.cu"), str(d / "poke.so")
    with open(src, "w") as f:
        f.write(POKE)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, src, "-o",
                    lib, build.LIB, "-Xlinker", "-rpath=" + build.OUT, "-cudart", "static"], check=True)
    return ctypes.CDLL(lib)


def _rows(rng, M, nk):
    """Integers X [nk][128][32] in units of 2^-55 (row norm of a block below sqrt(2)), distances d [nk][128]."""
    low = sum(1 << (8 * t) for t in range(6))  # one in each of the six lower digits
    X = np.zeros((nk, 128, 32), dtype=object)
    d = np.full((nk, 128), 112)
    for r in range(M):
        d[:, r] = rng.integers(0, 40, nk)
        d[rng.random(nk) < 0.1, r] = 112  # empty blocks
        d[rng.integers(0, nk), r] = 0
        for b in range(nk):
            if d[b, r] == 112:
                continue
            kind = rng.integers(0, 4)
            sgn = [1 if s else -1 for s in rng.integers(0, 2, 32)]
            if kind == 0:  # one entry close to sqrt(2), the others with digits of +-127, 128 from the second on
                x = [s * (127 if s > 0 else 128) * (low >> 8) * 256 // 256 for s in sgn]
                x[int(rng.integers(0, 32))] = 180 * (1 << 48) + 127 * low
            elif kind == 1:  # 32 entries of a quarter, all lower digits -128
                x = [s * (31 << 48) - 128 * low for s in sgn]
            elif kind == 2:  # all lower digits 127
                x = [s * (31 << 48) + 127 * low for s in sgn]
            else:
                x = [int(v) for v in rng.integers(-(1 << 52), 1 << 52, 32)]
            assert sum(v * v for v in x) < 2 << 110
            X[b, r] = x
    assert all(d[:, r].min() == 0 for r in range(M))
    return X, d


def _digits(X):
    y = X + sum(0x80 << (8 * t) for t in range(7))
    out = [y >> 48]
    out += [(y >> (8 * (6 - t))) & 255 for t in range(1, 7)]
    return [(o - 128).astype(np.int64) for o in out]  # [digit][nk][row][k]


def _expected(dig, d, rexp, M, gb, levels):
    nk = d.shape[0]
    ng = (nk + gb - 1) // gb
    gd = np.stack([d[g * gb:(g + 1) * gb].min(0) for g in range(ng)])
    B = np.zeros((M, M), dtype=np.float32)
    for s0 in range(0, ng, 8):
        s1 = min(ng, s0 + 8)
        least = (gd[s0:s1, :M, None] + gd[s0:s1, None, :M]).min(0)
        cnt = min(nk, s1 * gb) - s0 * gb
        B = (B.astype(np.float64) + cnt * 2.0 ** (100 - least)).astype(np.float32)
    H = 246 - ((B * np.float32(1.0 + 2.0**-10)).view(np.int32) >> 23)
    T = np.zeros((M, M), dtype=object)
    for b in range(nk):
        S = np.zeros((M, M), dtype=object)
        for g in range(levels):
            L = sum(dig[t][b][:M] @ dig[g - t][b][:M].T for t in range(max(0, g - 6), min(g, 6) + 1))
            assert np.abs(L).max() < 1 << 22
            S = S + (L.astype(object) << (48 - 8 * g) if g < 7 else (L.astype(object) + 128) >> 8)
        s = (d[b, :M, None] + d[b, None, :M] + 20 - H).astype(object)
        t = S >> s
        T = T + t + (t & 1)
    assert np.abs(T).max() < 1 << 63
    e = rexp[:, None] + rexp[None, :] - H - 42
    return np.ldexp(T.astype(np.float64), e), H


# N_chi, N_M, levels: below and above the entries from which seven levels serve; K blocks in groups of one and of four
@pytest.mark.parametrize("nchi,nm,levels,gb", [(16, 64, 8, 1), (130, 32, 7, 4), (2, 2, 8, 1)])
def test_extreme_digits(poke, nchi, nm, levels, gb):
    from paper_1812_07437_gb300.handle import Handle
    wl = workloads.get("tiny_2bin")
    wl["nz"].update(n_tomo=2, photoz_sigma0=0.05)
    wl["bins"].update(n_ell=4, ell_min=100.0, ell_max=800.0, n_chi=nchi, n_mass=nm)
    h = Handle(wl)
    M = h.M
    assert 30 < M <= 128
    C = torch.zeros((M, M), dtype=torch.float64, device="cuda")
    h.spectra()
    h.assemble(C, N.COV_TERM_1H, N.COV_FP64)  # (the buffers)
    nk = nchi * (32 if nm < 16 else nm) // 32
    rng = np.random.default_rng(nk)
    X, d = _rows(rng, M, nk)
    dig = _digits(X)
    rexp = rng.integers(-300, 300, M).astype(np.int32)
    want, H = _expected(dig, d, rexp, M, gb, levels)
    assert H.min() >= 0
    bits = np.stack([(x.astype(np.float32).view(np.uint32) >> 16).astype(np.uint16) for x in dig], axis=1)  # BF16
    ng = (nk + gb - 1) // gb
    gd = np.stack([d[g * gb:(g + 1) * gb].min(0) for g in range(ng)]).astype(np.uint16)
    buf = b"".join([bits.tobytes(), gd.tobytes(), np.zeros((nk, 128), np.int16).tobytes(), d.astype(np.uint8).tobytes(),
                    d.min(1).astype(np.uint8).tobytes()])
    assert poke.put(h.h, buf, ctypes.c_size_t(len(buf)), rexp.ctypes.data_as(ctypes.c_void_p)) == 0
    C.fill_(0.0)
    torch.cuda.synchronize()
    assert poke.contract(h.h, ctypes.c_void_p(C.data_ptr())) == 0
    torch.cuda.synchronize()
    i, j = np.tril_indices(M)
    assert np.array_equal(C.cpu().numpy()[i, j], want[i, j])
    h.close()
