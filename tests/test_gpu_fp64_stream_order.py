"""The FP64 assembly is stream-ordered: it returns before its kernels have run and can be captured into a graph of the
caller's, whose replays write what a direct call writes.  A wait that expired in its contraction is reported by the next call that
waits for the device: shown here by raising the report word from the host, through a helper built against the library's
private header (no kernel is made to fail)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1812_07437_gb300 import native as N  # noqa: E402
from paper_1812_07437_gb300 import workloads  # noqa: E402


POKE = r"""
#include "common.cuh"
extern "C" int report(cov_handle* h) {  // as k_syrk_sl does when a wait of its assembly has expired
  const int one = 1;
  return (int)cudaMemcpy(h->sl_report, &one, sizeof(int), cudaMemcpyHostToDevice);
}
extern "C" int spoil_table(cov_handle* h) {  // a trispectrum table whose tiles were left incomplete
  return (int)cudaMemset(h->Tmat, 0xFF, sizeof(double) * h->ntrow * h->ntrow);
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
                    lib, "-cudart", "static"], check=True)
    assert os.path.exists(lib)
    return ctypes.CDLL(lib)


def _handle():
    from paper_1812_07437_gb300.handle import Handle
    h = Handle(workloads.get("mid_2bin"))
    h.spectra()
    return h


def _call(h, C, band, terms, stream=None):
    if band:
        h.assemble_band(0, h.M, C, N.COV_LAYOUT_ROWS, terms, N.COV_FP64, stream=stream)
    else:
        h.assemble(C, terms, N.COV_FP64, stream=stream)


@pytest.mark.parametrize("band", [False, True])
@pytest.mark.parametrize("terms", [N.COV_TERMS_ALL, N.COV_TERM_1H, N.COV_TERM_BBPT])
def test_captured_by_the_caller(band, terms):
    h = _handle()
    C = [torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda") for _ in range(2)]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        _call(h, C[0], band, terms)  # what the capture needs is allocated by a direct call
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            _call(h, C[1], band, terms)
    torch.cuda.synchronize()
    assert float(C[1].abs().max()) == 0.0  # captured, not run
    for _ in range(2):
        C[1].zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(C[0], C[1])
    h.close()


def test_returns_before_the_stream_is_done():
    h = _handle()
    C = torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda")
    _call(h, C, False, N.COV_TERMS_ALL)
    torch.cuda.synchronize()
    ref = C.clone()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(200_000_000)  # ~0.1 s of work ahead of the call
        _call(h, C, False, N.COV_TERMS_ALL)
        assert not s.query()
    s.synchronize()
    assert torch.equal(C, ref)
    h.close()


def test_expired_wait_is_reported_by_the_next_synchronising_call(poke):
    h = _handle()
    C = torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda")
    D = torch.zeros(h.M, dtype=torch.float64, device="cuda")
    h.spectra(D)
    _call(h, C, False, N.COV_TERMS_ALL)
    ref = h.snr(C, D)
    for call in (lambda: h.snr(C, D), lambda: h.pca(C, D), lambda: h.batch_snr([h.wl["cosmology"]], precision=N.COV_FP64)):
        assert poke.report(h.h) == 0
        with pytest.raises(N.CovError) as e:
            call()
        assert e.value.code == N.COV_ERR_TIMEOUT and "earlier assembly" in str(e.value)
        assert np.array_equal(h.snr(C, D), ref)  # reported once
    h.close()


def test_a_reported_wait_makes_the_next_band_prepare_its_operands(poke):
    h = _handle()
    C = torch.zeros((h.M, h.M), dtype=torch.float64, device="cuda")
    D = torch.zeros(h.M, dtype=torch.float64, device="cuda")
    h.spectra(D)
    _call(h, C, True, N.COV_TERMS_ALL)
    torch.cuda.synchronize()
    ref = C.clone()
    assert poke.spoil_table(h.h) == 0 and poke.report(h.h) == 0
    _call(h, C, True, N.COV_TERMS_ALL)  # the operands of the first band, the spoilt table among them
    with pytest.raises(N.CovError) as e:
        h.snr(C, D)
    assert e.value.code == N.COV_ERR_TIMEOUT
    assert not torch.equal(C, ref)
    _call(h, C, True, N.COV_TERMS_ALL)
    torch.cuda.synchronize()
    assert torch.equal(C, ref)
    h.close()
