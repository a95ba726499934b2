"""The bounds checks of the one-block binning (k_bin_small): a check that fails
early in the kernel is still reported at its end.  The kernel is compiled alone
as the debug build has it and given one cell less than the particles' grid
(arrays sized for the whole grid): the particles of the last cell fail the
check of the counts, are skipped, and the control block says so."""
import ctypes
import os
import subprocess

import pytest

from paper_2406_16091_gb300 import build as pibuild

pytestmark = pytest.mark.gpu

HARNESS = r"""
#include <cstring>
#include "pi_internal.cuh"
using namespace pi;
// n particles in cells 0, 1, .. , 7, 0, .. of a 2 x 2 x 2 grid of the unit box
extern "C" int run_small(uint32_t n, uint32_t cells, int outside, uint32_t* words)
{
    struct Arrays {
        alignas(256) Ctrl ctrl;
        alignas(256) float p[3][64];
        alignas(256) SysDesc d;
        alignas(256) uint32_t pbase[4];
        alignas(256) uint32_t counts[16];
        alignas(256) uint32_t offsets[16];
        alignas(256) uint2 xbins[16];
        alignas(256) Rec rec[68];
    };
    static Arrays h;
    Arrays* d;
    std::memset(&h, 0xff, sizeof h);
    std::memset(&h.d, 0, sizeof h.d);
    for (int k = 0; k < 3; ++k) {
        h.d.g.lo[k] = 0.f; h.d.g.hi[k] = 1.f; h.d.g.inv_w[k] = 2.f; h.d.g.n[k] = 2;
        for (uint32_t i = 0; i < n; ++i) h.p[k][i] = (i >> k & 1) ? 0.75f : 0.25f;
    }
    if (outside) h.p[0][0] = 2.f;
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemcpy(d, &h, sizeof h, cudaMemcpyDefault) != cudaSuccess) return 1;
    Systems sy{};
    sy.sys = &d->d;
    sy.S = 1;
    cudaError_t e = launch_bin_small(d->p[0], d->p[1], d->p[2], n, sy, cells, d->pbase, d->counts, d->offsets, d->xbins,
                                     d->rec, &d->ctrl, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(&h, d, sizeof h, cudaMemcpyDefault);
    cudaFree(d);
    words[0] = h.ctrl.error; words[1] = h.ctrl.check_site; words[2] = h.ctrl.max_per_cell; words[3] = h.ctrl.ticket;
    words[4] = h.offsets[cells];
    return e == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("small_check")
    (d / "harness.cu").write_text(HARNESS)
    lib = d / "harness.so"
    cmd = [pibuild.nvcc(), *pibuild.NVCC_FLAGS, "-DPI_CHECK", "-shared", "-o", str(lib), str(d / "harness.cu"),
           os.path.join(pibuild.CSRC, "pi_bin.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("n,cells,outside,error,site,most", [
    (64, 8, 0, 0, 0, 8),   # in order
    (61, 8, 1, 1, 0, 9),   # a position outside the box, put into the next cell (ERR_OUT_OF_BOX)
    (64, 7, 0, 8, 1, 8),   # the last cell's particles fail the check (ERR_CHECK at CS_HIST_COUNTS)
    (64, 7, 1, 9, 1, 9),   # both
])
def test_failed_check_is_reported(harness, n, cells, outside, error, site, most):
    words = (ctypes.c_uint32 * 5)()
    assert harness.run_small(n, cells, outside, words) == 0
    assert list(words) == [error, site, most, 0, n]
