"""The one-launch binning of small systems (k_bin_small: up to 4,096
particles in up to 4,096 cells) against the oracle, at the edges of its
range and just past them, with empty and dense cells, after an error, and on
a context re-targeted from a larger grid."""
import numpy as np
import pytest

import oracle
from paper_2406_16091_gb300 import binding as B
from paper_2406_16091_gb300 import workloads as W

from gpu_harness import check_binning, check_interaction, oracle_run, run_gpu

pytestmark = pytest.mark.gpu

UNIT = ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0))


def _cube(cells):
    return (*UNIT, W.rc_for_cells(cells))


GRIDS = {
    "27_cells": _cube(3),
    "one_cell": (*UNIT, 1.5),
    "4096_cells": _cube(16),
    "3375_cells": _cube(15),
    "4913_cells": _cube(17),  # past the range: the five-kernel path
    "4096_long": ((0.0, 0.0, 0.0), (4.0, 1.0, 1.0), 0.1),
    "slab": ((-2.0, 0.5, 10.0), (2.0, 3.5, 11.0), 0.11),
}


@pytest.mark.parametrize("n", [1, 2, 31, 513, 1025, 4095, 4096, 4097])
@pytest.mark.parametrize("grid", list(GRIDS))
def test_small_binning_matches_the_oracle(grid, n):
    lo, hi, rc = GRIDS[grid]
    if grid in ("one_cell", "27_cells"):
        n = min(n, 4097)  # thousands of mutual neighbours
    x, y, z = W.uniform(n, 100 + n, lo, hi)
    b, r = oracle_run(x, y, z, lo, hi, rc, rc / 2)
    g = run_gpu(x, y, z, lo, hi, rc, rc / 2, repeat=2)
    check_binning(g, b)
    if n <= 4097 and grid not in ("one_cell", "27_cells"):
        check_interaction(g, r)
    else:
        assert np.array_equal(g["nbr"], r.nbr)


def test_small_binning_reports_out_of_box_and_recovers():
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    lo, hi, rc = GRIDS["4096_cells"]
    x, y, z = W.uniform(4000, 4, lo, hi)
    t = [torch.from_numpy(a).to(dev) for a in (x, y, z)]
    bad = t[0].clone()
    bad[3210] = float("nan")
    s = torch.cuda.current_stream()
    ctx = B.pi_create(lo, hi, rc, 4000)
    try:
        B.pi_bin(ctx, bad, t[1], t[2], 4000, s)
        assert B.pi_sync_status(ctx, s, raise_on_error=False)[0] == B.PI_ERR_OUT_OF_BOX
        B.pi_bin(ctx, *t, 4000, s)
        perm = torch.empty(4000, dtype=torch.int32, device=dev)
        B.pi_copy_binned(ctx, perm=perm, stream=s)
        st, mpc = B.pi_sync_status(ctx, s)
        b = oracle.bin_particles(x, y, z, lo, hi, rc)
        assert mpc == b.max_per_cell and np.array_equal(perm.cpu().numpy().view(np.uint32), b.perm)
    finally:
        B.pi_destroy(ctx)


def test_small_binning_between_larger_steps_of_one_context():
    """A context of a larger grid takes a large step, a small one after a
    re-target, and a large one again: each as if alone."""
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    s = torch.cuda.current_stream()
    ctx = B.pi_create(*_cube(40), 60000)
    try:
        for n, cells in ((60000, 40), (3001, 11), (4097, 20), (700, 40), (60000, 40)):
            lo, hi, rc = _cube(cells)
            x, y, z = W.uniform(n, n + cells)
            t = [torch.from_numpy(a).to(dev) for a in (x, y, z)]
            B.pi_reconfigure(ctx, lo, hi, rc, s)
            B.pi_bin(ctx, *t, n, s)
            out = [torch.empty(n, device=dev) for _ in range(4)]
            nb = torch.empty(n, dtype=torch.int32, device=dev)
            B.pi_interact(ctx, rc / 2, *out, nb, B.PI_ORDER_ORIGINAL, s)
            perm = torch.empty(n, dtype=torch.int32, device=dev)
            offs = torch.empty(cells ** 3 + 1, dtype=torch.int32, device=dev)
            B.pi_copy_binned(ctx, offsets=offs, perm=perm, stream=s)
            B.pi_sync_status(ctx, s)
            b, r = oracle_run(x, y, z, lo, hi, rc, rc / 2)
            assert np.array_equal(offs.cpu().numpy().view(np.uint32), b.offsets)
            assert np.array_equal(perm.cpu().numpy().view(np.uint32), b.perm)
            assert np.array_equal(nb.cpu().numpy().view(np.uint32)[b.perm], r.nbr)
    finally:
        B.pi_destroy(ctx)
