"""The one-launch binning of small systems (k_bin_small: up to 4,096
particles in up to 4,096 cells) against the oracle, at the edges of its
range and just past them, with empty and dense cells, after an error, captured
in a graph, and on a context re-targeted from a larger grid."""
import numpy as np
import pytest

import oracle
from paper_2406_16091_gb300 import binding as B
from paper_2406_16091_gb300 import workloads as W

from gpu_harness import TOL, check_binning, check_interaction, oracle_run, run_gpu

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
    x, y, z = W.uniform(n, 100 + n, lo, hi)
    b, r = oracle_run(x, y, z, lo, hi, rc, rc / 2)
    g = run_gpu(x, y, z, lo, hi, rc, rc / 2, repeat=2)
    check_binning(g, b)
    # FP32 sums of m terms in sequence carry (m + 1) 2^-24 beside the terms' own error: it counts in the grids of few
    # cells, where a target has thousands of neighbours
    most = int(r.nbr.max())
    check_interaction(g, r, tol=TOL if most < 150 else TOL + (most + 1) * 2.0 ** -24)


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


@pytest.mark.parametrize("n", [1, 1531, 4096])
@pytest.mark.parametrize("both", [False, True])
def test_captured_step_with_its_copies(n, both):
    """Binning, interaction and the copy of the binning results in one graph,
    replayed on changed positions.  both: two arrays into one destination,
    which takes memory copies instead of the copying launch."""
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    lo, hi, rc = GRIDS["3375_cells"]
    ins = [[torch.from_numpy(a).to(dev) for a in W.uniform(n, 60 + k, lo, hi)] for k in range(3)]
    pos = [t.clone() for t in ins[0]]
    out = [torch.zeros(n, device=dev) for _ in range(4)] + [torch.zeros(n, dtype=torch.int32, device=dev)
                                                            for _ in range(2)]
    ctx = B.pi_create(lo, hi, rc, n)

    def step(s):
        B.pi_bin(ctx, *pos, n, s)
        B.pi_interact(ctx, rc / 2, *out[:5], B.PI_ORDER_SORTED, s)
        B.pi_copy_binned(ctx, perm=out[5], sz=out[5] if both else None, stream=s)

    try:
        alone = []
        for t in ins:
            for p, q in zip(pos, t):
                p.copy_(q)
            step(torch.cuda.current_stream())
            B.pi_sync_status(ctx, torch.cuda.current_stream())
            alone.append([o.clone() for o in out])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step(torch.cuda.current_stream())
        for k in (1, 2, 0, 2):
            for o in out:
                o.zero_()
            for p, q in zip(pos, ins[k]):
                p.copy_(q)
            graph.replay()
            B.pi_sync_status(ctx, torch.cuda.current_stream())
            for a, b in zip(out, alone[k]):
                assert torch.equal(a.view(torch.int32), b.view(torch.int32))
        b = oracle.bin_particles(*(t.cpu().numpy() for t in ins[2]), lo, hi, rc)
        assert np.array_equal(out[5].cpu().numpy().view(np.uint32), b.sz.view(np.uint32) if both else b.perm)
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
