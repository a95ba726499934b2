"""pi_copy_binned's one launch for all the arrays: every subset and alignment
of the destinations, sizes that are no multiple of four, and nothing written
beside the requested entries."""
import numpy as np
import pytest

import oracle
from paper_2406_16091_gb300 import binding as B
from paper_2406_16091_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NAMES = ("counts", "offsets", "perm", "sx", "sy", "sz")


@pytest.mark.parametrize("n,cells", [(1, 1), (3, 2), (4099, 8), (70001, 21)])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("names", [NAMES, ("perm",), ("offsets", "sz"), ()])
def test_copies_every_subset_and_alignment(n, cells, shift, names):
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    rc = W.rc_for_cells(cells)
    x, y, z = W.uniform(n, 17)
    b = oracle.bin_particles(x, y, z, (0, 0, 0), (1, 1, 1), rc)
    want = {"counts": b.counts, "offsets": b.offsets, "perm": b.perm, "sx": b.sx, "sy": b.sy, "sz": b.sz}
    s = torch.cuda.current_stream()
    ctx = B.pi_create((0, 0, 0), (1, 1, 1), rc, n)
    try:
        t = [torch.from_numpy(a).to(dev) for a in (x, y, z)]
        B.pi_bin(ctx, *t, n, s)
        bufs = {k: torch.full((len(want[k]) + 8,), -7, dtype=torch.int32, device=dev) for k in names}
        B.pi_copy_binned(ctx, **{k: v[shift:] for k, v in bufs.items()}, stream=s)
        B.pi_sync_status(ctx, s)
        for k, v in bufs.items():
            a = v.cpu().numpy()
            m = len(want[k])
            assert np.array_equal(a[shift:shift + m].view(np.uint32), want[k].view(np.uint32)), k
            assert np.all(a[:shift] == -7) and np.all(a[shift + m:] == -7), k
    finally:
        B.pi_destroy(ctx)


def test_memory_copies_for_host_memory_and_shared_destinations():
    # Destinations that the launch must not write: page-locked host memory,
    # and one buffer named twice (the array copied last stands).
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    n, rc = 4099, W.rc_for_cells(8)
    x, y, z = W.uniform(n, 17)
    b = oracle.bin_particles(x, y, z, (0, 0, 0), (1, 1, 1), rc)
    s = torch.cuda.current_stream()
    ctx = B.pi_create((0, 0, 0), (1, 1, 1), rc, n)
    try:
        t = [torch.from_numpy(a).to(dev) for a in (x, y, z)]
        B.pi_bin(ctx, *t, n, s)
        host = torch.zeros(n, dtype=torch.int32).pin_memory()
        both = torch.zeros(n, dtype=torch.int32, device=dev)
        launched = B.pi_launch_count(ctx)
        B.pi_copy_binned(ctx, perm=host, stream=s)
        B.pi_copy_binned(ctx, perm=both, sz=both, stream=s)
        B.pi_sync_status(ctx, s)
        assert B.pi_launch_count(ctx) == launched
        assert np.array_equal(host.numpy().view(np.uint32), b.perm)
        assert np.array_equal(both.cpu().numpy().view(np.uint32), b.sz.view(np.uint32))
    finally:
        B.pi_destroy(ctx)
