"""pi_copy_binned's one launch for all the arrays: every subset and alignment
of the destinations, sizes that are no multiple of four, and nothing written
beside the requested entries."""
import ctypes

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


def runtime():
    """The CUDA runtime library that the process has loaded."""
    with open("/proc/self/maps") as f:
        paths = [line.split()[-1] for line in f if "libcudart" in line]
    return ctypes.CDLL(paths[0] if paths else "libcudart.so")


def neighbours(rt, size):
    """Two device allocations of `size` bytes that follow each other, and all that were made."""
    made = []
    for _ in range(256):
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
        made.append(p.value)
        if made[-1] - size in made:
            return made[-1] - size, made[-1], made
        if made[-1] + size in made:
            return made[-1], made[-1] + size, made
    raise AssertionError("no two allocations in a row")


def test_destination_that_ends_too_early_is_refused():
    # The end of one allocation, followed by memory of this test: an array
    # that just fits is copied, one that does not is refused and nothing written.
    torch = pytest.importorskip("torch")
    n, rc, size = 4099, W.rc_for_cells(8), 65536
    x, y, z = W.uniform(n, 17)
    b = oracle.bin_particles(x, y, z, (0, 0, 0), (1, 1, 1), rc)
    s = torch.cuda.current_stream()
    ctx = B.pi_create((0, 0, 0), (1, 1, 1), rc, n)
    rt = runtime()
    first, second, made = neighbours(rt, size)

    def words(ptr, count):
        a = np.empty(count, np.uint32)
        assert rt.cudaMemcpy(ctypes.c_void_p(a.ctypes.data), ctypes.c_void_p(ptr), ctypes.c_size_t(4 * count), 2) == 0
        return a

    try:
        B.pi_bin(ctx, *(torch.from_numpy(a).cuda() for a in (x, y, z)), n, s)
        for p in (first, second):
            assert rt.cudaMemset(ctypes.c_void_p(p), 0xF9, ctypes.c_size_t(size)) == 0
        torch.cuda.synchronize()
        launched = B.pi_launch_count(ctx)
        with pytest.raises(B.PiError) as e:
            B.pi_copy_binned(ctx, perm=first + size - 4 * n + 4, stream=s)
        assert e.value.status == B.PI_ERR_CUDA and B.pi_launch_count(ctx) == launched
        torch.cuda.synchronize()
        assert np.all(words(first, size // 4) == 0xF9F9F9F9) and np.all(words(second, size // 4) == 0xF9F9F9F9)
        B.pi_copy_binned(ctx, perm=first + size - 4 * n, stream=s)
        assert B.pi_launch_count(ctx) == launched + 1
        torch.cuda.synchronize()
        assert np.array_equal(words(first + size - 4 * n, n), b.perm)
        assert np.all(words(second, size // 4) == 0xF9F9F9F9)
    finally:
        B.pi_destroy(ctx)
        for p in made:
            rt.cudaFree(ctypes.c_void_p(p))
