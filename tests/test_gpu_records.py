"""Input-order outputs of large systems, written as records and copied to the
arrays by a second kernel: bitwise the sorted-order outputs in input order, at
the rule's edges, for both direct shapes, in dense cells, without neighbour
counts, at odd alignments, and nothing written beside the arrays.  Calls that may overlap
(another stream, an interaction captured alone) write straight to the arrays;
the launch counts tell the two ways apart."""
import numpy as np
import pytest

from paper_2406_16091_gb300 import binding as B
from paper_2406_16091_gb300 import workloads as W

pytestmark = pytest.mark.gpu

EDGE = 1000000  # from this many particles on
BOX = ((0, 0, 0), (1, 1, 1))


def setup(torch, n, cells, kernel=B.PI_KERNEL_GAUSSIAN, tile=-1):
    rc = W.rc_for_cells(cells)
    ctx = B.pi_create(*BOX, rc, n)
    B.pi_set_option(ctx, B.PI_OPT_KERNEL, kernel)
    B.pi_set_option(ctx, B.PI_OPT_TILE, tile)
    return ctx, rc / 2, [torch.from_numpy(a).cuda() for a in W.uniform(n, 5)]


def outputs(torch, n, shift=0):
    whole = [torch.full((n + 8,), -7.0, device="cuda") for _ in range(4)]
    whole.append(torch.full((n + 8,), -7, dtype=torch.int32, device="cuda"))
    return whole, [w[shift:shift + n] for w in whole]


def in_order(torch, ctx, h, n, s):
    """The sorted-order outputs, in input order."""
    _, out = outputs(torch, n)
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    B.pi_interact(ctx, h, *out, B.PI_ORDER_SORTED, s)
    B.pi_copy_binned(ctx, perm=perm, stream=s)
    want = [torch.empty_like(o) for o in out]
    for w, o in zip(want, out):
        w[perm.long()] = o
    return want


def clustered(n, cells):
    """Uniform but for a tight cluster of 6,000 at each of two places: cells of
    more than 255, whose targets take exact window bounds."""
    x = np.stack(W.uniform(n, 5), 1)
    rng = np.random.default_rng(9)
    for k, c in enumerate(((0.31, 0.42, 0.77), (0.8, 0.1, 0.25))):
        x[k * 6000:(k + 1) * 6000] = np.asarray(c) + 0.6 / cells * rng.standard_normal((6000, 3))
    x = np.clip(x, 0, np.nextafter(np.float32(1), np.float32(0))).astype(np.float32)
    x = x[rng.permutation(n)]
    return [np.ascontiguousarray(x[:, d]) for d in range(3)]


def same(torch, a, b):
    return all(torch.equal(x.view(torch.int32), y.view(torch.int32)) for x, y in zip(a, b))


@pytest.mark.parametrize("n,cells,records", [(EDGE - 1, 100, False), (EDGE, 100, True), (EDGE + 513, 70, True),
                                             (EDGE + 1, 60, False), (1500001, 60, True), (2097152, 64, False),
                                             (6000001, 90, True)])
@pytest.mark.parametrize("kernel", [B.PI_KERNEL_GAUSSIAN, B.PI_KERNEL_LOWFLOP, B.PI_KERNEL_LJ])
@pytest.mark.parametrize("tile,shift,counts", [(-1, 0, True), (5, 1, True), (6, 3, False)])
def test_records_equal_sorted_outputs(n, cells, records, kernel, tile, shift, counts):
    torch = pytest.importorskip("torch")
    s = torch.cuda.current_stream()
    ctx, h, pos = setup(torch, n, cells, kernel, tile)
    try:
        B.pi_bin(ctx, *pos, n, s)
        want = in_order(torch, ctx, h, n, s)
        whole, out = outputs(torch, n, shift)
        args = out if counts else out[:4] + [None]
        before = B.pi_launch_count(ctx)
        B.pi_interact(ctx, h, *args, B.PI_ORDER_ORIGINAL, s)
        assert B.pi_launch_count(ctx) - before == (2 if records else 1)
        B.pi_sync_status(ctx, s)
        used = 5 if counts else 4
        assert same(torch, out[:used], want[:used])
        for w in whole[:used]:
            assert bool((w[:shift] == -7).all()) and bool((w[shift + n:] == -7).all())
        assert counts or bool((whole[4] == -7).all())
    finally:
        B.pi_destroy(ctx)


@pytest.mark.parametrize("kernel", [B.PI_KERNEL_GAUSSIAN, B.PI_KERNEL_LOWFLOP, B.PI_KERNEL_LJ])
@pytest.mark.parametrize("tile", [5, 6])
def test_records_of_dense_cells(kernel, tile):
    torch = pytest.importorskip("torch")
    n, cells, s = EDGE + 17, 80, torch.cuda.current_stream()
    ctx, h, _ = setup(torch, n, cells, kernel, tile)
    try:
        pos = [torch.from_numpy(a).cuda() for a in clustered(n, cells)]
        B.pi_bin(ctx, *pos, n, s)
        want = in_order(torch, ctx, h, n, s)
        _, out = outputs(torch, n)
        before = B.pi_launch_count(ctx)
        B.pi_interact(ctx, h, *out, B.PI_ORDER_ORIGINAL, s)
        assert B.pi_launch_count(ctx) - before == 2
        assert B.pi_sync_status(ctx, s)[1] > 255
        assert same(torch, out, want)
    finally:
        B.pi_destroy(ctx)


def test_other_streams_and_lone_captures_write_straight():
    torch = pytest.importorskip("torch")
    n = EDGE + 3
    s, other = torch.cuda.current_stream(), torch.cuda.Stream()
    ctx, h, pos = setup(torch, n, 100)
    try:
        B.pi_bin(ctx, *pos, n, s)
        want = in_order(torch, ctx, h, n, s)
        torch.cuda.synchronize()
        # two interactions that may overlap, then one captured alone
        outs = [outputs(torch, n)[1] for _ in range(4)]
        before = B.pi_launch_count(ctx)
        B.pi_interact(ctx, h, *outs[0], B.PI_ORDER_ORIGINAL, s)
        B.pi_interact(ctx, h, *outs[1], B.PI_ORDER_ORIGINAL, other)
        assert B.pi_launch_count(ctx) - before == 3
        torch.cuda.synchronize()
        lone = torch.cuda.CUDAGraph()
        before = B.pi_launch_count(ctx)
        with torch.cuda.graph(lone):
            B.pi_interact(ctx, h, *outs[2], B.PI_ORDER_ORIGINAL, torch.cuda.current_stream())
        assert B.pi_launch_count(ctx) - before == 1
        lone.replay()
        torch.cuda.synchronize()
        # binning and interaction in one capture
        step = torch.cuda.CUDAGraph()
        with torch.cuda.graph(step):
            c = torch.cuda.current_stream()
            B.pi_bin(ctx, *pos, n, c)
            before = B.pi_launch_count(ctx)
            B.pi_interact(ctx, h, *outs[3], B.PI_ORDER_ORIGINAL, c)
            assert B.pi_launch_count(ctx) - before == 2
        for _ in range(2):
            step.replay()
        torch.cuda.synchronize()
        B.pi_sync_status(ctx, s)
        for out in outs:
            assert same(torch, out, want)
    finally:
        B.pi_destroy(ctx)


def test_outputs_stay_after_an_error():
    torch = pytest.importorskip("torch")
    n = EDGE + 3
    s = torch.cuda.current_stream()
    ctx, h, pos = setup(torch, n, 100)
    try:
        pos[0][n // 2] = 2.0  # outside the box
        B.pi_bin(ctx, *pos, n, s)
        whole, out = outputs(torch, n)
        B.pi_interact(ctx, h, *out, B.PI_ORDER_ORIGINAL, s)
        with pytest.raises(B.PiError):
            B.pi_sync_status(ctx, s)
        assert all(bool((w == -7).all()) for w in whole)
    finally:
        B.pi_destroy(ctx)


def test_batch_with_a_plan_of_both_shapes():
    torch = pytest.importorskip("torch")
    s = torch.cuda.current_stream()
    ns, cells = [700001, 3, 0, 800000], [90, 2, 1, 60]
    rcs = [W.rc_for_cells(c) for c in cells]
    ctx = B.pi_batch_create([BOX] * 4, rcs, [max(k, 1) for k in ns])
    try:
        p = [W.uniform(k, 7 + i) for i, k in enumerate(ns)]
        pos = [torch.from_numpy(np.concatenate([q[d] for q in p])).cuda() for d in range(3)]
        h, n = [r / 2 for r in rcs], sum(ns)
        B.pi_batch_bin(ctx, *pos, ns, s)
        results = []
        for plan in (None, [5, 6, 5, 6]):
            B.pi_batch_set_tiles(ctx, plan)
            for order in (B.PI_ORDER_SORTED, B.PI_ORDER_ORIGINAL):
                _, out = outputs(torch, n)
                B.pi_batch_interact(ctx, h, *out, order, s)
                if order == B.PI_ORDER_SORTED:
                    perm = torch.empty(n, dtype=torch.int32, device="cuda")
                    B.pi_copy_binned(ctx, perm=perm, stream=s)
                    got = [torch.empty_like(o) for o in out]
                    for g, o in zip(got, out):
                        g[perm.long()] = o
                    out = got
                results.append(out)
        B.pi_sync_status(ctx, s)
        for r in results[1:]:
            assert same(torch, r, results[0])
    finally:
        B.pi_destroy(ctx)


def test_autotuned_plans_are_timed_on_the_way_they_run():
    # a batch over three occupancy regimes whose plan writes records: so do the
    # trials of the regimes, each interaction one launch more than sorted
    torch = pytest.importorskip("torch")
    s = torch.cuda.current_stream()
    ns, rcs, reps = [600001, 600000, 300000], [W.rc_for_cells(c) for c in (100, 50, 30)], 3
    ctx = B.pi_batch_create([BOX] * 3, rcs, ns)
    try:
        p = [W.uniform(k, 7 + i) for i, k in enumerate(ns)]
        pos = [torch.from_numpy(np.concatenate([q[d] for q in p])).cuda() for d in range(3)]
        h, n, launches = [r / 2 for r in rcs], sum(ns), []
        _, out = outputs(torch, n)
        for order in (B.PI_ORDER_SORTED, B.PI_ORDER_ORIGINAL):
            B.pi_batch_set_tiles(ctx, None)
            B.pi_batch_bin(ctx, *pos, ns, s)
            before = B.pi_launch_count(ctx)
            B.pi_autotune(ctx, h, *out, order, reps, s)
            launches.append(B.pi_launch_count(ctx) - before)
        # shapes 5 and 6, three regimes and the resulting plan write records; that plan may take one launch (and one
        # that writes its ranges) fewer in this order than in the other
        assert launches[1] - launches[0] >= (reps + 1) * (6 - 1) - 2
    finally:
        B.pi_destroy(ctx)


@pytest.mark.parametrize("n,cells,launched", [(5000001, 84, 1), (5499999, 87, 1), (5500000, 87, 2), (5500000, 83, 1)])
@pytest.mark.parametrize("kernel", [B.PI_KERNEL_GAUSSIAN, B.PI_KERNEL_LJ])
def test_line_from_eight_per_cell(n, cells, launched, kernel):
    torch = pytest.importorskip("torch")
    s = torch.cuda.current_stream()
    ctx, h, pos = setup(torch, n, cells, kernel)
    try:
        B.pi_bin(ctx, *pos, n, s)
        want = in_order(torch, ctx, h, n, s)
        _, out = outputs(torch, n)
        before = B.pi_launch_count(ctx)
        B.pi_interact(ctx, h, *out, B.PI_ORDER_ORIGINAL, s)
        assert B.pi_launch_count(ctx) - before == launched
        B.pi_sync_status(ctx, s)
        assert same(torch, out, want)
    finally:
        B.pi_destroy(ctx)
