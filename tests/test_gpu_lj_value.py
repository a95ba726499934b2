"""The Lennard-Jones value of single pairs (approximate reciprocal and one
Newton step) against FP64, within the rounding of its FP32 steps: with s =
1/u, u = r^2/sigma^2 + 1/100, u carries the roundings of 1/sigma^2, r^2
(three) and its own sum, s one more and s^3 two products, at most (3 * 6 + 2)
half-ulps in s^3; K = s^3 (4 s^3 - 4) then differs by at most that share of
4 s^3 (|s^3 - 1| + s^3) plus two roundings of its own."""
import numpy as np
import pytest

from paper_2406_16091_gb300 import binding as B

from gpu_harness import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e6, 1e-12])
@pytest.mark.parametrize("hdiv", [1.5, 2.0, 10.0, 300.0])
@pytest.mark.parametrize("tile", [5, 6, 2])
def test_single_pairs(scale, hdiv, tile):
    # pairs on a lattice of 4 cutoffs, at distances from a fraction of sigma
    # up to the cutoff
    side, rc = 12, np.float32(scale)
    m = side ** 3
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(m, 3).astype(np.float64)
    base = ((g * 4.0 + 2.0) * scale).astype(np.float32)
    rng = np.random.default_rng(3)
    v = rng.standard_normal((m, 3))
    r = np.exp(np.linspace(np.log(1e-3), np.log(0.99), m))
    other = (base + (v / np.linalg.norm(v, axis=1, keepdims=True) * r[:, None] * scale)).astype(np.float32)
    p = np.concatenate([base, other])
    hi = float(np.float32(4.0 * side * scale))
    h = np.float32(rc / np.float32(hdiv))
    out = run_gpu(*(np.ascontiguousarray(p[:, d]) for d in range(3)), (0, 0, 0), (hi, hi, hi), float(rc), float(h),
                  kernel=B.PI_KERNEL_LJ, tile=tile, order=B.PI_ORDER_ORIGINAL, binned=False)
    assert out["status"] == B.PI_OK
    d = (other - base).astype(np.float64)  # FP32 differences, as the kernel takes them
    r2 = (d * d).sum(1)
    near = out["nbr"][:m] == 1
    assert near.sum() > 0.9 * m
    s3 = (1.0 / (r2 / float(h) ** 2 + 0.01)) ** 3
    K = 4.0 * s3 * (s3 - 1.0)
    bound = 2.0 ** -24 * 4.0 * s3 * (20.0 * (np.abs(s3 - 1.0) + s3) + 2.0 * np.abs(s3 - 1.0)) + 2.0 ** -126
    err = np.abs(out["S"][:m].astype(np.float64) - K)
    assert np.all(err[near] <= bound[near]), float((err / bound)[near].max())


# sigma^2 = h^2 beyond the range whose reciprocal is a normal FP32 number
# (h^2 below about 2.9e-39 or above 8.5e37): the pairs lie along x at multiples
# of h (of a cutoff's quarter, for the long h), a third particle farther off
# inside the cutoff.
STEPS = np.array([0.0, 0.08, 0.3, 0.8, 1.0, 1.13, 1.2, 1.7, 2.0, 3.1])


def edge_sites(h, rc):
    """Sites 4 cutoffs apart: particles at x = 0, a step and 0.95 rc."""
    m = len(STEPS)
    y, z = ((np.arange(m) % 4) * 4.0 + 2.0) * rc, ((np.arange(m) // 4) * 4.0 + 2.0) * rc
    x = np.stack([np.zeros(m), STEPS * min(h, 0.25 * rc), np.full(m, 0.95 * rc)]).astype(np.float32)
    return x.ravel(), np.tile(y, 3).astype(np.float32), np.tile(z, 3).astype(np.float32), (16.0 * rc,) * 3


def edge_expected(x, h):
    """S and Vx of each site's first particle with their bounds: as above, r^2
    (one product) and its scale rounded once each, r^2 to 2^-150 at the least;
    two roundings each for the sums and the products of V."""
    m, sigma2, e = len(STEPS), float(np.float32(h)) ** 2, 2.0 ** -24
    S, V, bS, bV = (np.zeros(m) for _ in range(4))
    for d in (x[m:2 * m].astype(np.float64), x[2 * m:].astype(np.float64)):
        u = d * d / sigma2 + 0.01
        rho = 3.0 * (5.0 * e + 2.0 ** -150 / sigma2 / u) + 2.0 * e
        s3 = u ** -3.0
        K = 4.0 * s3 * (s3 - 1.0)
        b = 4.0 * s3 * (rho * (np.abs(s3 - 1.0) + s3) + 4.0 * e * np.abs(s3 - 1.0)) + 2.0 ** -126
        S, V, bS, bV = S + K, V + d * K, bS + b, bV + d * (b + 2.0 * e * np.abs(K)) + 2.0 ** -126
    return S, V, bS, bV


TINY = [5.6e-20, 5.4e-20, 5e-20, 3e-20, 1e-20, 1e-21]


def check_edge(out, x, h, first=0):
    S, V, bS, bV = edge_expected(x, h)
    k = slice(first, first + len(STEPS))
    for got, want, bound in ((out["S"][k], S, bS), (out["Vx"][k], V, bV)):
        err = np.abs(got.astype(np.float64) - want)
        assert np.all(err <= bound), float((err / bound).max())
    assert np.all(out["nbr"][k] == 2)


@pytest.mark.parametrize("h,rc", [(h, 1.0) for h in TINY] + [(9e18, 3e17), (1.1e19, 3e17), (1.8e19, 3e17)])
@pytest.mark.parametrize("form", [dict(tile=5), dict(tile=6), dict(tile=2), dict(algo=B.PI_ALGO_PPNL),
                                  dict(tile=5, precision=B.PI_PREC_KAHAN), dict(tile=5, kernel=B.PI_KERNEL_HIGHFLOP)])
def test_scales_at_the_ends_of_fp32(h, rc, form):
    x, y, z, hi = edge_sites(h, rc)
    out = run_gpu(x, y, z, (0, 0, 0), hi, rc, h, order=B.PI_ORDER_ORIGINAL, binned=False,
                  **{"kernel": B.PI_KERNEL_LJ, **form})
    assert out["status"] == B.PI_OK
    check_edge(out, x, h)


@pytest.mark.parametrize("tiles", [None, 5, 6])
def test_scales_at_the_ends_of_fp32_in_one_batch(tiles):
    # an ordinary system between the extremes; a plan runs the two- and four-target forms
    torch = pytest.importorskip("torch")
    hs, rcs = [3e-20, 0.25, 1.5e19, 5e-20], [1.0, 1.0, 3e17, 1.0]
    sites = [edge_sites(h, rc) for h, rc in zip(hs, rcs)]
    s, n = torch.cuda.current_stream(), len(sites[0][0])
    ctx = B.pi_batch_create([((0, 0, 0), q[3]) for q in sites], rcs, [n] * 4)
    try:
        B.pi_set_option(ctx, B.PI_OPT_KERNEL, B.PI_KERNEL_LJ)
        if tiles:
            B.pi_batch_set_tiles(ctx, [tiles] * 4)
        pos = [torch.from_numpy(np.concatenate([q[d] for q in sites])).cuda() for d in range(3)]
        out = [torch.full((4 * n,), float("nan"), device="cuda") for _ in range(4)]
        nbr = torch.empty(4 * n, dtype=torch.int32, device="cuda")
        B.pi_batch_bin(ctx, *pos, [n] * 4, s)
        B.pi_batch_interact(ctx, hs, *out, nbr, B.PI_ORDER_ORIGINAL, s)
        B.pi_sync_status(ctx, s)
        got = {"S": out[0].cpu().numpy(), "Vx": out[1].cpu().numpy(), "nbr": nbr.cpu().numpy()}
        for k, h in enumerate(hs):
            check_edge(got, sites[k][0], h, k * n)
    finally:
        B.pi_destroy(ctx)


def test_length_whose_square_leaves_fp32_is_rejected():
    x, y, z, hi = edge_sites(1.0, 1.0)
    for h in (1e-23, 2e19):
        with pytest.raises(B.PiError) as e:
            run_gpu(x, y, z, (0, 0, 0), hi, 1.0, h, kernel=B.PI_KERNEL_LJ)
        assert e.value.status == B.PI_ERR_INVALID_ARG
