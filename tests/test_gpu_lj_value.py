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
