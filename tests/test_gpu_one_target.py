"""Shape 5's form with one target per thread (small systems and the costlier
kernels) against the four-target and the staged shapes, bit for bit, and
against the oracle: sizes on both sides of the lines where it is chosen,
ragged ones, rows of sentinels and single particles, dense cells (exact
window bounds), both precision modes and output orders."""
import numpy as np
import pytest

from paper_2406_16091_gb300 import binding as B
from paper_2406_16091_gb300 import workloads as W

from gpu_harness import check_interaction, oracle_run, run_gpu

pytestmark = pytest.mark.gpu


def _sms():
    torch = pytest.importorskip("torch")
    return torch.cuda.get_device_properties(0).multi_processor_count


def _uniform(n, ppc, seed=31):
    cells = max(1, int(round((n / ppc) ** (1.0 / 3.0))))
    rc = W.rc_for_cells(cells)
    return (*W.uniform(n, seed), (0, 0, 0), (1, 1, 1), rc)


def _dense(n, seed=7):
    rng = np.random.default_rng(seed)
    bg = rng.random((n // 2, 3))
    cl = np.clip(0.5 + 0.01 * rng.standard_normal((n - n // 2, 3)), 0, np.nextafter(np.float32(1), np.float32(0)))
    p = np.concatenate([bg, cl]).astype(np.float32)
    return p[:, 0], p[:, 1], p[:, 2], (0, 0, 0), (1, 1, 1), 1.0 / 16


CASES = {
    "one": lambda: _uniform(1, 1),
    "ragged_4099": lambda: _uniform(4099, 6),
    "long_rows": lambda: (*W.uniform(5001, 6, (0, 0, 0), (3.0, 0.04, 0.04)), (0, 0, 0), (3.0, 0.04, 0.04), 0.01),
    "dense": lambda: _dense(6001),
    "line_256": lambda: _uniform(_sms() * 256, 3),
    "past_256": lambda: _uniform(_sms() * 256 + 1, 5),
    "larger": lambda: _uniform(_sms() * 1024 + 1, 3),
}
FORMS = [(B.PI_KERNEL_GAUSSIAN, B.PI_PREC_FP32, 2), (B.PI_KERNEL_GAUSSIAN, B.PI_PREC_KAHAN, 2),
         (B.PI_KERNEL_GAUSSIAN, B.PI_PREC_FP32, 8), (B.PI_KERNEL_LJ, B.PI_PREC_FP32, 2),
         (B.PI_KERNEL_HIGHFLOP, B.PI_PREC_KAHAN, 2), (B.PI_KERNEL_LOWFLOP, B.PI_PREC_FP32, 2)]


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("kern,prec,hdiv", FORMS)
def test_one_target_form_matches_the_other_shapes(name, kern, prec, hdiv):
    x, y, z, lo, hi, rc = CASES[name]()
    h = rc / hdiv
    runs = [run_gpu(x, y, z, lo, hi, rc, h, tile=t, kernel=kern, precision=prec, order=o, binned=False)
            for t, o in ((5, B.PI_ORDER_SORTED), (6, B.PI_ORDER_SORTED), (2, B.PI_ORDER_SORTED),
                         (5, B.PI_ORDER_ORIGINAL), (6, B.PI_ORDER_ORIGINAL))]
    for g in runs:
        assert g["status"] == B.PI_OK
    for got, ref in ((0, 1), (2, 1), (3, 4)):
        for k in ("S", "Vx", "Vy", "Vz", "nbr"):
            assert np.array_equal(runs[got][k].view(np.uint32), runs[ref][k].view(np.uint32)), (got, k)
    if name in ("one", "ragged_4099", "long_rows"):
        _, r = oracle_run(x, y, z, lo, hi, rc, h, kern)
        check_interaction(runs[0], r, rc=rc)


@pytest.mark.parametrize("past", [0, 1])
@pytest.mark.parametrize("prec", [B.PI_PREC_FP32, B.PI_PREC_KAHAN])
def test_compensated_exponent_on_both_sides_of_its_line(past, prec):
    # 9 to 16 per cell: one target per thread up to 6,500 particles per SM, and with compensated sums
    x, y, z, lo, hi, rc = _uniform(_sms() * 6500 + past, 12)
    runs = [run_gpu(x, y, z, lo, hi, rc, rc / 8, tile=t, precision=prec, binned=False) for t in (5, 6)]
    for g in runs:
        assert g["status"] == B.PI_OK
    for k in ("S", "Vx", "Vy", "Vz", "nbr"):
        assert np.array_equal(runs[0][k].view(np.uint32), runs[1][k].view(np.uint32)), k
