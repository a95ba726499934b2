"""Steps in a row on one stream with nothing between them: every kernel of a
step is a dependent launch, the first one included, so a step's clearing has
to wait for the interaction (and the copy) of the step before it."""
import pytest

from paper_2406_16091_gb300 import binding as B
from paper_2406_16091_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("binning", [B.PI_BIN_PER_PARTICLE, B.PI_BIN_BUCKETED, B.PI_BIN_RADIX])
@pytest.mark.parametrize("n", [700, 32768, 200001])
def test_steps_in_a_row_match_steps_alone(n, binning):
    torch = pytest.importorskip("torch")
    dev = torch.device("cuda", 0)
    w = W.scaled(W.SMALL, n)
    s = torch.cuda.current_stream()
    ins = [[torch.from_numpy(a).to(dev) for a in W.uniform(n, 50 + k)] for k in range(3)]

    def buffers():
        return [torch.zeros(n, device=dev) for _ in range(4)] + [torch.zeros(n, dtype=torch.int32, device=dev)
                                                                 for _ in range(2)]

    def step(ctx, pos, out):
        B.pi_bin(ctx, *pos, n, s)
        B.pi_interact(ctx, w.h, *out[:5], B.PI_ORDER_SORTED, s)
        B.pi_copy_binned(ctx, perm=out[5], stream=s)

    ctx = B.pi_create(w.lo, w.hi, w.rc, n)
    try:
        B.pi_set_option(ctx, B.PI_OPT_BINNING, binning)
        alone = []
        for pos in ins:
            out = buffers()
            step(ctx, pos, out)
            B.pi_sync_status(ctx, s)
            alone.append(out)
        rows = [buffers() for _ in range(12)]
        torch.cuda.synchronize()
        for k, out in enumerate(rows):
            step(ctx, ins[k % 3], out)
        B.pi_sync_status(ctx, s)
        for k, out in enumerate(rows):
            for a, b in zip(out, alone[k % 3]):
                assert torch.equal(a.view(torch.int32), b.view(torch.int32))
    finally:
        B.pi_destroy(ctx)
