"""The channel-mean scan with two steps per thread (chunks of 64 or 128 steps, 8 or
16 padded states, even L): ybar and the merged map bit for bit against the one-step kernel
(which the same call runs on tensors one element into an allocation, where pairs
of steps cannot be loaded as one), and against the fp64 oracle.  Sizes: a ragged
last chunk of two steps, one chunk, channels around the 16-channel request
batches and the 128-channel groups, padded states, bf16."""
import pytest

import oracle
import workloads
from tests.parity import check, to_device, to_numpy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped by marker
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2412_16602_gb300 as vmb  # noqa: E402

DEV = torch.device("cuda", 0)

CASES = [
    # (B, D, N, H, W, dtype, flags beyond softplus)
    (1, 15, 16, 13, 10, "f32", 0),    # L = 130
    (2, 17, 16, 9, 14, "f32", 0),     # one chunk
    (1, 128, 8, 16, 24, "f32", 0),
    (1, 131, 16, 16, 24, "f32", 0),
    (1, 300, 13, 12, 22, "f32", vmb.VMB_FLAG_SKIP_MEAN),
    (1, 131, 16, 16, 24, "bf16", 0),
    (2, 40, 5, 10, 13, "bf16", vmb.VMB_FLAG_SKIP_MEAN),
]


@pytest.mark.parametrize("tc", [64, 128])
@pytest.mark.parametrize("case", CASES, ids=["B{}_D{}_N{}_{}x{}_{}_f{}".format(*c) for c in CASES])
def test_two_steps_per_thread(case, tc, force_plan):
    B, D, N, H, W, dt, extra = case
    force_plan.mean(tc)
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype=dt, seed=900 + D + N)
    inp = workloads.make_inputs(wl, params="random")
    g = to_device(inp, DEV)
    flags = vmb.VMB_FLAG_SOFTPLUS | extra

    def block(delta):
        return vmb.vmb_ss2d_mean_fwd(g["x"], delta, g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], flags=flags)

    out, ybar = block(g["draw"])
    buf = torch.empty(g["draw"].numel() + 1, dtype=g["draw"].dtype, device=DEV)
    shifted = buf[1:].view(g["draw"].shape)
    shifted.copy_(g["draw"])
    out1, ybar1 = block(shifted)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    assert torch.equal(ybar, ybar1) and torch.equal(out, out1)
    mode = dict(skip_mode=oracle.SKIP_MEAN) if extra else {}
    _, _, _, out_ref = oracle.ss2d_mean(inp, **mode)
    check(to_numpy(out), out_ref, dt, "mean out from the map")
