"""The channel-mean scan with two steps per thread (chunks of 64 or 128 steps, 8 or
16 padded states, even L): every form that takes it (the block from the map; in bf16 also
y written, saved means, groups and low-rank Delta) bit for bit against the one-step
kernel, and the block and the scan against the fp64 oracle.  The number of steps is
forced, two steps through a control that refuses calls which cannot take them.  Sizes: a
ragged last chunk of two steps, one chunk, several chunks over more than one group of
128 channels, channels around the 16-channel request batches, padded states, bf16."""
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

    force_plan.mean_steps(2)
    out, ybar = block(g["draw"])
    buf = torch.empty(g["draw"].numel() + 1, dtype=g["draw"].dtype, device=DEV)
    shifted = buf[1:].view(g["draw"].shape)
    shifted.copy_(g["draw"])
    with pytest.raises(vmb.VmbError):  # pairs of steps cannot be loaded as one
        block(shifted)
    force_plan.mean_steps(1)
    out1, ybar1 = block(g["draw"])
    force_plan.mean_steps(0)
    out2, ybar2 = block(shifted)
    assert torch.equal(ybar, ybar2) and torch.equal(out, out2)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    assert torch.equal(ybar, ybar1) and torch.equal(out, out1)
    mode = dict(skip_mode=oracle.SKIP_MEAN) if extra else {}
    _, _, _, out_ref = oracle.ss2d_mean(inp, **mode)
    check(to_numpy(out), out_ref, dt, "mean out from the map")


@pytest.mark.parametrize("tc", [64, 128])
@pytest.mark.parametrize("form", ["y", "train", "grouped", "lowrank"])
@pytest.mark.parametrize("shape", [(2, 40, 5, 10, 13), (1, 264, 16, 12, 26)], ids=["D40_N5", "D264_N16"])
def test_two_steps_with_y_in_bf16(shape, form, tc, force_plan):
    B, D, N, H, W = shape
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype="bf16", seed=40 + D)
    inp = workloads.make_inputs(wl, params="random")
    g = to_device(inp, DEV)
    xs = vmb.vmb_cross_scan(g["x"])
    args = (xs, g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W)
    gen = torch.Generator(device=DEV).manual_seed(D)
    z = torch.randn(B, 4, 6, H * W, device=DEV, generator=gen)
    wup = 0.2 * torch.randn(4, D, 6, device=DEV, generator=gen)
    force_plan.mean(tc)

    def run():
        if form == "y":
            return vmb.vmb_mean_scan_fwd(*args, want_ybar=True)
        if form == "train":
            return vmb.vmb_mean_scan_train_fwd(*args)[:2]
        if form == "grouped":
            return vmb.vmb_mean_scan_grouped_fwd(*args, 4, want_ybar=True)
        return vmb.vmb_mean_scan_lowrank_fwd(xs, z, wup, g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W,
                                             want_ybar=True)

    force_plan.mean_steps(2)
    two = run()
    force_plan.mean_steps(1)
    one = run()
    assert vmb.vmb_read_status() == vmb.VMB_OK
    assert all(torch.equal(a, b) for a, b in zip(two, one))
    if form == "y":
        check(to_numpy(two[0]), oracle.ss2d_mean(inp)[1], "bf16", "mean y")
