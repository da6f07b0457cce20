"""The whole-sequence kernel of short sequences (full-scan shapes 20 to 22: 1, 4
and 16 lanes a channel), alone and as the one-launch block, against the fp64
oracle; the block bit for bit against the three separate calls.  Sizes sit at
the edges of its tiles: one step, lengths around the step blocks (4 and 16),
the longest sequence of each rule, ragged channel tiles, padded states, bf16,
odd rows and a plane one pixel wide."""
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

SHAPES = [
    # (B, D, N, H, W, dtype)
    (1, 5, 16, 1, 1, "f32"),
    (2, 33, 16, 1, 7, "f32"),
    (1, 9, 16, 5, 3, "bf16"),
    (3, 70, 16, 7, 7, "f32"),
    (2, 40, 13, 4, 4, "bf16"),
    (1, 34, 16, 17, 1, "f32"),
    (2, 32, 9, 8, 12, "f32"),
    (1, 19, 16, 16, 16, "f32"),
    (8, 512, 16, 4, 4, "f32"),   # planner: the block with one lane a channel, the scan alone warp-specialised
    (8, 500, 16, 3, 5, "bf16"),  # planner: one lane a channel for both
]


@pytest.mark.parametrize("plan", ["20", "21", "22", ""])
@pytest.mark.parametrize("shape", SHAPES, ids=[f"B{s[0]}_D{s[1]}_N{s[2]}_{s[3]}x{s[4]}_{s[5]}" for s in SHAPES])
def test_short_sequences(shape, plan, force_plan):
    B, D, N, H, W, dt = shape
    if plan:
        force_plan.full(plan)
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype=dt, seed=300 + D + N)
    inp = workloads.make_inputs(wl, params="random")
    g = to_device(inp, DEV)
    args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
    y = vmb.vmb_selective_scan_fwd(vmb.vmb_cross_scan(g["x"]), *args, H, W)
    out, ym = vmb.vmb_ss2d_full_fwd(g["x"], *args)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    _, y_ref, out_ref = oracle.ss2d_full(inp)
    check(to_numpy(y), y_ref, dt, "full y")
    assert torch.equal(ym, y) and torch.equal(out, vmb.vmb_cross_merge(y, H, W))
    check(to_numpy(out), out_ref, dt, "full out from the map")


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[3] * s[4] > 1], ids=lambda s: "B{}_D{}_N{}_{}x{}_{}".format(*s))
def test_whole_sequences_and_lane_per_state_agree_bit_for_bit(shape, force_plan):
    """4 and 16 lanes of whole sequences (the block) add the states in the order of the
    lane-per-state kernel (shape 7), which the scan alone may take instead."""
    B, D, N, H, W, dt = shape
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype=dt, seed=310 + D)
    g = to_device(workloads.make_inputs(wl, params="random"), DEV)
    args = (vmb.vmb_cross_scan(g["x"]), g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W)
    ys = []
    for plan in ("7", "21", "22"):
        force_plan.full(plan)
        ys.append(vmb.vmb_selective_scan_fwd(*args))
    assert vmb.vmb_read_status() == vmb.VMB_OK
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])


@pytest.mark.parametrize("shape", [(3, 70, 16, 9, 9, "bf16"), (2, 130, 9, 7, 11, "bf16"), (1, 40, 13, 5, 15, "f32")],
                         ids=lambda s: "B{}_D{}_N{}_{}x{}_{}".format(*s))
def test_whole_sequences_and_packed_agree_bit_for_bit(shape, force_plan):
    """One lane of whole sequences (the block) and the packed streaming kernel (shape 16),
    which the scan alone may take instead, on rows out of line."""
    B, D, N, H, W, dt = shape
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype=dt, seed=320 + D)
    g = to_device(workloads.make_inputs(wl, params="random"), DEV)
    args = (vmb.vmb_cross_scan(g["x"]), g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W)
    ys = []
    for plan in ("16", "20"):
        force_plan.full(plan)
        ys.append(vmb.vmb_selective_scan_fwd(*args))
    assert vmb.vmb_read_status() == vmb.VMB_OK
    assert torch.equal(ys[0], ys[1])


LANES, PACKED, ONE, FOUR, SIXTEEN = 7, 16, 20, 21, 22


@pytest.mark.parametrize("case,map_shape,scan_shape", [
    # (B, D, H, W, dtype): rows per SM from 2 to 50
    ((2, 32, 8, 8, "f32"), SIXTEEN, LANES), ((12, 32, 14, 16, "f32"), FOUR, LANES), ((19, 32, 4, 56, "bf16"), FOUR, LANES),
    ((2, 32, 2, 4, "f32"), SIXTEEN, SIXTEEN), ((36, 32, 5, 8, "f32"), FOUR, FOUR), ((36, 32, 8, 12, "f32"), FOUR, LANES),
    ((1, 40, 10, 10, "f32"), SIXTEEN, SIXTEEN), ((3, 64, 16, 18, "f32"), LANES, LANES),
    ((30, 64, 16, 18, "f32"), 23, 23), ((60, 32, 8, 12, "f32"), FOUR, FOUR), ((60, 32, 8, 10, "bf16"), FOUR, LANES),
    # rows out of line, up to four CTAs of the lane-per-state kernel per SM
    ((71, 32, 7, 29, "f32"), LANES, LANES), ((44, 32, 13, 23, "bf16"), LANES, LANES),
    # few channels per sequence: tiles of the chunked three launches would be mostly padding
    ((19, 7, 20, 20, "f32"), LANES, LANES), ((7, 32, 20, 20, "bf16"), LANES, LANES), ((7, 32, 32, 32, "f32"), 9, 9),
    ((6, 24, 20, 20, "bf16"), 9, 9),
    # the scan alone, rows out of line
    ((16, 32, 7, 29, "bf16"), FOUR, LANES), ((16, 32, 7, 29, "f32"), FOUR, LANES), ((110, 7, 7, 29, "f32"), FOUR, FOUR),
    ((51, 7, 13, 13, "f32"), SIXTEEN, SIXTEEN), ((51, 7, 13, 13, "bf16"), SIXTEEN, LANES),
    ((49, 400, 9, 9, "bf16"), ONE, PACKED), ((49, 400, 9, 9, "f32"), ONE, ONE), ((40, 400, 9, 9, "bf16"), ONE, ONE),
])
def test_planner_of_short_sequences(case, map_shape, scan_shape, full_plan):
    B, D, H, W, dt = case
    assert full_plan(B, 4, D, 16, H, W, dt, map=True)[0] == map_shape
    assert full_plan(B, 4, D, 16, H, W, dt)[0] == scan_shape
    wl = workloads.small_case(B=B, D=D, N=16, H=H, W=W, dtype=dt, seed=B)
    g = workloads.make_device_inputs(wl, DEV, seed=B, params="random")
    args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
    out, y = vmb.vmb_ss2d_full_fwd(g["x"], *args)
    y2 = vmb.vmb_selective_scan_fwd(vmb.vmb_cross_scan(g["x"]), *args, H, W)
    assert torch.equal(y, y2) and torch.equal(out, vmb.vmb_cross_merge(y2, H, W))


@pytest.mark.parametrize("case", [(8, 512, 10, 12, "f32"), (8, 512, 8, 13, "bf16"), (3, 700, 9, 12, "f32"),
                                  (8, 512, 8, 8, "f32"), (2, 40, 10, 12, "f32"), (8, 256, 12, 12, "f32"), (2, 64, 28, 28, "f32"),
                                  (1, 40, 40, 42, "bf16")],
                         ids=lambda c: "B{}_D{}_{}x{}_{}".format(*c))
@pytest.mark.parametrize("which", ["x", "xt"])
def test_block_of_an_unaligned_map(case, which):
    """x or xt one element past 16-byte alignment: y and out are those of the three calls
    on aligned sequences, bit for bit, with a workspace of the queried size."""
    B, D, H, W, dt = case
    wl = workloads.small_case(B=B, D=D, N=16, H=H, W=W, dtype=dt, seed=B + D)
    g = workloads.make_device_inputs(wl, DEV, seed=3, params="random")
    args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
    x = g["x"]
    off = torch.empty(x.numel() + 1, dtype=x.dtype, device=DEV)[1:]
    ws = torch.zeros(vmb.vmb_scan_workspace_bytes(vmb.VMB_PATH_FULL, B, 4, D, 16, H, W, x.dtype), dtype=torch.uint8,
                     device=DEV)
    if which == "x":
        out, y = vmb.vmb_ss2d_full_fwd(off.view(x.shape).copy_(x), *args, workspace=ws)
    else:
        out, y = vmb.vmb_ss2d_full_fwd(x, *args, xt=off.view(B, D, W, H), workspace=ws)
    y2 = vmb.vmb_selective_scan_fwd(vmb.vmb_cross_scan(x), *args, H, W)
    assert vmb.vmb_read_status(ws) == vmb.VMB_OK
    assert torch.equal(y, y2) and torch.equal(out, vmb.vmb_cross_merge(y2, H, W))
