"""The map transpose of the blocks from the map, and the scan CTAs that run beside
it: the channel-mean block and the full block bit for bit against the calls on
cross-scanned sequences.  The planner's choice three times in a row with new inputs; then
the gathering scans themselves (the full scan's plans forced: one pass and chunks, one
and two lanes; many maps, so that the channel-mean scan runs beside the transpose too) on
the same buffers, call after call with nothing in between, so that the next call's
transpose follows the last one's readers at once.  Sizes: 16-byte vectors and
single elements, several planes an item and a ragged last item, the largest
plane of each form, and planes that fall back to 32 x 32 tiles."""
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped by marker
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2412_16602_gb300 as vmb  # noqa: E402

DEV = torch.device("cuda", 0)

CASES = [
    # (B, D, H, W, dtype)
    (1, 1, 4, 4, "f32"),
    (3, 331, 4, 8, "f32"),      # several planes an item, the last item ragged
    (2, 40, 28, 28, "f32"),
    (2, 307, 14, 14, "f32"),    # single elements
    (1, 3, 88, 92, "f32"),      # near the largest vector plane
    (1, 2, 90, 91, "f32"),      # near the largest element plane
    (1, 2, 128, 128, "f32"),    # tiles
    (1, 3, 128, 128, "bf16"),   # the largest bf16 vector plane
    (2, 35, 9, 16, "bf16"),
    (1, 5, 1, 40, "f32"),
]


@pytest.mark.parametrize("case", CASES, ids=["B{}_D{}_{}x{}_{}".format(*c) for c in CASES])
def test_blocks_from_the_map_match_cross_scanned_calls(case):
    B, D, H, W, dt = case
    wl = workloads.small_case(B=B, D=D, N=16, H=H, W=W, dtype=dt, seed=D + H)
    for rep in range(3):
        g = workloads.make_device_inputs(wl, DEV, seed=rep, params="random")
        args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
        om, ybar = vmb.vmb_ss2d_mean_fwd(g["x"], *args)
        of, y = vmb.vmb_ss2d_full_fwd(g["x"], *args)
        xs = vmb.vmb_cross_scan(g["x"])
        om2, ybar2 = vmb.vmb_mean_scan_merge_fwd(xs, *args, g["x"], H, W)
        y2 = vmb.vmb_selective_scan_fwd(xs, *args, H, W)
        assert vmb.vmb_read_status() == vmb.VMB_OK
        assert torch.equal(ybar, ybar2) and torch.equal(om, om2)
        assert torch.equal(y, y2) and torch.equal(of, vmb.vmb_cross_merge(y2, H, W))


@pytest.mark.parametrize("plan", ["19", "19,4", "23", "23,4"])
@pytest.mark.parametrize("case", [(6, 72, 20, 24, "f32"), (3, 130, 16, 44, "bf16"), (2, 33, 28, 28, "f32"),
                                  (1, 40, 96, 96, "f32")], ids=lambda c: "B{}_D{}_{}x{}_{}".format(*c))
def test_calls_in_a_row_on_the_same_buffers(case, plan, force_plan):
    B, D, H, W, dt = case
    force_plan.full(plan)
    wl = workloads.small_case(B=B, D=D, N=16, H=H, W=W, dtype=dt, seed=D)
    sets = [workloads.make_device_inputs(wl, DEV, seed=i, params="random") for i in range(4)]
    want = []
    for g in sets:
        args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
        xs = vmb.vmb_cross_scan(g["x"])
        y = vmb.vmb_selective_scan_fwd(xs, *args, H, W)
        om, yb = vmb.vmb_mean_scan_merge_fwd(xs, *args, g["x"], H, W)
        want.append((y, vmb.vmb_cross_merge(y, H, W), om, yb))
    x, xt = torch.empty_like(sets[0]["x"]), torch.empty(B, D, W, H, dtype=sets[0]["x"].dtype, device=DEV)
    delta, y = torch.empty_like(sets[0]["draw"]), torch.empty_like(sets[0]["draw"])
    out, om, yb = torch.empty_like(x), torch.empty_like(x), torch.empty(B, 4, H * W, device=DEV)
    ws = torch.zeros(32 << 20, dtype=torch.uint8, device=DEV)
    got = []
    torch.cuda.synchronize()
    for rep in range(8):
        g = sets[rep % 4]
        x.copy_(g["x"])
        delta.copy_(g["draw"])
        args = (delta, g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
        vmb.vmb_ss2d_full_fwd(x, *args, out=out, y=y, xt=xt, workspace=ws)
        vmb.vmb_ss2d_mean_fwd(x, *args, out=om, ybar=yb, xt=xt, workspace=ws)
        vmb.vmb_ss2d_full_fwd(x, *args, out=out, y=y, xt=xt, workspace=ws)
        got.append(tuple(t.clone() for t in (y, out, om, yb)))
    assert vmb.vmb_read_status(ws) == vmb.VMB_OK
    for rep, outs in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(outs, want[rep % 4])), rep


@pytest.mark.parametrize("case,beside", [
    # (B, D, N, H, W, dtype, x out of line): 16 states in at most a CTA per SM, four states, two CTAs per SM
    ((1, 1536, 16, 32, 32, "f32", 0), 1), ((1, 1536, 16, 28, 20, "bf16", 1), 1), ((1, 1536, 4, 32, 32, "f32", 0), 0),
    ((2, 1024, 16, 30, 30, "f32", 0), 0), ((1, 1024, 4, 48, 72, "f32", 0), 1), ((1, 1024, 4, 48, 72, "f32", 1), 0),
    ((1, 1024, 8, 28, 28, "f32", 0), 1), ((1, 1536, 8, 30, 30, "f32", 0), 0), ((1, 1536, 8, 32, 32, "bf16", 0), 1),
    ((2, 1024, 16, 22, 48, "f32", 1), 0), ((8, 1024, 16, 28, 28, "f32", 0), 1), ((1, 1536, 16, 10, 10, "f32", 0), 1),
])
def test_mean_scan_beside_the_transpose(case, beside):
    import ctypes

    i = ctypes.c_int
    vmb.lib.vmb_testing_mean_beside.argtypes = [i] * 7
    B, D, N, H, W, dt, off = case
    assert vmb.lib.vmb_testing_mean_beside(B, D, N, H, W, vmb.VMB_F32 if dt == "f32" else vmb.VMB_BF16, off) == beside


def test_mean_block_of_many_maps_in_a_row():
    """Enough CTAs that the channel-mean scan starts beside the transpose by planes."""
    B, D, H, W = 40, 24, 24, 28
    wl = workloads.small_case(B=B, D=D, N=16, H=H, W=W, seed=9)
    sets = [workloads.make_device_inputs(wl, DEV, seed=i, params="random") for i in range(2)]
    out, yb = torch.empty_like(sets[0]["x"]), torch.empty(B, 4, H * W, device=DEV)
    xt, got, want = torch.empty(B, D, W, H, device=DEV), [], []
    for g in sets:
        args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
        want.append(vmb.vmb_mean_scan_merge_fwd(vmb.vmb_cross_scan(g["x"]), *args, g["x"], H, W))
    for rep in range(6):
        g = sets[rep % 2]
        args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
        for _ in range(3):
            vmb.vmb_ss2d_mean_fwd(g["x"], *args, out=out, ybar=yb, xt=xt)
        got.append((out.clone(), yb.clone()))
    assert vmb.vmb_read_status() == vmb.VMB_OK
    for rep, (o, y) in enumerate(got):
        assert torch.equal(o, want[rep % 2][0]) and torch.equal(y, want[rep % 2][1])
