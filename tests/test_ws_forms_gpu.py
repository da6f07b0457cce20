"""The forms of the warp-specialised full scan beyond one lane per channel and 16
states: two lanes per channel (shape 23, with 8 padded states 3), L cut into chunks by
two launches (chunks of shapes 19 and 23 and of fewer states), and 1 to 8 states (shape 1,
with 8 padded states 2), against the fp64 oracle, deterministic, and as the
block from the map bit for bit against the three separate calls.  Sizes: ragged
last stages and chunks, ragged channel tiles, padded states, bf16."""
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
    # (plan, B, D, N, H, W, dtype)
    ("23", 1, 72, 16, 9, 12, "f32"),     # L = 108: a ragged last 16-step stage; a tile with one of four warps short
    ("23", 2, 40, 13, 16, 24, "bf16"),
    ("23", 1, 65, 16, 56, 56, "f32"),    # one channel in the second tile
    ("23,3", 1, 72, 16, 20, 30, "f32"),  # L = 600: chunks of 208 steps, the last one ragged
    ("23,7", 2, 40, 16, 16, 24, "bf16"),
    ("23,25", 1, 33, 16, 40, 40, "f32"),  # 24 aggregates to fold
    ("19,4", 1, 130, 16, 20, 30, "f32"),
    ("1", 2, 72, 1, 9, 12, "f32"),
    ("1", 1, 130, 2, 16, 24, "bf16"),
    ("1", 1, 40, 3, 20, 30, "f32"),      # padded to 4 states
    ("2", 2, 72, 5, 9, 12, "f32"),       # padded to 8 states
    ("2", 1, 40, 8, 16, 24, "bf16"),
    ("1,4", 1, 130, 1, 20, 30, "f32"),
    ("2,5", 1, 40, 8, 20, 30, "f32"),
    ("3", 2, 72, 5, 9, 12, "f32"),       # padded to 8 states, two lanes
    ("3", 1, 65, 8, 16, 24, "bf16"),
    ("3,5", 1, 40, 8, 20, 30, "f32"),
]


@pytest.mark.parametrize("case", CASES, ids=["plan{}_B{}_D{}_N{}_{}x{}_{}".format(*c) for c in CASES])
def test_warp_specialised_forms(case, force_plan):
    plan, B, D, N, H, W, dt = case
    force_plan.full(plan)
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype=dt, seed=500 + D + N)
    inp = workloads.make_inputs(wl, params="random")
    g = to_device(inp, DEV)
    args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
    xs = vmb.vmb_cross_scan(g["x"])
    y = vmb.vmb_selective_scan_fwd(xs, *args, H, W)
    y2 = vmb.vmb_selective_scan_fwd(xs, *args, H, W)
    out, ym = vmb.vmb_ss2d_full_fwd(g["x"], *args)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    _, y_ref, out_ref = oracle.ss2d_full(inp)
    check(to_numpy(y), y_ref, dt, "full y")
    check(to_numpy(out), out_ref, dt, "full out from the map")
    assert torch.equal(y, y2), "deterministic"
    assert torch.equal(ym, y) and torch.equal(out, vmb.vmb_cross_merge(y, H, W))


@pytest.mark.parametrize("N", [16, 4])
def test_workspace_of_the_query_serves_any_alignment(N):
    """A workspace of exactly the queried size: aligned tensors take the chunked
    warp-specialised plan, the same tensors one element into an allocation
    another one with another workspace."""
    B, D, H, W = 4, 64, 33, 32
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, seed=77)
    inp = workloads.make_inputs(wl, params="random")
    g = to_device(inp, DEV)
    xs = vmb.vmb_cross_scan(g["x"])
    _, y_ref, _ = oracle.ss2d_full(inp)
    for shift in (0, 1):
        buf = torch.empty(xs.numel() + shift, device=DEV)
        u = buf[shift:].view(xs.shape)
        u.copy_(xs)
        ws = torch.zeros(vmb.vmb_scan_workspace_bytes(vmb.VMB_PATH_FULL, B, 4, D, N, H, W), dtype=torch.uint8,
                         device=DEV)
        y = vmb.vmb_selective_scan_fwd(u, g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W, workspace=ws)
        assert vmb.vmb_read_status(ws) == vmb.VMB_OK
        check(to_numpy(y), y_ref, "f32", f"full y, shifted by {shift}")


@pytest.mark.parametrize("case,shape", [
    # (B, D, N, H, W, dtype): 8 padded states take two lanes for few rows of 16 steps or more
    ((38, 64, 8, 8, 8, "f32"), 3), ((38, 64, 5, 8, 8, "bf16"), 3), ((4, 64, 8, 128, 128, "bf16"), 3),
    ((38, 64, 8, 2, 4, "f32"), 2), ((160, 64, 8, 8, 8, "f32"), 2), ((38, 64, 4, 8, 8, "f32"), 1),
])
def test_planner_of_eight_states(case, shape, full_plan):
    B, D, N, H, W, dt = case
    assert full_plan(B, 4, D, N, H, W, dt)[0] == shape
    assert full_plan(B, 4, D, N, H, W, dt, map=True)[0] == shape


@pytest.mark.parametrize("case,chunks", [((4, 192, 8, 16, 18, "f32"), 4), ((8, 192, 8, 16, 18, "bf16"), 1),
                                         ((4, 192, 8, 8, 16, "f32"), 1)])
def test_planner_cuts_eight_states_into_chunks(case, chunks, full_plan):
    B, D, N, H, W, dt = case
    assert full_plan(B, 4, D, N, H, W, dt)[:2] == (3, chunks)


@pytest.mark.parametrize("case,early", [
    # (B, D, N, H, W, dtype, off, flags beyond softplus): barrier-staged plans; a grid of less than one wave
    # of long-lived CTAs is not launched early, tiny sequences and full waves are
    ((36, 64, 16, 12, 12, "f32", 0, vmb.VMB_FLAG_B_ZOH), 0), ((3, 1536, 3, 2, 64, "bf16", 1, 0), 0),
    ((2, 256, 4, 28, 28, "f32", 0, vmb.VMB_FLAG_B_ZOH), 0), ((2, 96, 5, 20, 20, "bf16", 1, 0), 0),
    ((2, 96, 16, 20, 20, "bf16", 1, 0), 1), ((3, 1536, 3, 2, 16, "bf16", 1, 0), 1), ((128, 512, 4, 8, 8, "f32", 1, 0), 1),
])
def test_barrier_staged_grids_launched_early(case, early, full_plan):
    B, D, N, H, W, dt, off, flags = case
    assert full_plan(B, 4, D, N, H, W, dt, off=off, flags=vmb.VMB_FLAG_SOFTPLUS | flags)[2] == early


@pytest.mark.parametrize("case", [
    # (plan, B, D, N, H, W, dtype)
    ("", 2, 200, 1, 16, 24, "f32"), ("", 4, 200, 4, 20, 30, "bf16"), ("", 2, 200, 8, 16, 24, "f32"),
    ("23", 2, 72, 16, 20, 30, "f32"), ("23,4", 1, 72, 16, 20, 30, "bf16"), ("19", 2, 130, 13, 9, 12, "f32"),
    ("19,4", 1, 130, 16, 20, 30, "f32"),
], ids=lambda c: "plan{}_B{}_D{}_N{}_{}x{}_{}".format(*c))
def test_tensor_maps_refused(case, force_plan, full_plan):
    """Where the driver refuses the tensor maps, a call runs on kernels without tensor
    copies: the scan, the block from the map and the low-rank form."""
    plan, B, D, N, H, W, dt = case
    if plan:
        force_plan.full(plan)
    else:
        shape = full_plan(B, 4, D, N, H, W, dt)[0]
        assert shape >= (1 if N <= 4 else 2)  # the warp-specialised kernel
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype=dt, seed=600 + D + N)
    inp = workloads.make_inputs(wl, params="random")
    g = to_device(inp, DEV)
    args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
    xs = vmb.vmb_cross_scan(g["x"])
    gen = torch.Generator(device=DEV).manual_seed(7)
    z = torch.randn(B, 4, 5, H * W, device=DEV, generator=gen)
    wup = 0.2 * torch.randn(4, D, 5, device=DEV, generator=gen)
    low = (xs, z, wup, g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W)
    y_low = vmb.vmb_selective_scan_lowrank_fwd(*low)
    force_plan.refuse_tensor_maps()
    force_plan.full("-1")
    y = vmb.vmb_selective_scan_fwd(xs, *args, H, W)
    out, ym = vmb.vmb_ss2d_full_fwd(g["x"], *args)
    y_low2 = vmb.vmb_selective_scan_lowrank_fwd(*low)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    _, y_ref, out_ref = oracle.ss2d_full(inp)
    check(to_numpy(y), y_ref, dt, "full y")
    check(to_numpy(ym), y_ref, dt, "full y from the map")
    check(to_numpy(out), out_ref, dt, "full out from the map")
    # (the raw Deltas are rounded to bf16 where they are materialised)
    check(to_numpy(y_low2), to_numpy(y_low).astype("float64"), dt, "low rank")


@pytest.mark.parametrize("case", [
    # (plan, B, D, N, R, H, W, dtype)
    ("23", 1, 72, 16, 5, 20, 30, "f32"), ("23", 2, 40, 13, 12, 9, 12, "f32"), ("23,4", 1, 65, 16, 16, 20, 30, "f32"),
    ("23", 1, 72, 16, 7, 16, 24, "bf16"), ("23,3", 2, 33, 9, 11, 20, 30, "bf16"),
    ("3", 1, 72, 8, 5, 20, 30, "f32"), ("3,4", 1, 72, 5, 9, 20, 30, "f32"), ("1,4", 1, 130, 2, 3, 20, 30, "f32"),
    ("2", 1, 40, 8, 16, 16, 24, "bf16"), ("1,5", 2, 40, 4, 6, 20, 30, "bf16"),
], ids=lambda c: "plan{}_B{}_D{}_N{}_R{}_{}x{}_{}".format(*c))
def test_lowrank_forms(case, force_plan):
    """The low-rank Delta with two lanes per channel and in chunks, and, for 8 states or
    fewer, expanded into y and scanned in place: against the scan of the materialised
    raw Deltas with the same plan (bit for bit in fp32, and in bf16 in place)."""
    plan, B, D, N, R, H, W, dt = case
    force_plan.full(plan)
    wl = workloads.small_case(B=B, D=D, N=N, H=H, W=W, dtype=dt, seed=700 + D + R)
    g = to_device(workloads.make_inputs(wl, params="random"), DEV)
    xs = vmb.vmb_cross_scan(g["x"])
    gen = torch.Generator(device=DEV).manual_seed(R)
    z = torch.randn(B, 4, R, H * W, device=DEV, generator=gen)
    wup = 0.3 * torch.randn(4, D, R, device=DEV, generator=gen)
    y = vmb.vmb_selective_scan_lowrank_fwd(xs, z, wup, g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W)
    raw = torch.zeros(B, 4, D, H * W, device=DEV, dtype=torch.float64)
    for r in range(R):  # in the kernel's order, every fused multiply-add rounded to fp32
        raw = (raw + wup[None, :, :, r, None].double() * z[:, :, None, r].double()).float().double()
    y2 = vmb.vmb_selective_scan_fwd(xs, raw.to(xs.dtype), g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"], H, W)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    if dt == "f32" or N <= 8:
        assert torch.equal(y, y2)
    else:
        check(to_numpy(y), to_numpy(y2).astype("float64"), dt, "low rank")


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("case", [
    # (B, K, D, N, L, dtype): narrow tiles, whole tiles and one row more, stages cut short
    (2, 4, 3, 2, 67, "bf16"), (1, 4, 3, 8, 67, "f32"), (1, 2, 129, 1, 51, "bf16"), (1, 2, 129, 4, 51, "f32"),
    (2, 4, 35, 9, 301, "bf16"), (1, 4, 16, 16, 1201, "f32"), (1, 2, 65, 16, 1201, "bf16"), (3, 4, 17, 5, 130, "bf16"),
], ids=lambda c: "B{}_K{}_D{}_N{}_L{}_{}".format(*c))
def test_rows_out_of_line(case, off):
    """Rows that are not 16-byte aligned, by length (off 0) or also by address (off 1),
    in every barrier-staged plan that the planner takes for them: against the oracle."""
    B, K, D, N, L, dt = case
    gen = torch.Generator().manual_seed(L + D)
    td = torch.float32 if dt == "f32" else torch.bfloat16
    u, delta = (torch.randn(B, K, D, L, generator=gen).to(td) for _ in range(2))
    Bs, Cs = (torch.randn(B, K, N, L, generator=gen).to(td) for _ in range(2))
    A = -(torch.arange(N) + 1.0) * (0.8 + 0.4 * torch.rand(K * D, N, generator=gen))
    dsk, bias = 0.75 + 0.5 * torch.rand(K * D, generator=gen), torch.randn(K * D, generator=gen) * 0.3 - 3.0

    def put(t):
        buf = torch.empty(t.numel() + off, dtype=t.dtype, device=DEV)[off:]
        return buf.view(t.shape).copy_(t)

    y = vmb.vmb_selective_scan_fwd(put(u), put(delta), A.to(DEV), put(Bs), put(Cs), dsk.to(DEV), bias.to(DEV), 1, L)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    # Eqs. 3, 4 and 6 in fp64
    d = torch.nn.functional.softplus(delta.double() + bias.double().view(1, K, D, 1))
    h = torch.zeros(B, K, D, N, dtype=torch.float64)
    ref = torch.empty(B, K, D, L, dtype=torch.float64)
    a64 = A.double().view(1, K, D, N)
    for t in range(L):
        h = torch.exp(d[..., t, None] * a64) * h + (d[..., t] * u[..., t].double())[..., None] * Bs.double()[:, :, None, :, t]
        ref[..., t] = (h * Cs.double()[:, :, None, :, t]).sum(-1) + dsk.double().view(1, K, D) * u[..., t].double()
    check(to_numpy(y), ref.numpy(), dt, "y of rows out of line")
