"""The fused broadcast + merge with two, four and eight positions a thread (fp32
and bf16; by the row length and the alignment of x and out): every width gives
the bits of the element path, which the same call takes on a map one element
into an allocation.  Channels around the batches of four."""
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped by marker
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2412_16602_gb300 as vmb  # noqa: E402

DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("shape", [(1, 1, 4, 4), (2, 7, 6, 6), (1, 70, 9, 10), (3, 5, 16, 40), (1, 13, 7, 9)],
                         ids=lambda s: "B{}_D{}_{}x{}".format(*s))
def test_merge_widths(shape, dt):
    B, D, H, W = shape
    wl = workloads.small_case(B=B, D=D, N=16, H=H, W=W, dtype=dt, seed=D)
    g = workloads.make_device_inputs(wl, DEV, params="random")
    args = (g["draw"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["bias"])
    xs = vmb.vmb_cross_scan(g["x"])
    out, _ = vmb.vmb_mean_scan_merge_fwd(xs, *args, g["x"], H, W)
    buf = torch.empty(g["x"].numel() + 1, dtype=g["x"].dtype, device=DEV)
    x1 = buf[1:].view(g["x"].shape)
    x1.copy_(g["x"])
    out1, _ = vmb.vmb_mean_scan_merge_fwd(xs, *args, x1, H, W)
    assert vmb.vmb_read_status() == vmb.VMB_OK
    assert torch.equal(out, out1)
