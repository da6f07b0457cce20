"""The map transpose of the blocks from the map, and the scan CTAs that run beside
it: the channel-mean block and the full block bit for bit against the calls on
cross-scanned sequences, several times in a row on one stream (the next call's
transpose follows the last one's readers at once).  Sizes: 16-byte vectors and
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
