"""Cross-scan (bit for bit) and cross-merge (integer values, exact) at the edges of
their kernels: planes of one pixel, one row or one column, a grid of one plane a
CTA and of many, the largest plane-kernel map (1023 pixels), the band kernels on
a plane larger than shared memory, and rows too long for a band."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped by marker
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2412_16602_gb300 as vmb  # noqa: E402

DEV = torch.device("cuda", 0)

CASES = [(1, 1, 1, 1), (2, 3, 1, 9), (3, 2, 31, 33), (1, 3, 33, 31), (2, 2, 1, 1023), (1, 2, 1023, 1), (7, 900, 4, 4),
         (5, 130, 3, 5), (1, 2, 230, 232), (1, 1, 3, 3300),
         # long rows and tall planes: whole planes without index tables, bands, single elements
         (1, 3, 1, 9000), (2, 2, 7, 3201), (1, 2, 2, 8001), (1, 2, 3, 8793), (1, 1, 201, 201), (1, 2, 14, 1948),
         (1, 1, 300, 256), (1, 1, 7001, 12), (1, 1, 128, 800),
         # enough planes of long rows: whole planes, in line and not
         (2, 10, 1, 9000), (1, 80, 3, 6401), (2, 40, 7, 6999), (2, 80, 2, 7000), (1, 160, 1, 6403)]


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("case", CASES, ids=["B{}_D{}_{}x{}".format(*c) for c in CASES])
def test_cross_scan_and_merge(case, dt):
    B, D, H, W = case
    g = torch.Generator().manual_seed(H * W + D)
    x = torch.randint(-30, 31, (B, D, H, W), generator=g).to(dt)
    ys = torch.randint(-30, 31, (B, 4, D, H * W), generator=g).to(dt)
    rows, cols = x.reshape(B, D, -1), x.transpose(2, 3).reshape(B, D, -1)
    ref = torch.stack([rows, cols, rows.flip(-1), cols.flip(-1)], 1)
    assert torch.equal(vmb.vmb_cross_scan(x.to(DEV)).cpu(), ref)
    f = ys.float()
    merged = (f[:, 0] + f[:, 2].flip(-1)).reshape(B, D, H, W) + \
        (f[:, 1] + f[:, 3].flip(-1)).reshape(B, D, W, H).transpose(2, 3)  # |sums| <= 120: exact in both types
    assert torch.equal(vmb.vmb_cross_merge(ys.to(DEV), H, W).float().cpu(), merged)
