"""The work this library is timed on: SS2D blocks and scans over the range of maps, batches, state counts and
storage types that its workloads span, through the public Python entry points.

A case is a dict of plain values:
    kind   "full_map"   vmb_ss2d_full_fwd: cross-scan, full-channel selective scan and cross-merge from the map
           "mean_map"   vmb_ss2d_mean_fwd: cross-scan, channel-mean scan and cross-merge from the map
           "full_scan"  vmb_selective_scan_fwd on sequences that are already cross-scanned
           "mean_scan"  vmb_mean_scan_grouped_fwd on such sequences, `groups` channel groups, with ybar
           "projected"  a block with its selection functions: vmb_cross_scan, vmb_selection_lowrank_fwd, the low-rank
                        scan (`path`: "full" or "mean"), vmb_cross_merge
           "train"      a training step of the channel-mean scan: vmb_mean_scan_train_fwd and vmb_mean_scan_bwd
    B, D, N, H, W       batch, inner channels, states, map height and width (K = 4 directions, L = H * W steps)
    R, groups, path     where the kind takes them
    dtype               "f32" or "bf16": storage type of the maps, sequences, B, C and outputs
    sigma               per-channel noise of the map around the image that its channels share
"""
import math

import torch

import paper_2412_16602_gb300 as vmb

K = 4  # SS2D scan directions
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(kind, B, D, N, H, W, dtype="f32", sigma=0.1, R=0, groups=1, path=""):
    return dict(kind=kind, B=B, D=D, N=N, H=H, W=W, dtype=dtype, sigma=sigma, R=R, groups=groups, path=path)


def listed():
    named = {
        # one image at a late stage: a small map, where launches and latency are all there is
        "full_map_b1_d192_14x14": _case("full_map", 1, 192, 16, 14, 14),
        # one 224 x 224 image at the first stage: few channel rows, a long sequence
        "full_scan_b1_d192_56x56": _case("full_scan", 1, 192, 16, 56, 56),
        # two images of an odd size: a ragged map whose rows are not 16-byte multiples
        "mean_map_b2_d192_45x37": _case("mean_map", 2, 192, 16, 45, 37),
        # the four stages of a classifier's batch of 32 (224 x 224 images): the first as a full block,
        "full_map_b32_d192_56x56": _case("full_map", 32, 192, 16, 56, 56),
        # the second as a training step of the channel-mean layer,
        "train_b32_d384_28x28": _case("train", 32, 384, 16, 28, 28),
        # the third with its selection functions (rank 12 Delta projection),
        "projected_b32_d768_14x14": _case("projected", 32, 768, 16, 14, 14, R=12, path="full"),
        # the last: many channels, very short odd sequences
        "full_map_b32_d1536_7x7": _case("full_map", 32, 1536, 16, 7, 7),
        # segmentation of 512 x 512 images in bf16: very long sequences, both forms of the block
        "full_map_b8_d192_128x128_bf16": _case("full_map", 8, 192, 16, 128, 128, "bf16"),
        "mean_map_b8_d192_128x128_bf16": _case("mean_map", 8, 192, 16, 128, 128, "bf16"),
        # batch-128 classification, 16 states, both forms of the block: the largest work
        "full_map_b128_d256_56x56": _case("full_map", 128, 256, 16, 56, 56, sigma=0.05),
        "mean_map_b128_d256_56x56": _case("mean_map", 128, 256, 16, 56, 56, sigma=0.05),
        # the same batch with one state per channel, where memory and not arithmetic is the limit
        "full_scan_b128_d256_n1_56x56": _case("full_scan", 128, 256, 1, 56, 56, sigma=0.05),
    }
    return [dict(c, name=name) for name, c in named.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes spread over their logarithm, even and odd maps, and at most a third of the largest
    listed case's elements (ragged rows and training steps, which cost more an element, fewer still)."""
    kind = rng.choice(["full_map", "full_map", "mean_map", "mean_map", "full_scan", "mean_scan", "projected", "train"])
    dtype = rng.choice(["f32", "f32", "bf16"])
    N = rng.choice([16, 16, 16, 16, 8, 4, 1])
    if rng.random() < 0.5:  # stage-like maps: multiples of 7 or 8, square
        H = W = rng.choice([7, 14, 28, 56, 112]) if rng.random() < 0.5 else rng.choice([8, 16, 32, 64, 128])
    else:
        H, W = _log_int(rng, 6, 128), _log_int(rng, 6, 128)
    D = rng.choice([1, 2, 3, 4, 6, 8]) * 32 * rng.choice([1, 2, 4]) if rng.random() < 0.7 else _log_int(rng, 24, 1024)
    R = rng.randint(2, 16) if kind == "projected" else 0
    path = rng.choice(["full", "mean"]) if kind == "projected" else ""
    groups = rng.choice([1, 1, 2, 4]) if kind in ("mean_scan", "train") else 1
    D = D // groups * groups
    most = 12_000_000 if kind == "train" or (H * W) % 8 else 34_000_000
    B = min(_log_int(rng, 1, 128), max(1, most // (D * H * W)))
    return _case(kind, B, D, N, H, W, dtype, rng.choice([0.05, 0.1, 0.5]), R, groups, path)


def prepare(case, seed):
    """The tensors a layer holds when it calls the scan.  x = s + sigma e (an image shared by the channels plus
    per-channel noise), raw Delta ~ N(0, 0.5^2), B and C ~ N(0, 1), a Delta bias whose softplus is log-uniform in
    [1e-3, 0.1], A near -(n + 1) and the skip weight near 1, both varying from channel to channel."""
    B, D, N, H, W, L = case["B"], case["D"], case["N"], case["H"], case["W"], case["H"] * case["W"]
    dt = DTYPES[case["dtype"]]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(shape, device="cuda", generator=gen)

    def uniform(*shape):
        return torch.rand(shape, device="cuda", generator=gen)

    st = {"case": case}
    x = (normal(B, 1, H, W) + case["sigma"] * normal(B, D, H, W)).to(dt)
    step = torch.exp(math.log(1e-3) + uniform(K * D).double() * math.log(100.0))
    st["bias"] = (step + torch.log(-torch.expm1(-step))).float()
    st["A"] = -(torch.arange(N, device="cuda") + 1.0) * (0.8 + 0.4 * uniform(K * D, N))
    st["Dskip"] = 0.75 + 0.5 * uniform(K * D)
    if case["kind"] == "projected":
        st["WB"], st["WC"] = normal(K, N, D) / math.sqrt(D), normal(K, N, D) / math.sqrt(D)
        st["Wz"] = normal(K, case["R"], D) / math.sqrt(D)
        st["Wup"] = normal(K, D, case["R"]) * (0.5 / math.sqrt(case["R"]))
    else:
        st["delta"] = (0.5 * normal(B, K, D, L)).to(dt)
        st["Bs"], st["Cs"] = normal(B, K, N, L).to(dt), normal(B, K, N, L).to(dt)
    if case["kind"] in ("full_scan", "mean_scan", "train"):
        st["u"] = vmb.vmb_cross_scan(x)
    else:
        st["x"] = x
    if case["kind"] == "train":
        st["gy"] = normal(B, K, D, L).to(dt)
    return st


def run(st):
    case = st["case"]
    H, W, kind = case["H"], case["W"], case["kind"]
    if kind == "full_map":
        return vmb.vmb_ss2d_full_fwd(st["x"], st["delta"], st["A"], st["Bs"], st["Cs"], st["Dskip"], st["bias"])
    if kind == "mean_map":
        return vmb.vmb_ss2d_mean_fwd(st["x"], st["delta"], st["A"], st["Bs"], st["Cs"], st["Dskip"], st["bias"])
    if kind == "projected":
        xs = vmb.vmb_cross_scan(st["x"])
        z, Bs, Cs = vmb.vmb_selection_lowrank_fwd(xs, st["WB"], st["WC"], st["Wz"], H, W)
        if case["path"] == "full":
            y = vmb.vmb_selective_scan_lowrank_fwd(xs, z, st["Wup"], st["A"], Bs, Cs, st["Dskip"], st["bias"], H, W)
        else:
            y, _ = vmb.vmb_mean_scan_lowrank_fwd(xs, z, st["Wup"], st["A"], Bs, Cs, st["Dskip"], st["bias"], H, W)
        return vmb.vmb_cross_merge(y, H, W), y, z, Bs, Cs
    args = (st["u"], st["delta"], st["A"], st["Bs"], st["Cs"], st["Dskip"], st["bias"])
    if kind == "full_scan":
        return vmb.vmb_selective_scan_fwd(*args, H, W)
    if kind == "mean_scan":
        return vmb.vmb_mean_scan_grouped_fwd(*args, H, W, case["groups"], want_ybar=True)
    y, saved, _ = vmb.vmb_mean_scan_train_fwd(*args, H, W, groups=case["groups"])
    g = vmb.vmb_mean_scan_bwd(*args, st["gy"], H, W, groups=case["groups"], saved=saved)
    return y, g["u"], g["delta"], g["A"], g["Bs"], g["Cs"], g["Dskip"], g["delta_bias"]


def work(case):
    """Inputs read once, outputs written once; per (b, k, d, l, n) one exponential and, per state, its product, the
    input term's product, the recurrence and the output sum (the channel-mean forms: the product and the sum)."""
    B, D, N, L, R = case["B"], case["D"], case["N"], case["H"] * case["W"], case["R"]
    s = 4 if case["dtype"] == "f32" else 2
    bdl, bkdl, bkl = B * D * L, B * K * D * L, B * K * L
    par = 4 * K * D * (N + 2)
    kind = case["kind"]
    full, mean = bkdl * (7 * N + 12), bkdl * (3 * N + 12)
    if kind == "full_map":
        return {"bytes": s * (2 * bdl + 2 * bkdl + 2 * bkl * N) + par, "flops": full + 3 * bdl}
    if kind == "mean_map":
        return {"bytes": s * (2 * bdl + bkdl + 2 * bkl * N) + 4 * bkl + par, "flops": mean + 8 * bdl}
    if kind == "full_scan":
        return {"bytes": s * (3 * bkdl + 2 * bkl * N) + par, "flops": full}
    if kind == "mean_scan":
        return {"bytes": s * (3 * bkdl + 2 * bkl * N) + 4 * bkl * case["groups"] + par, "flops": mean}
    if kind == "projected":
        weights = 4 * K * D * (2 * N + 2 * R)
        return {"bytes": s * (2 * bdl + bkdl + 2 * bkl * N) + 4 * bkl * R + weights + par,
                "flops": (full if case["path"] == "full" else mean) + 2 * bkdl * (2 * N + 2 * R)}
    # u, raw Delta, B, C and the output gradient read; y and the gradients written
    return {"bytes": s * (6 * bkdl + 4 * bkl * N) + 2 * par, "flops": mean + bkdl * (7 * N + 24)}


def tolerance(case):
    """About four times the distance from `exact` that was measured over these ranges: fp32 scans up to 1.1e-6; with the
    selection functions 6.4e-6 (768 channels summed by split tf32 products); bf16 1.9e-3 (the output's rounding), and
    4.4e-3 where B and C are rounded on the way."""
    if case["dtype"] == "bf16":
        return {"rel": 2e-2 if case["kind"] == "projected" else 8e-3}
    return {"rel": 2.5e-5 if case["kind"] == "projected" else 5e-6}


# ------------------------------------------------------------------ the same in 64 bits, plain torch


def _cross_scan64(x):
    B, D, H, W = x.shape
    rows, cols = x.reshape(B, D, H * W), x.transpose(2, 3).reshape(B, D, H * W)
    return torch.stack([rows, cols, rows.flip(-1), cols.flip(-1)], 1)


def _cross_merge64(y, H, W):
    B, _, D, L = y.shape
    rows = y[:, 0] + y[:, 2].flip(-1)
    cols = (y[:, 1] + y[:, 3].flip(-1)).reshape(B, D, W, H).transpose(2, 3).reshape(B, D, L)
    return (rows + cols).reshape(B, D, H, W)


def _discrete(u, raw, A, bias, lo, hi):
    """delta [B, K, D, T] and exp(delta A) [B, K, D, N, T] of the steps lo .. hi - 1."""
    D = u.shape[2]
    v = raw[..., lo:hi].double() + bias.double().view(1, K, D, 1)
    dl = torch.clamp(v, min=0.0) + torch.log1p(torch.exp(-v.abs()))
    return dl, torch.exp(dl.unsqueeze(3) * A.double().view(1, K, D, -1, 1))


def _steps(elements, L):
    return max(1, min(L, 120_000_000 // max(1, elements)))


def _full64(u, raw, A, Bs, Cs, Dskip, bias):
    B, _, D, L = u.shape
    N = Bs.shape[2]
    y = torch.empty(B, K, D, L, dtype=torch.float64, device=u.device)
    h = torch.zeros(B, K, D, N, dtype=torch.float64, device=u.device)
    T = _steps(B * K * D * N, L)
    for lo in range(0, L, T):
        hi = min(L, lo + T)
        dl, a = _discrete(u, raw, A, bias, lo, hi)
        uu = u[..., lo:hi].double()
        x = (dl * uu).unsqueeze(3) * Bs[..., lo:hi].double().unsqueeze(2)
        a, x = a.movedim(-1, 0).contiguous(), x.movedim(-1, 0).contiguous()
        for t in range(hi - lo):
            h = torch.addcmul(x[t], a[t], h)
            x[t] = h
        y[..., lo:hi] = torch.einsum("tbkdn,bknt->bkdt", x, Cs[..., lo:hi].double())
        y[..., lo:hi] += Dskip.double().view(1, K, D, 1) * uu
    return y


def _means64(u, raw, A, bias, G):
    """Group means of exp(delta A) [B, K, G, N, L] and of delta u [B, K, G, L]."""
    B, _, D, L = u.shape
    N = A.shape[1]
    am = torch.empty(B, K, G, N, L, dtype=torch.float64, device=u.device)
    sm = torch.empty(B, K, G, L, dtype=torch.float64, device=u.device)
    T = _steps(B * K * D * N, L)
    for lo in range(0, L, T):
        hi = min(L, lo + T)
        dl, a = _discrete(u, raw, A, bias, lo, hi)
        am[..., lo:hi] = a.view(B, K, G, D // G, N, hi - lo).mean(3)
        sm[..., lo:hi] = (dl * u[..., lo:hi].double()).view(B, K, G, D // G, hi - lo).mean(3)
    return am, sm


def _states64(am, x, reverse=False):
    """h(t) = am(t) h(t - 1) + x(t) over the last axis (reverse: h(t) = am(t + 1) h(t + 1) + x(t))."""
    L = am.shape[-1]
    a, h = am.movedim(-1, 0).contiguous(), x.movedim(-1, 0).clone(memory_format=torch.contiguous_format)
    if reverse:
        for t in range(L - 2, -1, -1):
            h[t] = torch.addcmul(h[t], a[t + 1], h[t + 1])
    else:
        for t in range(1, L):
            h[t] = torch.addcmul(h[t], a[t], h[t - 1])
    return h.movedim(0, -1)


def _mean64(u, raw, A, Bs, Cs, Dskip, bias, G=1):
    B, _, D, L = u.shape
    am, sm = _means64(u, raw, A, bias, G)
    h = _states64(am, Bs.double().unsqueeze(2) * sm.unsqueeze(3))
    ybar = (h * Cs.double().unsqueeze(2)).sum(3)
    y = ybar.repeat_interleave(D // G, 2) + Dskip.double().view(1, K, D, 1) * u.double()
    return y, ybar, am, sm, h


def _train64(st, G):
    u, raw, A, Bs, Cs, Dskip, bias, gy = (st[n] for n in ("u", "delta", "A", "Bs", "Cs", "Dskip", "bias", "gy"))
    B, _, D, L = u.shape
    N, M = A.shape[1], D // G
    y, _, am, sm, h = _mean64(u, raw, A, Bs, Cs, Dskip, bias, G)
    g = gy.double()
    gyb = g.view(B, K, G, M, L).sum(3)
    lam = _states64(am, Cs.double().unsqueeze(2) * gyb.unsqueeze(3), reverse=True)
    gC = (gyb.unsqueeze(3) * h).sum(2)
    gB = (lam * sm.unsqueeze(3)).sum(2)
    prev = torch.zeros_like(h)
    prev[..., 1:] = h[..., :-1]
    ga, gs = lam * prev / M, (lam * Bs.double().unsqueeze(2)).sum(3) / M
    gu = torch.empty(B, K, D, L, dtype=torch.float64, device=u.device)
    graw = torch.empty_like(gu)
    gA = torch.zeros(K, D, N, dtype=torch.float64, device=u.device)
    A64 = A.double().view(1, K, D, N, 1)
    T = _steps(2 * B * K * D * N, L)
    for lo in range(0, L, T):
        hi = min(L, lo + T)
        dl, a = _discrete(u, raw, A, bias, lo, hi)
        w = ga[..., lo:hi].repeat_interleave(M, 2) * a  # [B, K, D, N, T]
        gsd = gs[..., lo:hi].repeat_interleave(M, 2)
        gA += (w * dl.unsqueeze(3)).sum((0, 4))
        gdl = gsd * u[..., lo:hi].double() + (w * A64).sum(3)
        v = raw[..., lo:hi].double() + bias.double().view(1, K, D, 1)
        graw[..., lo:hi] = gdl * torch.sigmoid(v)
        gu[..., lo:hi] = Dskip.double().view(1, K, D, 1) * g[..., lo:hi] + gsd * dl
    return (y, gu, graw, gA.reshape(K * D, N), gB, gC, (g * u.double()).sum((0, 3)).reshape(-1),
            graw.sum((0, 3)).reshape(-1))


def exact(case, seed):
    st = prepare(case, seed)
    H, W, kind = case["H"], case["W"], case["kind"]
    if kind == "train":
        return _train64(st, case["groups"])
    u = st["u"] if "u" in st else _cross_scan64(st["x"])
    par = (st["Dskip"], st["bias"])
    if kind == "projected":
        u64 = u.double()
        Bs, Cs, z = (torch.einsum("knd,bkdl->bknl", st[n].double(), u64) for n in ("WB", "WC", "Wz"))
        raw = torch.einsum("kdr,bkrl->bkdl", st["Wup"].double(), z)
        y = _full64(u, raw, st["A"], Bs, Cs, *par) if case["path"] == "full" else _mean64(u, raw, st["A"], Bs, Cs, *par)[0]
        return _cross_merge64(y, H, W), y, z, Bs, Cs
    args = (u, st["delta"], st["A"], st["Bs"], st["Cs"], *par)
    if kind in ("full_map", "full_scan"):
        y = _full64(*args)
        return y if kind == "full_scan" else (_cross_merge64(y, H, W), y)
    y, ybar = _mean64(*args, case["groups"])[:2]
    if kind == "mean_scan":
        return y, ybar
    return _cross_merge64(y, H, W), ybar.view(case["B"], K, H * W)
