"""Performance cases of the SGM stereo library: what its users run, through its public entry points.

A case is one call: a single pair (device, host or raw images; integer or sub-pixel map; census or
NCC cost; approximate or exact left-right check; with a context or on the fixed scratch array) or
a batch of pairs of even or uneven sizes. Sizes, windows, penalties and path counts are those of
the repository's scenes, tests, benchmark and serving mix, and generic odd ones. Inputs are seeded
synthetic pairs made on the GPU: a textured scene with a ground plane, slanted surfaces and
occlusions whose disparities span the searched range, sensor noise on the right image.

Every result but the sub-pixel map is a map of whole numbers that follows from integer arithmetic,
so it has to be equal. The sub-pixel map takes one fp32 division and addition per pixel.
"""
from __future__ import annotations

import math

import torch

from paper_2106_07927_gb300 import binding

INVALID = 0xFFFF
MAX_DE = 3840 * 2160 * 256  # disparity estimates of the largest pair
STATIC_BYTES = binding.RES2TAC_STATIC_SCRATCH_BYTES
LR_MEDIAN = binding.RES2TAC_LR_CHECK | binding.RES2TAC_MEDIAN
# The batch and serving workloads' sizes.
WIDTHS, HEIGHTS, DISPS = (320, 640, 1024, 1242, 1920), (240, 375, 512, 768, 1080), (64, 128, 256)


def _case(name, call, W, H, D, cw=9, ch=7, p1=10, p2=120, paths=8, flags=LR_MEDIAN, pairs=1,
          uneven=False, mix=0):
    """call: device | host | static | raw | subpixel | batch. A batch has `pairs` pairs of W x H,
    D, or (uneven) of sizes drawn from the batch workload's lists with the seed `mix`."""
    return dict(name=name, call=call, W=W, H=H, D=D, cw=cw, ch=ch, p1=p1, p2=p2, paths=paths,
                flags=flags, pairs=pairs, uneven=uneven, mix=mix)


def listed():
    return [
        # The paper's embedded setting: a small frame, 5x5 census, 4 paths, no post-processing.
        # A frame is some 50 microseconds: launches and chain latency.
        _case("small_320x240_d64_4paths", "device", 320, 240, 64, 5, 5, 10, 120, 4, 0),
        # An onboard loop that may not allocate: an odd small frame on the fixed scratch array.
        _case("static_413x307_d48", "static", 413, 307, 48),
        # The benchmark's pair (KITTI-sized frame), all 8 paths, check and median.
        _case("road_1242x375_d128", "device", 1242, 375, 128),
        # Host buffers in, host map out: the end-to-end call on the aerial workload's shape.
        _case("host_1024x768_d128", "host", 1024, 768, 128, p1=8, p2=96),
        # A ragged shape: odd width and height, a disparity count that fills no power of two.
        _case("ragged_803x601_d144_5x5", "device", 803, 601, 144, 5, 5, 7, 86),
        # Full HD at the largest disparity range.
        _case("hd_1920x1080_d256", "device", 1920, 1080, 256),
        # The largest request of the serving mix.
        _case("uhd_3840x2160_d256", "device", 3840, 2160, 256),
        # Sub-pixel refinement ("fine") of the benchmark's pair.
        _case("subpixel_1242x375_d128", "subpixel", 1242, 375, 128),
        # From raw camera images: rectification, then the exact left-right check (two matchings).
        _case("raw_exact_1242x375_d128", "raw", 1242, 375, 128,
              flags=LR_MEDIAN | binding.RES2TAC_EXACT_CC),
        # NCC cost with the paper's NCC penalties (large P2).
        _case("ncc9_1242x375_d128", "device", 1242, 375, 128, 9, 9, 90, 880,
              flags=LR_MEDIAN | binding.RES2TAC_NCC),
        # Batch of many small equal frames (a camera array, a replayed sequence).
        _case("batch64_320x240_d64", "batch", 320, 240, 64, pairs=64),
        # Batch of uneven pairs, as the serving loop forms them.
        _case("batch16_uneven", "batch", 1920, 1080, 256, pairs=16, uneven=True, mix=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _draw(rng)
    del case["name"]
    return case


def _draw(rng):
    call = rng.choice(["device", "device", "device", "host", "static", "raw", "subpixel", "ncc",
                       "batch", "batch"])
    cw, ch = rng.choice([(9, 7), (9, 7), (5, 5)])
    p1 = rng.randint(4, 24)
    p2 = rng.randint(max(48, p1), 240)
    paths = rng.choice([8, 8, 8, 4])
    flags = rng.choice([LR_MEDIAN, LR_MEDIAN, binding.RES2TAC_LR_CHECK, 0])
    if call == "batch":
        if rng.random() < 0.5:
            return _case("", "batch", 1920, 1080, 256, cw, ch, p1, p2, paths, flags,
                         pairs=rng.randint(2, 16), uneven=True, mix=rng.randint(0, 1 << 20))
        W, H, D = _log(rng, 160, 1300), _log(rng, 120, 800), 16 * rng.randint(2, 8)
        n = max(2, min(64, _log(rng, 2, 64), MAX_DE // 2 // (W * H * D)))
        return _case("", "batch", W, H, D, cw, ch, p1, p2, paths, flags, pairs=n)
    most = MAX_DE // 4 if call in ("raw", "ncc") else MAX_DE
    while True:
        W, H, D = _log(rng, 160, 3840), _log(rng, 120, 2160), 16 * rng.randint(1, 16)
        if W * H * D <= most and (call != "static" or W * H * (3 * D + 25) + 4096 <= STATIC_BYTES):
            break
    if call == "ncc":
        n = rng.choice([5, 9])
        return _case("", "device", W, H, D, n, n, rng.randint(40, 120), rng.randint(400, 1200),
                     paths, flags | binding.RES2TAC_NCC)
    if call == "raw" and flags and rng.random() < 0.5:
        flags |= binding.RES2TAC_EXACT_CC
    return _case("", call, W, H, D, cw, ch, p1, p2, paths, flags)


# ------------------------------------------------------------------------------- inputs
def _sizes(case):
    """(W, H, D) of every pair."""
    if case["uneven"]:
        import random
        r = random.Random(case["mix"])
        return [(r.choice(WIDTHS), r.choice(HEIGHTS), r.choice(DISPS))
                for _ in range(case["pairs"])]
    return [(case["W"], case["H"], case["D"])] * case["pairs"]


def _scene(gen, n, W, H, D):
    """n rectified pairs: uint8 [n, H, W] left and right images."""
    dev = "cuda"
    img = torch.zeros(n, 1, H, W, device=dev)
    amp, cell = 1.0, 24
    for _ in range(4):  # four octaves of value noise
        g = torch.rand(n, 1, H // cell + 2, W // cell + 2, generator=gen, device=dev)
        img += amp * torch.nn.functional.interpolate(g, size=(H, W), mode="bilinear",
                                                     align_corners=True)
        amp, cell = amp / 2, max(cell // 2, 1)
    lo, hi = img.amin((1, 2, 3), True), img.amax((1, 2, 3), True)
    left = ((img - lo) / (hi - lo).clamp_min(1e-6) * 255).round()[:, 0]
    # ground plane rising towards the bottom, and slanted boxes in front of it
    yy = torch.arange(H, device=dev).view(1, H, 1)
    xx = torch.arange(W, device=dev).view(1, 1, W)
    disp = (110 * yy / max(H - 1, 1)).expand(n, H, W).clone()
    for _ in range(20):
        u = torch.rand(n, 7, generator=gen, device=dev).view(n, 7, 1, 1)
        dx, dy = xx - u[:, 0] * W, yy - u[:, 1] * H
        inside = (dx.abs() <= W / 30 + u[:, 2] * W / 8) & (dy.abs() <= H / 20 + u[:, 3] * H / 5)
        plane = 2 + 118 * u[:, 4] + 0.4 * (u[:, 5] - 0.5) * dx + 0.4 * (u[:, 6] - 0.5) * dy
        disp = torch.where(inside, torch.maximum(disp, plane), disp)
    disp = (disp * D / 128).round().clamp(0, D - 1).long()
    # R(x - d) = L(x), the nearest surface in front; holes get noise
    tgt = xx - disp
    row = torch.arange(n * H, device=dev).view(n, H, 1) * W
    ok = tgt >= 0
    key = torch.full((n * H * W,), -1, dtype=torch.int64, device=dev)
    key.scatter_reduce_(0, (row + tgt)[ok], (disp * 256 + left.long())[ok], "amax")
    noise = torch.randint(0, 256, key.shape, generator=gen, device=dev)
    right = torch.where(key < 0, noise, key % 256).view(n, H, W).float()
    right = (right + 3 * torch.randn(right.shape, generator=gen, device=dev)).round()
    return left.to(torch.uint8), right.clamp(0, 255).to(torch.uint8)


def _inputs(case, seed):
    """[(left, right)] of every pair, equal sizes made together."""
    gen = torch.Generator("cuda").manual_seed(seed)
    sizes = _sizes(case)
    out = [None] * len(sizes)
    for s in sorted(set(sizes)):
        at = [i for i, t in enumerate(sizes) if t == s]
        left, right = _scene(gen, len(at), *s)
        for k, i in enumerate(at):
            out[i] = (left[k], right[k])
    return out


def _maps(case, seed):
    """Rectification maps of both cameras, float32 [H, W]: a small rotation, shift and radial
    distortion, as a calibration gives them."""
    W, H = case["W"], case["H"]
    gen = torch.Generator("cpu").manual_seed(seed)
    f = 0.9 * max(W, H)
    y, x = torch.meshgrid(torch.arange(H, dtype=torch.float64, device="cuda"),
                          torch.arange(W, dtype=torch.float64, device="cuda"), indexing="ij")
    xn, yn = (x - (W - 1) / 2) / f, (y - (H - 1) / 2) / f
    r2 = ((W / 2 / f) ** 2 + (H / 2 / f) ** 2)
    maps = []
    for _ in range(2):
        u = (2 * torch.rand(4, generator=gen) - 1).tolist()
        c, s = math.cos(u[0] * math.pi / 180), math.sin(u[0] * math.pi / 180)
        xr, yr = c * xn - s * yn, s * xn + c * yn
        k = 1 + 0.08 * u[1] * (xr * xr + yr * yr) / r2
        maps += [(f * xr * k + (W - 1) / 2 + 1.5 * u[2]).float().contiguous(),
                 (f * yr * k + (H - 1) / 2 + 1.5 * u[3]).float().contiguous()]
    return maps


def _params(case, W, H, D):
    return binding.make_params(W, H, D, case["cw"], case["ch"], case["p1"], case["p2"],
                               case["paths"], case["flags"])


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.call = case["call"]
    st.images = _inputs(case, seed)
    W, H, D = case["W"], case["H"], case["D"]
    if st.call == "batch":
        st.ctx = binding.Stereo(_params(case, 64, 64, 64))
        st.out = [torch.empty(t[0].shape, dtype=torch.int16, device="cuda") for t in st.images]
        st.pairs = [binding.res2tac_pair(a.data_ptr(), b.data_ptr(), a.stride(0), o.data_ptr(),
                                         2 * o.stride(0), w, h, d, 0)
                    for (a, b), o, (w, h, d) in zip(st.images, st.out, _sizes(case))]
        prm = _params(case, 64, 64, 64)
        binding.res2tac_batch_reserve(st.ctx.handle,
                                      binding.res2tac_batch_workspace_bytes(prm, st.pairs),
                                      len(st.pairs))
        return st
    st.left, st.right = st.images[0]
    st.params = _params(case, W, H, D)
    if st.call == "host":
        st.left, st.right = st.left.cpu().pin_memory(), st.right.cpu().pin_memory()
        st.out = torch.empty(H, W, dtype=torch.int16).pin_memory()
    elif st.call == "subpixel":
        st.out = torch.empty(H, W, dtype=torch.float32, device="cuda")
    else:
        st.out = torch.empty(H, W, dtype=torch.int16, device="cuda")
    if st.call != "static":
        st.ctx = binding.Stereo(st.params)
    if st.call == "raw":
        m = _maps(case, seed)
        binding.res2tac_set_rectification(st.ctx.handle, m[0].data_ptr(), m[1].data_ptr(),
                                          m[2].data_ptr(), m[3].data_ptr(), 4 * W, W, H,
                                          torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()  # the context has its own copy of the maps from here on
    return st


def run(st):
    if st.call == "device":
        return st.ctx.compute(st.left, st.right, st.out)
    if st.call == "subpixel":
        return st.ctx.compute_subpixel(st.left, st.right, st.out)
    stream = torch.cuda.current_stream().cuda_stream
    if st.call == "batch":
        binding.res2tac_compute_batch(st.ctx.handle, st.pairs, stream)
        return st.out
    W = st.params.width
    a, b, o = st.left.data_ptr(), st.right.data_ptr(), st.out.data_ptr()
    if st.call == "host":
        binding.res2tac_compute_host(st.ctx.handle, a, b, W, o, 2 * W, stream)
    elif st.call == "raw":
        binding.res2tac_compute_raw(st.ctx.handle, a, b, W, o, 2 * W, stream)
    else:
        binding.res2tac_compute_static(st.params, a, b, W, o, 2 * W, stream)
    return st.out


def work(case):
    """Both images read and the map written once (the rectification's maps too). Operations: per
    disparity estimate the cost (XOR and count) and, per path, the 9 additions and minima of the
    recurrence and its sum; the selection of both maps; per pixel the census or the patch
    statistics and the median. Counted once more for the exact check's second matching."""
    nbytes = ops = 0
    n = case["cw"] * case["ch"] - 1
    for W, H, D in _sizes(case):
        px = W * H
        nbytes += px * (2 + (4 if case["call"] == "subpixel" else 2) +
                        (16 if case["call"] == "raw" else 0))
        per = px * D * (2 + 9 * case["paths"] + 2) + px * 2 * n
        if case["flags"] & binding.RES2TAC_NCC:  # sliding row sums: n products per estimate
            per += px * D * 2 * case["cw"]
        ops += per * (2 if case["flags"] & binding.RES2TAC_EXACT_CC else 1)
        if case["flags"] & binding.RES2TAC_MEDIAN:
            ops += px * 40
    return {"bytes": nbytes, "flops": ops}


def tolerance(case):
    if case["call"] == "subpixel":
        # one fp32 division and one addition at up to 256: half an ulp each (measured against
        # fp64: rel 2.2e-8, max 4.5e-8); four times that
        return {"rel": 9e-8, "max": 1.8e-7}
    return "exact"


# ------------------------------------------------------------------------------- exact results
# The method in plain torch. Everything but the sub-pixel step is integer arithmetic far below
# 2^31, so 32-bit integers hold it exactly; the sub-pixel step and the NCC rounding take 64 bits.
def _shifted(a, dy, dx):
    """a(y + dy, x + dx) with zeros outside the image, over [n, H, W]."""
    H, W = a.shape[-2:]
    p = torch.nn.functional.pad(a, (max(-dx, 0), max(dx, 0), max(-dy, 0), max(dy, 0)))
    return p[..., max(dy, 0):max(dy, 0) + H, max(dx, 0):max(dx, 0) + W]


def _popcount(v):
    v = v - ((v >> 1) & 0x5555555555555555)
    v = (v & 0x3333333333333333) + ((v >> 2) & 0x3333333333333333)
    v = (v + (v >> 4)) & 0x0F0F0F0F0F0F0F0F
    v = v + (v >> 8)
    v = v + (v >> 16)
    return (v + (v >> 32)) & 0x7F


def _cost_census(a, b, D, cw, ch):
    def census(im):
        im = im.to(torch.int16)
        c = torch.zeros(im.shape, dtype=torch.int64, device=im.device)
        k = 0
        for j in range(-(ch // 2), ch // 2 + 1):
            for i in range(-(cw // 2), cw // 2 + 1):
                if i or j:
                    c |= (_shifted(im, j, i) < im).long() << k
                    k += 1
        return c
    ca, cb = census(a), census(b)
    n, H, W = a.shape
    C = torch.full((n, H, W, D), 255, dtype=torch.uint8, device=a.device)
    for d in range(min(D, W)):
        C[:, :, d:, d] = _popcount(ca[:, :, d:] ^ cb[:, :, :W - d]).to(torch.uint8)
    return C


def _cost_ncc(a, b, D, n):
    r, N = n // 2, n * n

    def box(v):  # zero-margin n x n sums of int64 [1, H, W']
        v = torch.nn.functional.pad(v, (r + 1, r, r + 1, r)).cumsum(-1)
        v = (v[..., n:] - v[..., :-n]).cumsum(-2)
        return v[..., n:, :] - v[..., :-n, :]
    a, b = a.long(), b.long()
    sa, sb = box(a), box(b)
    va, vb = (N * box(a * a) - sa * sa).double(), (N * box(b * b) - sb * sb).double()
    m, H, W = a.shape
    C = torch.full((m, H, W, D), 255, dtype=torch.uint8, device=a.device)
    for d in range(min(D, W)):
        # the patch around x - d of the right image: its columns move as one, margin included
        prod = torch.zeros_like(a)
        prod[:, :, d:] = a[:, :, d:] * b[:, :, :W - d]
        cov = N * box(prod) - sa * torch.nn.functional.pad(sb, (d, 0))[..., :W]
        v = va[..., d:] * vb[..., :W - d]
        cov = cov[..., d:].clamp_min(0).double()
        q = torch.where(v > 0, 255 * cov / v.clamp_min(1).sqrt(), torch.zeros_like(v))
        C[:, :, d:, d] = (255 - q.round().clamp_max(255)).to(torch.uint8)
    return C


def _sums(C, p1, p2, paths):
    """Sum of the path costs, int32 [n, H, W, D]."""
    n, H, W, D = C.shape
    S = torch.zeros(C.shape, dtype=torch.int32, device=C.device)
    big = 1 << 28

    def g(L):  # min over d' of L(d') + V, minus the least L
        m = L.amin(-1, keepdim=True)
        t = torch.minimum(L, m + p2)
        pad = torch.nn.functional.pad(L, (1, 1), value=big)
        return torch.minimum(t, torch.minimum(pad[..., :-2], pad[..., 2:]) + p1) - m
    dirs = [(0, 1), (0, -1), (1, 0), (-1, 0)]
    if paths == 8:
        dirs += [(1, 1), (-1, -1), (1, -1), (-1, 1)]
    for dy, dx in dirs:
        L = None
        for k in range(H if dy else W):
            if dy:
                y = k if dy > 0 else H - 1 - k
                cur, acc = C[:, y].int(), S[:, y]
                if L is not None:
                    q = g(L)
                    if dx > 0:
                        cur[:, 1:] += q[:, :-1]
                    elif dx < 0:
                        cur[:, :-1] += q[:, 1:]
                    else:
                        cur += q
            else:
                x = k if dx > 0 else W - 1 - k
                cur, acc = C[:, :, x].int(), S[:, :, x]
                if L is not None:
                    cur += g(L)
            acc += cur
            L = cur
    return S.clamp_max_(65535)


def _first_min(v):
    """Smallest index of the least value along the last dimension (values below 2^16)."""
    d = torch.arange(v.shape[-1], device=v.device, dtype=torch.int32)
    out = torch.empty(v.shape[:-1], dtype=torch.int32, device=v.device)
    for y in range(v.shape[1]):
        out[:, y] = ((v[:, y] << 8) | d).amin(-1) & 255
    return out


def _match(a, b, case, D):
    if case["flags"] & binding.RES2TAC_NCC:
        C = _cost_ncc(a, b, D, case["cw"])
    else:
        C = _cost_census(a, b, D, case["cw"], case["ch"])
    S = _sums(C, case["p1"], case["p2"], case["paths"])
    return S, _first_min(S)


def _median(v, inv):
    n, H, W = v.shape
    p = torch.nn.functional.pad(v, (1, 1, 1, 1), value=inv)
    nine = torch.stack([p[:, j:j + H, i:i + W] for j in range(3) for i in range(3)])
    return torch.where(v == inv, v, nine.sort(0).values[4])


def _exact_pairs(a, b, case, D):
    """Final maps of n pairs, uint8 [n, H, W] images: int16 bits, or fp64 for the sub-pixel map."""
    n, H, W = a.shape
    S, dl = _match(a, b, case, D)
    x = torch.arange(W, device=a.device, dtype=torch.int32)
    keep = torch.ones(dl.shape, dtype=torch.bool, device=a.device)
    if case["flags"] & binding.RES2TAC_LR_CHECK:
        if case["flags"] & binding.RES2TAC_EXACT_CC:
            dr = _match(b.flip(-1), a.flip(-1), case, D)[1].flip(-1)
        else:
            best = torch.full(dl.shape, 1 << 30, dtype=torch.int32, device=a.device)
            for d in range(min(D, W)):
                best[..., :W - d] = torch.minimum(best[..., :W - d], (S[:, :, d:, d] << 8) | d)
            dr = best & 255
        at = x - dl
        keep = (at >= 0) & ((dl - dr.gather(-1, at.clamp_min(0).long())).abs() <= 1)
    if case["call"] == "subpixel":
        i = dl.long().clamp(1, D - 2).unsqueeze(-1)
        s0, s1, s2 = (S.gather(-1, i + k).squeeze(-1).double() for k in (-1, 0, 1))
        edge = (dl < 1) | (dl > D - 2)
        v = dl.double() + torch.where(edge, 0.0, (s0 - s2) / (2 * (s0 - 2 * s1 + s2)).clamp_min(1))
        inv = math.inf
    else:
        v, inv = dl, INVALID
    v = torch.where(keep, v, torch.full_like(v, inv))
    if case["flags"] & binding.RES2TAC_MEDIAN:
        v = _median(v, inv)
    return v if case["call"] == "subpixel" else v.to(torch.int16)


def _rectify(raw, mapx, mapy):
    H, W = raw.shape
    X, Y = (mapx * 32).round().long(), (mapy * 32).round().long()
    x0, y0, fx, fy = X >> 5, Y >> 5, X & 31, Y & 31

    def at(y, x):
        ok = (x >= 0) & (x < W) & (y >= 0) & (y < H)
        return torch.where(ok, raw.long()[y.clamp(0, H - 1), x.clamp(0, W - 1)], 0)
    v = (at(y0, x0) * (32 - fx) * (32 - fy) + at(y0, x0 + 1) * fx * (32 - fy) +
         at(y0 + 1, x0) * (32 - fx) * fy + at(y0 + 1, x0 + 1) * fx * fy + 512) >> 10
    return v.to(torch.uint8)


def exact(case, seed):
    images, sizes = _inputs(case, seed), _sizes(case)
    if case["call"] == "raw":
        m = _maps(case, seed)
        a, b = images[0]
        images = [(_rectify(a, m[0], m[1]), _rectify(b, m[2], m[3]))]
    out = [None] * len(sizes)
    for s in sorted(set(sizes)):
        at = [i for i, t in enumerate(sizes) if t == s]
        group = max(1, (1 << 28) // (s[0] * s[1] * s[2]))  # pairs computed together
        for k in range(0, len(at), group):
            some = at[k:k + group]
            v = _exact_pairs(torch.stack([images[i][0] for i in some]),
                             torch.stack([images[i][1] for i in some]), case, s[2])
            for j, i in enumerate(some):
                out[i] = v[j]
    if case["call"] == "batch":
        return out
    return out[0].cpu() if case["call"] == "host" else out[0]
