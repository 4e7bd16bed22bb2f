"""The calls a user of the SGM library makes, as measurable cases.

Every case is one call (or one set of calls) of the public Python binding on
synthetic rectified pairs: smoothed random texture, a background disparity
with random rectangles in front of it, and Gaussian noise on the right image.
Sizes, disparity counts, path counts and penalties are those of the
repository's workloads (320x240, 640x480, 1242x375 and 1920x1080 with D of 64,
128 and 256), of its tests (small and odd sizes, D that is no multiple of 64)
and of its allocation-free and batched forms.

Kinds of case ("op"):
  async   sgm_compute_async on device images, enqueued on torch's current stream
  host    Context.compute on pinned host images with a pinned host output
  ex      sgm_compute_ex_async with post-filters ("post"), uint16 output
  static  sgm_compute_static, the allocation-free form
  batch   sgm_compute_batch over "pairs" uneven pairs drawn from the pool
"""
import functools
import math
import random

import torch

from paper_1610_04121_gb300 import sgm

# The uneven batch's pool (sizes, D, paths).
POOL_SIZES = ((320, 240), (640, 480), (1242, 375), (1920, 1080))
POOL_DS = (64, 128, 256)
POOL_PATHS = (4, 8)

# Scratch of sgm_compute_static: what a problem may take.
STATIC_BYTES = 48 << 20

SUBPIXEL, LR_CHECK, ADAPTIVE_P2 = 1, 2, 4


def _case(name, op, W, H, D, paths, P1=7, P2=84, full=False, post=0):
    c = {"op": op, "W": W, "H": H, "D": D, "paths": paths, "P1": P1, "P2": P2, "full": full, "post": post}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a thumbnail or a region of interest: launches and latency count
        _case("roi_96x64_d64_p4", "async", 96, 64, 64, 4),
        # a small camera
        _case("qvga_320x240_d64_p4", "async", 320, 240, 64, 4),
        # the headline frame of the paper
        _case("vga_640x480_d128_p4", "async", 640, 480, 128, 4),
        # the same frame from and to host memory, as a camera loop hands it over
        _case("vga_host_640x480_d128_p4", "host", 640, 480, 128, 4),
        # the paper's cheapest configuration, two paths
        _case("vga_640x480_d128_p2", "async", 640, 480, 128, 2),
        # cropped images: odd sizes, D no multiple of 64, the full 9x7 Census
        _case("crop_641x479_d96_p4_full", "async", 641, 479, 96, 4, full=True),
        # driving scenes: wide and low, eight paths
        _case("road_1242x375_d128_p8", "async", 1242, 375, 128, 8, 10, 120),
        # HD with the largest disparity range
        _case("hd_1920x1080_d256_p4", "async", 1920, 1080, 256, 4),
        # HD at the paper's D with eight paths
        _case("hd_1920x1080_d128_p8", "async", 1920, 1080, 128, 8, 10, 120),
        # sub-pixel disparity with the left-right check and adaptive P2
        _case("vga_post_640x480_d128_p4", "ex", 640, 480, 128, 4, post=SUBPIXEL | LR_CHECK | ADAPTIVE_P2),
        # an embedding runtime that may not allocate
        _case("static_320x240_d64_p8", "static", 320, 240, 64, 8, 10, 120),
        # offline processing of uneven pairs
        {"name": "batch_12_pool", "op": "batch", "pairs": 12, "pool": 3, "area": 1 << 21},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _static_bytes(W, H, D, paths):
    return W * H * (9 + (3 if paths == 2 else 4) * D) + 4096


def draw(rng):
    op = rng.choice(("async", "async", "async", "async", "host", "ex", "static", "batch"))
    if op == "batch":
        return {"op": op, "pairs": rng.randint(2, 10), "pool": rng.randrange(1 << 20), "area": 1 << 19}
    while True:
        W, H = _log_int(rng, 64, 1920), _log_int(rng, 48, 1080)
        D, paths = 32 * rng.randint(1, 8), rng.choice((2, 4, 4, 8, 8))
        P1, P2 = rng.choice(((7, 84), (10, 120)))
        if not 0.5 <= W / H <= 5:
            continue
        if op == "static" and _static_bytes(W, H, D, paths) > STATIC_BYTES:
            continue
        post = rng.randint(1, 7) if op == "ex" else 0
        if W * H * D * paths * (2 if post & LR_CHECK else 1) <= 1920 * 1080 * 128 * 8:
            return _case(None, op, W, H, D, paths, P1, P2, full=op in ("async", "host") and rng.random() < 0.25, post=post)


def _pairs(case):
    """The (W, H, D, paths, P1, P2) of every pair of a case."""
    if case["op"] != "batch":
        return [tuple(case[k] for k in ("W", "H", "D", "paths", "P1", "P2"))]
    rng = random.Random(case["pool"])
    sizes = [s for s in POOL_SIZES if s[0] * s[1] <= case["area"]]
    return [(*rng.choice(sizes), rng.choice(POOL_DS), rng.choice(POOL_PATHS), 7, 84) for _ in range(case["pairs"])]


def _images(W, H, D, seed):
    """A rectified pair (uint8, on the host) from the seed alone."""
    g = torch.Generator().manual_seed(seed)
    wide = torch.randint(0, 256, (H + 2, W + D + 2), generator=g, dtype=torch.uint8).to(torch.int32)
    rows = wide[:, :-2] + wide[:, 1:-1] + wide[:, 2:]
    scene = (rows[:-2] + rows[1:-1] + rows[2:] + 4) // 9  # [H, W + D]
    disp = torch.full((H, W), min(10, D - 1), dtype=torch.int64)
    for _ in range(12):
        w, h = (int(torch.randint(max(1, n // 10), max(2, n // 3), (1,), generator=g)) for n in (W, H))
        x, y = (int(torch.randint(0, n, (1,), generator=g)) for n in (W - w + 1, H - h + 1))
        disp[y:y + h, x:x + w] = int(torch.randint(2, max(3, D - 8), (1,), generator=g))
    # right[y, x] shows the scene at x, left[y, x] at x - disp (D columns of margin on the left)
    left = torch.gather(scene, 1, torch.arange(W).expand(H, W) + D - disp)
    right = scene[:, D:] + torch.round(2.0 * torch.randn((H, W), generator=g)).to(torch.int32)
    return left.to(torch.uint8).contiguous(), right.clamp(0, 255).to(torch.uint8).contiguous()


@functools.lru_cache(maxsize=None)
def _context(full):
    """The context a program keeps for its life, on torch's current stream."""
    ctx = sgm.Context(0, flags=sgm.SGM_FLAG_CENSUS_FULL if full else 0)
    sgm.sgm_set_stream(ctx.handle, torch.cuda.current_stream())
    return ctx


def prepare(case, seed):
    op, jobs = case["op"], []
    for i, (W, H, D, paths, P1, P2) in enumerate(_pairs(case)):
        left, right = _images(W, H, D, seed * 1009 + i)
        if op == "host":
            left, right = left.pin_memory(), right.pin_memory()
            out = torch.zeros((H, W), dtype=torch.uint8).pin_memory()
        else:
            left, right = left.cuda(), right.cuda()
            out = torch.zeros((H, W), dtype=torch.int16 if op == "ex" else torch.uint8, device="cuda")
        jobs.append((left, right, out, W, H, D, P1, P2, paths))
    ctx = None if op == "static" else _context(bool(case.get("full")))
    return {"op": op, "ctx": ctx, "jobs": jobs, "post": case.get("post", 0)}


def run(state):
    op, jobs = state["op"], state["jobs"]
    if op == "batch":
        sgm.sgm_compute_batch(state["ctx"].handle, jobs)
        return [j[2] for j in jobs]
    left, right, out, W, H, D, P1, P2, paths = jobs[0]
    if op == "async":
        sgm.sgm_compute_async(state["ctx"].handle, left, right, W, H, D, P1, P2, paths, out)
    elif op == "host":
        state["ctx"].compute(left, right, D, P1, P2, paths, out)
    elif op == "ex":
        sgm.sgm_compute_ex_async(state["ctx"].handle, left, right, W, H, D, P1, P2, paths, state["post"], out)
    else:
        sgm.sgm_compute_static(left, right, W, H, D, P1, P2, paths, out, torch.cuda.current_stream())
    return out


def work(case):
    """Both images read and the disparity written once; per disparity and path
    the eight integer operations of the recursion, plus the sums and the
    minimum, twice with the left-right check."""
    nbytes = ops = 0
    post = case.get("post", 0)
    for W, H, D, paths, _, _ in _pairs(case):
        nbytes += W * H * (4 if case["op"] == "ex" else 3)
        ops += W * H * D * (9 * paths + 2) * (2 if post & LR_CHECK else 1)
    return {"bytes": nbytes, "flops": ops}


# ---------------------------------------------------------------------------
# The same results by plain torch in 64-bit integers.
# ---------------------------------------------------------------------------
def _census(img, full):
    """9x7 features of a [H, W] int64 image, 0 where the window leaves it: the
    center-symmetric comparisons, or every window pixel against the centre."""
    H, W = img.shape
    f = torch.zeros_like(img)
    if W < 9 or H < 7:
        return f
    at = lambda i, j: img[3 + j:H - 3 + j, 4 + i:W - 4 + i]  # noqa: E731
    if full:
        bits = [at(i, j) >= at(0, 0) for j in range(-3, 4) for i in range(-4, 5) if (i, j) != (0, 0)]
    else:
        bits = [at(i, j) >= at(-i, -j) for i in range(1, 5) for j in range(-3, 4)]
        bits += [at(0, j) >= at(0, -j) for j in range(1, 4)]
    for k, b in enumerate(bits):
        f[3:H - 3, 4:W - 4] |= b.to(torch.int64) << k
    return f


def _popcount(v):
    v = v - ((v >> 1) & 0x5555555555555555)
    v = (v & 0x3333333333333333) + ((v >> 2) & 0x3333333333333333)
    v = (v + (v >> 4)) & 0x0F0F0F0F0F0F0F0F
    return (v * 0x0101010101010101) >> 56


def _costs(left, right, D, full):
    fb, fm = _census(left, full), _census(right, full)
    H, W = left.shape
    mc = torch.empty((H, W, D), dtype=torch.int64, device=left.device)
    for d in range(D):
        m = torch.zeros_like(fm)
        if d < W:
            m[:, d:] = fm[:, :W - d]
        mc[:, :, d] = _popcount(fb ^ m)
    return mc


def _add_path(S, mc, img, P1, P2, adaptive, dx, dy):
    """S += the aggregated costs of the direction (dx, dy)."""
    H, W, D = mc.shape
    if dy == 0:  # rows walked side by side: transpose to a walk along the first axis
        S, mc, img = S.transpose(0, 1), mc.transpose(0, 1), img.transpose(0, 1)
        dx, dy = 0, dx
    n, across = mc.shape[:2]
    order = range(n) if dy > 0 else range(n - 1, -1, -1)
    prev = prev_img = None
    for y in order:
        L = mc[y].clone()
        if prev is not None:
            lo, hi = max(0, dx), across + min(0, dx)  # pixels with a predecessor
            q = prev[lo - dx:hi - dx]
            p2 = torch.full((hi - lo, 1), P2, dtype=torch.int64, device=mc.device)
            if adaptive:
                step = (img[y, lo:hi] - prev_img[lo - dx:hi - dx]).abs()
                p2 = torch.clamp(P2 // (1 + step), min=P1)[:, None]
            m = q.min(dim=1, keepdim=True).values
            best = torch.minimum(q, m + p2)
            best[:, 1:] = torch.minimum(best[:, 1:], q[:, :-1] + P1)
            best[:, :-1] = torch.minimum(best[:, :-1], q[:, 1:] + P1)
            L[lo:hi] += best - m
        S[y] += L
        prev, prev_img = L, img[y]


def _match(left, right, D, P1, P2, paths, full, adaptive):
    """The summed costs and the winner (the lowest disparity among equals)."""
    mc = _costs(left, right, D, full)
    S = torch.zeros_like(mc)
    ways = {2: ((1, 0), (0, 1)), 4: ((1, 0), (-1, 0), (0, 1), (0, -1))}
    ways[8] = ways[4] + ((1, 1), (-1, -1), (1, -1), (-1, 1))
    for dx, dy in ways[paths]:
        _add_path(S, mc, left, P1, P2, adaptive, dx, dy)
    d = torch.arange(D, device=mc.device)
    for y in range(S.shape[0]):  # keys S * D + d, a row at a time
        mc[y] = S[y] * D + d
    return S, mc.min(dim=2).values % D


def _median(v):
    H, W = v.shape
    out = v.clone()
    if H >= 3 and W >= 3:
        nine = torch.stack([v[j:H - 2 + j, i:W - 2 + i] for j in range(3) for i in range(3)])
        out[1:-1, 1:-1] = nine.sort(dim=0).values[4]
    return out


def _exact_one(left, right, W, H, D, paths, P1, P2, full, post, ex):
    S, d = _match(left, right, D, P1, P2, paths, full, bool(post & ADAPTIVE_P2))
    if not ex:
        return _median(d)
    v = 16 * d
    if post & SUBPIXEL:
        s0, sm, sp = (torch.gather(S, 2, (d + k).clamp(0, D - 1)[:, :, None])[:, :, 0] for k in (0, -1, 1))
        den = sm + sp - 2 * s0
        off = torch.div(16 * (sm - sp) + den, (2 * den).clamp(min=1), rounding_mode="floor")
        v = torch.where((d > 0) & (d < D - 1), v + off, v)
    v = _median(v)
    if post & LR_CHECK:
        del S
        dr = _match(right.flip(1), left.flip(1), D, P1, P2, paths, full, bool(post & ADAPTIVE_P2))[1].flip(1)
        x = torch.arange(W, device=d.device).expand(H, W) - d
        ok = (x >= 0) & ((d - torch.gather(dr, 1, x.clamp(min=0))).abs() <= 1)
        v = torch.where(ok, v, torch.full_like(v, -1))  # 0xFFFF
    return v


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    pairs = _pairs(case)
    if sum(W * H * D * paths for W, H, D, paths, _, _ in pairs) > (1 << 30 if device == "cuda" else 1 << 28):
        return None
    outs = []
    for i, (W, H, D, paths, P1, P2) in enumerate(pairs):
        left, right = (t.to(device, torch.int64) for t in _images(W, H, D, seed * 1009 + i))
        v = _exact_one(left, right, W, H, D, paths, P1, P2, bool(case.get("full")), case.get("post", 0),
                       case["op"] == "ex")
        outs.append(v)
    return outs if case["op"] == "batch" else outs[0]
