"""The work that users of this library have it do, as cases to be timed.

listed() gives the cases, draw(rng) more of the same ranges.  Inputs are
synthetic plane scenes made on the GPU from the seed alone, after the recipe
of paper_2203_02300_gb300/scenes.py: textured surfaces from nearly flat to
busy (short and long support arms), slanted planes, sensor noise, a right
view with another gain and offset, occlusions filled with fresh texture.
"""
import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_2203_02300_gb300 import binding

# Sizes of the 32-pair batch of uneven shapes (tests and bench: the same four).
BATCH_SHAPES = ((320, 240, 32), (640, 480, 64), (960, 540, 128), (1280, 720, 128))
FOCAL_PX, BASELINE = 700.0, 0.12
# The largest listed single pair; a drawn one costs no more.
MOST = 1920 * 1080 * 256


def listed():
    return [
        # A thumbnail-sized pair: the smallest frame in use, all launch latency.
        {"name": "match_96x64_d16", "kind": "match", "W": 96, "H": 64, "D": 16},
        # QVGA frame, the plain single-pair path of a small camera.
        {"name": "match_320x240_d32", "kind": "match", "W": 320, "H": 240, "D": 32},
        # The headline workload: one VGA pair, both views and the consistency check.
        {"name": "match_640x480_d64", "kind": "match", "W": 640, "H": 480, "D": 64},
        # The same from the caller's pinned host buffers, as a capture loop calls it.
        {"name": "host_640x480_d64", "kind": "host", "W": 640, "H": 480, "D": 64},
        # Both views' maps and minimum costs of a ragged size (rectified crops), a
        # disparity count that fills no group of 32.
        {"name": "views_333x211_d50", "kind": "views", "W": 333, "H": 211, "D": 50},
        # The full quality setting: smoothed arms and two rounds of the Eq. 4 vote.
        {"name": "vote_640x480_d64", "kind": "match", "W": 640, "H": 480, "D": 64, "vote_iters": 2, "smooth_arms": 1},
        # The other aggregation order (vertical sums first).
        {"name": "vh_640x480_d64", "kind": "match", "W": 640, "H": 480, "D": 64, "agg_order": 1},
        # HD camera stream frame.
        {"name": "match_1280x720_d128", "kind": "match", "W": 1280, "H": 720, "D": 128},
        # The largest single pair: full HD with the widest disparity range.
        {"name": "match_1920x1080_d256", "kind": "match", "W": 1920, "H": 1080, "D": 256},
        # 32 uneven pairs in one call (offline processing of recordings).
        {"name": "batch_32_uneven", "kind": "batch", "W": 1280, "H": 720, "D": 128, "n": 32, "mix": 3},
        # Full-size sparse depth through the quarter-size input (the mixed reality frame).
        {"name": "depth_1280x720_d64", "kind": "depth", "W": 1280, "H": 720, "D": 64},
        # The Eq. 20 densification of such a depth map, of a first frame (no previous depth).
        {"name": "densify_1280x720", "kind": "densify", "W": 1280, "H": 720, "D": 64, "pre": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["match", "match", "match", "views", "host", "batch", "depth", "densify"])
    if kind == "batch":
        return {"kind": "batch", "W": 1280, "H": 720, "D": 128, "n": rng.randint(2, 24), "mix": rng.randint(4, 10 ** 6)}
    W = _log_int(rng, 96, 1920)
    H = max(64, min(1080, int(W * rng.uniform(0.5, 0.8))))
    D = min(_log_int(rng, 12, 256), W // 2)
    case = {"kind": kind, "W": W, "H": H, "D": D}
    if kind == "depth":
        case["D"] = min(D, 128, W // 4)
    elif kind == "densify":
        case["W"], case["H"], case["D"], case["pre"] = min(W, 1280), min(H, 720), min(D, 64), rng.randint(0, 1)
    elif kind in ("match", "views") and rng.random() < 0.5:
        option = rng.choice(["vote_iters", "smooth_arms", "agg_order", "d_min", "arm_l1"])
        if option == "d_min":
            case["d_min"] = rng.randint(1, max(1, min(256, W) - D)) // 2
        elif option == "arm_l1":
            case["arm_l1"], case["arm_l2"] = 17, 8
        else:
            case[option] = 1
    if case["W"] * case["H"] * case["D"] > MOST:
        case["D"] = 128
    return case


# ------------------------------------------------------------------ inputs
class _Maker:
    """Plane scenes on the GPU: pixel noise from a torch generator, geometry from `random`."""

    def __init__(self, seed):
        self.dev = torch.device("cuda:0")
        self.gen = torch.Generator(self.dev).manual_seed(seed)
        self.rng = random.Random(seed)
        k = torch.exp(-0.5 * torch.arange(-3, 4, device=self.dev, dtype=torch.float32) ** 2)
        self.blur = (k / k.sum()).view(1, 1, 7, 1)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.gen, device=self.dev)

    def texture(self, h, w):
        """(3, h, w) albedo of one surface: a base colour, smooth shading, fine
        texture of a contrast from nearly flat to busy."""
        base = torch.tensor([self.rng.uniform(40.0, 215.0) for _ in range(3)], device=self.dev).view(3, 1, 1)
        low = F.interpolate(self.normal(1, 3, h // 32 + 2, w // 32 + 2), size=(h, w), mode="bicubic",
                            align_corners=False)[0]
        fine = F.pad(self.normal(3, 1, h, w), (3, 3, 3, 3), mode="replicate")
        fine = F.conv2d(F.conv2d(fine, self.blur), self.blur.transpose(2, 3))[:, 0]
        contrast = self.rng.choice((2.0, 5.0, 12.0, 30.0))
        return base + low * (10.0 / (low.std() + 1e-6)) + fine * (contrast / (fine.std() + 1e-6))

    def scene(self, W, H, dlo, dhi, planes):
        """(left, right, disparity): uint8 (H, W, 3) views and the (H, W) ground truth."""
        rng, dev = self.rng, self.dev
        disp = torch.full((H, W), float(dlo), device=dev)
        left = self.texture(H, W)
        for _ in range(planes):
            w, h = rng.randint(max(4, W // 8), max(5, W // 2)), rng.randint(max(4, H // 8), max(5, H // 2))
            x0, y0 = rng.randint(-(w // 4), W - 3 * w // 4), rng.randint(-(h // 4), H - 3 * h // 4)
            c, a, b = rng.uniform(dlo, dhi), rng.uniform(-0.2, 0.2), rng.uniform(-0.2, 0.2)
            tex = self.texture(h, w)
            ax, ay, bx, by = max(0, x0), max(0, y0), min(W, x0 + w), min(H, y0 + h)
            xs = torch.arange(ax - x0, bx - x0, device=dev, dtype=torch.float32) - (w - 1) / 2
            ys = torch.arange(ay - y0, by - y0, device=dev, dtype=torch.float32) - (h - 1) / 2
            d = (c + a * xs[None, :] + b * ys[:, None]).clamp(dlo, dhi)
            win = d > disp[ay:by, ax:bx]
            disp[ay:by, ax:bx] = torch.where(win, d, disp[ay:by, ax:bx])
            left[:, ay:by, ax:bx] = torch.where(win, tex[:, ay - y0:by - y0, ax - x0:bx - x0], left[:, ay:by, ax:bx])
        # the right view: L(x, y) warped to (x - d, y), the nearer surface in front
        di = torch.round(disp).long()
        xs = torch.arange(W, device=dev)[None, :].expand(H, W)
        rows = torch.arange(H, device=dev)[:, None] * W
        ok = xs - di >= 0
        key = torch.full((H * W,), -1, dtype=torch.long, device=dev)
        key = key.scatter_reduce(0, (rows + xs - di)[ok], (di * W + xs)[ok], "amax")
        src = (rows + key.view(H, W).clamp(min=0) % W).view(-1)
        right = torch.where((key >= 0).view(1, H, W), left.reshape(3, -1)[:, src].view(3, H, W), self.texture(H, W))
        left = (left + 2.0 * self.normal(3, H, W)).round().clamp(0, 255)
        right = (right + 2.0 * self.normal(3, H, W)).round().clamp(0, 255)
        right = (1.03 * right + 5.0).round().clamp(0, 255)
        return tuple(t.permute(1, 2, 0).contiguous().to(torch.uint8) for t in (left, right)) + (disp,)


def _planes(case):
    return 32 if case["W"] * case["H"] >= 1920 * 1080 else 12


def _pair(case, seed, half=False):
    """The pair of a case; `half`: matched at half of each axis."""
    D = (2 if half else 1) * case["D"]
    dlo = case.get("d_min", 0) + 2
    return _Maker(seed).scene(case["W"], case["H"], dlo, max(dlo, case.get("d_min", 0) + D - 3), _planes(case))


def _batch_shapes(case):
    pick = random.Random(case["mix"])
    return [BATCH_SHAPES[pick.randrange(4)] for _ in range(case["n"])]


def _dense_inputs(case, seed):
    """Sparse depth (0 = missing), contour, fused flow magnitude and normalised edge
    strength, and the previous frame's depth, as the densification takes them."""
    W, H = case["W"], case["H"]
    m = _Maker(seed)
    left, _, disp = m.scene(W, H, 4.0, 2.0 * case["D"] - 8.0, 12)
    z = FOCAL_PX * BASELINE / disp
    # matched at half size, so known in 2x2 blocks; about a fifth is missing: scattered and in patches
    gone = (torch.rand(H // 2, W // 2, generator=m.gen, device=m.dev) < 0.06).float()
    patch = F.interpolate(m.normal(1, 1, H // 24 + 2, W // 24 + 2), size=(H // 2, W // 2), mode="bicubic",
                          align_corners=False)[0, 0]
    gone = (gone + (patch > 0.75).float() > 0).float()
    gone = F.pad(gone.repeat_interleave(2, 0).repeat_interleave(2, 1), (0, W % 2, 0, H % 2), value=1.0)
    sparse = torch.where(gone > 0, torch.zeros_like(z), z).contiguous()
    jump = torch.zeros((H, W), dtype=torch.bool, device=m.dev)
    jump[:, :-1] |= (disp[:, 1:] - disp[:, :-1]).abs() > 1
    jump[:-1] |= (disp[1:] - disp[:-1]).abs() > 1
    grey = left.float().mean(2)
    gx, gy = torch.zeros_like(grey), torch.zeros_like(grey)
    gx[:, 1:-1] = (grey[:, 2:] - grey[:, :-2]) / 2
    gy[1:-1] = (grey[2:] - grey[:-2]) / 2
    edge = torch.sqrt(gx * gx + gy * gy)
    edge = (edge / edge.max()).contiguous()
    fuse = torch.rand(H, W, generator=m.gen, device=m.dev)
    pre = (z * (1 + 0.01 * m.normal(H, W))).contiguous() if case["pre"] else None
    return sparse, jump.to(torch.uint8).contiguous(), fuse, edge, pre


def _params(case):
    over = {k: case[k] for k in ("vote_iters", "smooth_arms", "agg_order", "d_min", "arm_l1", "arm_l2") if k in case}
    return binding.Params.default(**over) if over else None


def prepare(case, seed):
    st = {"kind": case["kind"], "stereo": binding.Stereo(0), "D": case["D"], "params": _params(case)}
    W, H, kind = case["W"], case["H"], case["kind"]
    if kind == "batch":
        st["pairs"] = []
        for i, (w, h, d) in enumerate(_batch_shapes(case)):
            left, right, _ = _Maker(1000003 * seed + i).scene(w, h, 2, d - 2, 8)
            st["pairs"].append((left, right, d, torch.empty((h, w), dtype=torch.int16, device=left.device)))
        return st
    if kind == "densify":
        st["in"] = _dense_inputs(case, seed)
        st["out"] = torch.empty_like(st["in"][0])
        return st
    left, right, _ = _pair(case, seed, kind == "depth")
    if kind == "host":
        # pinned host frames and map, as a capture loop holds them
        keep = [left.cpu().pin_memory(), right.cpu().pin_memory(), torch.empty((H, W), dtype=torch.int16).pin_memory()]
        st["keep"], (st["left"], st["right"], st["out"]) = keep, [t.numpy() for t in keep]
        return st
    st["left"], st["right"] = left, right
    if kind == "match":
        st["out"] = torch.empty((H, W), dtype=torch.int16, device=left.device)
    elif kind == "depth":
        st["out"] = torch.empty((H, W), dtype=torch.float32, device=left.device)
        st["half"] = torch.empty((H // 2, W // 2), dtype=torch.int16, device=left.device)
    return st


def run(st):
    h, kind = st["stereo"], st["kind"]
    if kind == "match":
        return h.match(st["left"], st["right"], st["D"], st["params"], st["out"])
    if kind == "views":
        return h.match_views(st["left"], st["right"], st["D"], st["params"])
    if kind == "host":
        return h.match_host(st["left"], st["right"], st["D"], st["params"], st["out"])
    if kind == "batch":
        h.match_batch(st["pairs"])
        return [p[3] for p in st["pairs"]]
    if kind == "depth":
        return h.depth(st["left"], st["right"], st["D"], FOCAL_PX, BASELINE, st["params"], st["out"], st["half"]), st["half"]
    sparse, contour, fuse, edge, pre = st["in"]
    return h.densify(sparse, contour, fuse, edge, pre, None, st["out"])


# Operations per pixel and disparity of one reference view that the method
# cannot do without: two 32-bit differences and bit counts and their sum, the
# three channel differences and their sum, the two exponential terms weighted
# and added (Eq. 1), two 1-D sums as one addition and one subtraction each
# (Eq. 2), the comparison (Eq. 3).
OPS_PER_EVALUATION = 18
# Multiplications and additions per pixel and conjugate-gradient iteration of
# the five-point system, and iterations to the default tolerance without and
# with a previous depth map.
OPS_PER_CG_STEP, CG_STEPS = 20, (200, 50)


def work(case):
    W, H, D = case["W"], case["H"], case["D"]
    kind = case["kind"]
    if kind == "batch":
        shapes = _batch_shapes(case)
        return {"bytes": sum(8 * w * h for w, h, _ in shapes),
                "flops": sum(2 * OPS_PER_EVALUATION * w * h * d for w, h, d in shapes)}
    if kind == "densify":
        return {"bytes": (17 + 4 * case["pre"]) * W * H, "flops": OPS_PER_CG_STEP * CG_STEPS[case["pre"]] * W * H}
    if kind == "depth":
        return {"bytes": (6 + 4) * W * H + W * H // 2, "flops": 2 * OPS_PER_EVALUATION * (W // 2) * (H // 2) * D}
    out = 14 if kind == "views" else 2
    return {"bytes": (6 + out) * W * H, "flops": 2 * OPS_PER_EVALUATION * W * H * D}


# ------------------------------------------------- the same in 64 bits
def _census(img):
    """(H, W, 3) uint8 -> 62-bit census strings of the grey level, 9 x 7 window."""
    c = img.long()
    y = (77 * c[..., 0] + 150 * c[..., 1] + 29 * c[..., 2] + 128) >> 8
    H, W = y.shape
    pad = F.pad(y[None, None].double(), (4, 4, 3, 3), mode="replicate")[0, 0].long()
    bits, k = torch.zeros_like(y), 0
    for dy in range(7):
        for dx in range(9):
            if (dy, dx) != (3, 4):
                bits |= (pad[dy:dy + H, dx:dx + W] < y).long() << k
                k += 1
    return bits


def _arms(img, L1, L2, tau1=20, tau2=6):
    """Arm lengths (left, right, up, down) of the colour and distance double threshold."""
    c = img.permute(2, 0, 1).long()
    _, H, W = c.shape
    xs = torch.arange(W, device=c.device)[None, :].expand(H, W)
    ys = torch.arange(H, device=c.device)[:, None].expand(H, W)
    arms = []
    for sx, sy in ((-1, 0), (1, 0), (0, -1), (0, 1)):
        n, is_open, prev = torch.zeros_like(xs), torch.ones_like(xs, dtype=torch.bool), c
        for j in range(1, L1 + 1):
            x, y = xs + sx * j, ys + sy * j
            inside = (x >= 0) & (x < W) & (y >= 0) & (y < H)
            q = c[:, y.clamp(0, H - 1), x.clamp(0, W - 1)]
            to_p, to_prev = (q - c).abs().amax(0), (q - prev).abs().amax(0)
            is_open = is_open & inside & (to_p < tau1) & (to_prev < tau1)
            if j > L2:
                is_open = is_open & (to_p < tau2)
            n, prev = n + is_open.long(), q
        arms.append(n)
    return arms


def _popcount(v):
    n = torch.zeros_like(v)
    for k in range(62):
        n += (v >> k) & 1
    return n


def _exact_view(case, ref, oth, sign):
    """Eq. 3 of one reference view in FP64: (disparity, minimum aggregated cost)."""
    L1, L2 = case.get("arm_l1", 34), case.get("arm_l2", 17)
    dmin, D, order = case.get("d_min", 0), case["D"], case.get("agg_order", 0)
    l, r, u, d = _arms(ref, L1, L2)
    if case.get("smooth_arms"):
        def opened(a):
            a = F.pad(a[None, None].double(), (1, 1, 1, 1), value=1e9)
            a = -F.max_pool2d(-a, 3, 1)
            return F.max_pool2d(F.pad(a, (1, 1, 1, 1), value=-1e9), 3, 1)[0, 0].long()
        l, r, u, d = (opened(a) for a in (l, r, u, d))
    H, W = l.shape
    lmin = torch.stack((l, r, u, d)).amin(0).double()
    alpha = 1 - torch.exp(-1.0 / (lmin + float(np.float32(0.8))))
    cr, co = _census(ref), _census(oth)
    ir, io = ref.permute(2, 0, 1).double(), oth.permute(2, 0, 1).double()
    xs = torch.arange(W, device=ref.device)
    ys = torch.arange(H, device=ref.device)

    def segment_sums(v, dim):
        F_ = F.pad(torch.cumsum(v, dim), (1, 0) if dim == 1 else (0, 0, 1, 0))
        if dim == 1:
            return F_.gather(1, xs[None, :] + r + 1) - F_.gather(1, xs[None, :] - l)
        return F_.gather(0, ys[:, None] + d + 1) - F_.gather(0, ys[:, None] - u)

    dims = (1, 0) if order == 0 else (0, 1)
    count = segment_sums(segment_sums(torch.ones_like(alpha), dims[0]), dims[1])
    best, arg = torch.full_like(alpha, math.inf), torch.zeros_like(l)
    for k in range(dmin, dmin + D):
        x = xs + sign * k
        inside = ((x >= 0) & (x < W))[None, :]
        x = x.clamp(0, W - 1)
        ad = (ir - io[:, :, x]).abs().sum(0) / 3.0
        ham = _popcount(cr ^ co[:, x]).double()
        cost = alpha * (1 - torch.exp(-ad / 10.0)) + (1 - alpha) * (1 - torch.exp(-ham / 40.0))
        cost = torch.where(inside, cost, torch.ones_like(cost))
        mean = segment_sums(segment_sums(cost, dims[0]), dims[1]) / count
        better = mean < best
        best, arg = torch.where(better, mean, best), torch.where(better, torch.full_like(arg, k), arg)
    return arg, best


def _exact_match(case, left, right):
    dl, cl = _exact_view(case, left, right, -1)
    dr, cr = _exact_view(case, right, left, 1)
    W = dl.shape[1]
    x = torch.arange(W, device=dl.device)[None, :] - dl
    ok = (x >= 0) & ((dl - dr.gather(1, x.clamp(min=0))).abs() <= 1)
    return torch.where(ok, dl, torch.full_like(dl, -1)), cl, cr


def _exact_dense(case, seed):
    """Eq. 20 (default weights) solved by conjugate gradients in FP64 to the end."""
    sparse, contour, fuse, edge, pre = (t.double() if t is not None else None for t in _dense_inputs(case, seed))
    pre = torch.zeros_like(sparse) if pre is None else pre
    f32 = lambda v: float(np.float32(v))  # noqa: E731  (the parameters are FP32 numbers)
    ld, ls, ls2 = f32(0.80), f32(1.20), f32(0.02)
    s, cut = fuse * edge, contour > 0

    def weight(a, b):
        w = (1 - torch.minimum(s[a], s[b])).clamp(min=0)
        return torch.where(cut[a] != cut[b], torch.zeros_like(w), w)

    al = slice(None)
    wr = weight((al, slice(None, -1)), (al, slice(1, None)))
    wd = weight((slice(None, -1), al), (slice(1, None), al))
    data = ld * (sparse > 0) + ls2 * (pre > 0)
    b = ld * (sparse > 0) * sparse + ls2 * (pre > 0) * pre

    def apply(v):
        out = data * v
        ex, ey = 2 * ls * wr * (v[:, 1:] - v[:, :-1]), 2 * ls * wd * (v[1:] - v[:-1])
        out[:, 1:] += ex
        out[:, :-1] -= ex
        out[1:] += ey
        out[:-1] -= ey
        return out

    diag = data.clone()
    diag[:, 1:] += 2 * ls * wr
    diag[:, :-1] += 2 * ls * wr
    diag[1:] += 2 * ls * wd
    diag[:-1] += 2 * ls * wd
    x = torch.where(sparse > 0, sparse, pre)
    r = b - apply(x)
    z = r / diag
    p, rz, end = z.clone(), (r * z).sum(), 1e-13 * b.norm()
    for it in range(4000):
        ap = apply(p)
        step = rz / (p * ap).sum()
        x += step * p
        r -= step * ap
        if it % 50 == 49 and r.norm() < end:
            break
        z = r / diag
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "views":
        if case.get("vote_iters"):   # the costs are those before the vote
            case = {k: v for k, v in case.items() if k != "vote_iters"}
        left, right, _ = _pair(case, seed)
        _, cl, cr = _exact_match(case, left, right)
        return (None, None, None, cl, cr)
    if kind == "depth":
        full = _pair(case, seed, True)[:2]

        def reduced(img):
            H, W = img.shape[0] // 2, img.shape[1] // 2
            t = img[:2 * H, :2 * W].long().view(H, 2, W, 2, 3).sum((1, 3))
            return ((t + 2) >> 2).to(torch.uint8)

        disp, _, _ = _exact_match(case, *(reduced(t) for t in full))
        z = torch.where(disp > 0, FOCAL_PX * BASELINE / (2.0 * disp.clamp(min=1).double()),
                        torch.zeros(disp.shape, dtype=torch.float64, device=disp.device))
        H, W = case["H"], case["W"]
        z = F.pad(z.repeat_interleave(2, 0).repeat_interleave(2, 1), (0, W % 2, 0, H % 2))
        return (z, None)
    if kind == "densify":
        return _exact_dense(case, seed)
    return None   # whole numbers
