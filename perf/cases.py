"""The work a user of this package has it do, as cases that can be timed and compared.

Every case goes through a public entry point: one pair on the device
(``Stereo``), one pair in host buffers (``Stereo.compute_host``), a batch
(``stereo_compute_batch``) and a training step (``soft_argmin_disparity`` and its
gradients). The shapes are those of ``scenes.paper_shapes``, the tests and the
benchmark; a 4K pair is the largest.

``exact`` restates the method with torch in 64-bit integers and floats.
"""
import math

import numpy as np
import torch

from paper_2212_00488_gb300 import Stereo, _lib
from paper_2212_00488_gb300.diff import soft_argmin_disparity
from paper_2212_00488_gb300.stereo import stream_handle

MIX = ((640, 480, 64), (1024, 768, 96), (1436, 992, 145), (1920, 1080, 192))
MAX_CELLS = 3840 * 2160 // 4 * 128        # processed (x, y, d) cells of the largest listed case


def _pair(name, W, H, dmax, downscale=1, wx=21, maps=True):
    return {"name": name, "kind": "pair", "W": W, "H": H, "dmax": dmax, "downscale": downscale, "wx": wx,
            "maps": maps}


def listed():
    return [
        # a small pair without downscaling, with every map read: the smallest frame of the method
        _pair("pair_360x248_d36", 360, 248, 36, downscale=0),
        # a VGA camera pair, only the final map wanted: a real-time loop where launches count
        _pair("pair_640x480_d64", 640, 480, 64, maps=False),
        # the paper's shape (Adirondack, half size) with the whole pipeline
        _pair("pair_1436x992_d145", 1436, 992, 145),
        # a Pipes-like pair: width not a multiple of four
        _pair("pair_1482x994_d128", 1482, 994, 128),
        # a full-HD pair, only the final map wanted
        _pair("pair_1920x1080_d192", 1920, 1080, 192, maps=False),
        # a 4K pair: the largest frame
        _pair("pair_3840x2160_d256", 3840, 2160, 256),
        # a wide horizontal window (61 per side, the window study of the paper's Table I)
        _pair("pair_1436x992_d145_wx61", 1436, 992, 145, wx=61),
        # a program without device buffers: pinned host images in, the host map out
        {"name": "host_1436x992_d145", "kind": "host", "W": 1436, "H": 992, "dmax": 145},
        # what a server at low load hands over: two small requests at once
        {"name": "batch2_vga", "kind": "batch", "n": 2, "sizes": "vga"},
        # a full batch of mixed resolutions
        {"name": "batch16_mix", "kind": "batch", "n": 16, "sizes": "mix"},
        # a training step on small odd-sized crops: forward and all gradients
        {"name": "train_2x205x123_d24", "kind": "train", "B": 2, "W": 205, "H": 123, "D": 24},
        # a training step at the paper's processed shape
        {"name": "train_4x718x496_d73", "kind": "train", "B": 4, "W": 718, "H": 496, "D": 73},
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(("pair", "pair", "pair", "host", "batch", "train", "train"))
    if kind in ("pair", "host"):
        while True:
            W = _log(rng, 320, 3840)
            H = max(240, int(W * rng.uniform(0.5, 0.8)))
            dmax = _log(rng, 24, 384)
            # frames small enough to need no downscaling are taken as they are, half of the time
            down = 0 if W <= 800 and dmax <= 128 and kind == "pair" and rng.random() < 0.5 else 1
            if W * H * dmax // (8 if down else 1) <= MAX_CELLS and dmax < W:
                break
        if kind == "host":
            return {"kind": "host", "W": W, "H": H, "dmax": dmax}
        wx = rng.choice((21, 21, 21, 21, 11, 41, 61))
        return {"kind": "pair", "W": W, "H": H, "dmax": dmax, "downscale": down, "wx": wx,
                "maps": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(1, 16), "sizes": "mix", "order": rng.randrange(1 << 16)}
    while True:
        B, W, D = rng.randint(1, 4), _log(rng, 96, 718), _log(rng, 12, 96)
        H = max(64, int(W * rng.uniform(0.5, 0.8)))
        if B * W * H * D <= 4 * 718 * 496 * 73:
            return {"kind": "train", "B": B, "W": W, "H": H, "D": D}


def _frames(case):
    """(W, H, dmax) of every pair of a plain case."""
    if case["kind"] != "batch":
        return [(case["W"], case["H"], case["dmax"])]
    if case["sizes"] == "vga":
        return [MIX[0]] * case["n"]
    order = np.random.Generator(np.random.PCG64(case.get("order", 0))).integers(0, len(MIX), case["n"])
    return [MIX[int(i)] for i in order]


# ------------------------------------------------------------------ inputs

def _scene(W, H, dmax, gen, planes=40):
    """A piecewise-planar pair on the GPU, as scenes.make_scene draws it (Voronoi
    planes, the right image warped along the rows with the nearer surface in
    front, fresh noise in the holes, sensor noise of 2 grey levels), with a
    texture strength of its own for each plane, from almost flat to the 20
    levels of scenes.make_scene, so that short and long cross arms both occur."""
    dev = "cuda"

    def u(a, b, *shape):
        return torch.rand(*shape, generator=gen, device=dev) * (b - a) + a

    xs = torch.arange(W, device=dev, dtype=torch.float32)[None, :]
    ys = torch.arange(H, device=dev, dtype=torch.float32)[:, None]
    sx, sy = u(0, W, planes).tolist(), u(0, H, planes).tolist()
    best = torch.full((H, W), 3.0e38, device=dev)
    lab = torch.zeros((H, W), dtype=torch.int64, device=dev)
    for k in range(planes):
        dist = (xs - sx[k]) ** 2 + (ys - sy[k]) ** 2
        near = dist < best
        best = torch.where(near, dist, best)
        lab.masked_fill_(near, k)
    a, b, c = u(0, dmax - 1, planes), u(-0.05, 0.05, planes), u(-0.05, 0.05, planes)
    disp = (a[lab] + b[lab] * xs + c[lab] * ys).clamp(0, dmax - 1).round().long()
    amp = torch.exp(u(math.log(2.0), math.log(20.0), planes)) * math.sqrt(3.0)
    tex = u(-1, 1, H, W) * amp[lab]
    base, gx, gy = u(40, 215, planes, 3), u(-60, 60, planes, 3) / W, u(-60, 60, planes, 3) / H
    left = base[lab] + gx[lab] * xs[..., None] + gy[lab] * ys[..., None] + tex[..., None]
    # forward warp: the largest (disparity, column) that lands on a pixel wins
    col = torch.arange(W, device=dev)[None, :].expand(H, W)
    tgt = col - disp
    key = torch.where(tgt >= 0, disp * W + col, -torch.ones_like(col))
    front = torch.full((H, W), -1, dtype=torch.int64, device=dev)
    front.scatter_reduce_(1, tgt.clamp(min=0), key, "amax")
    src = (front % W).clamp(min=0)[..., None].expand(H, W, 3)
    right = torch.where((front >= 0)[..., None], left.gather(1, src), u(20, 235, H, W, 3))

    def finish(img):
        noise = torch.randn(H, W, 3, generator=gen, device=dev) * 2.0
        return (img + noise).round().clamp(0, 255).to(torch.uint8).contiguous()
    return finish(left), finish(right)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _pairs(case, seed):
    g = _gen(seed)
    return [_scene(W, H, d, g) for W, H, d in _frames(case)]


def _train_inputs(case, seed):
    B, W, H, D = case["B"], case["W"], case["H"], case["D"]
    g = _gen(seed)
    s = [_scene(W, H, D, g, planes=12) for _ in range(B)]
    lu, ru = torch.stack([p[0] for p in s]), torch.stack([p[1] for p in s])
    theta = torch.tensor([1.0, 1.0, 0.3, 2.3], device="cuda")
    # the loss gradient of an L1 loss: a sign for each pixel, over their number
    go = torch.where(torch.rand(B, H, W, generator=g, device="cuda") < 0.5, -1.0, 1.0) / (B * H * W)
    return lu, ru, lu.float() / 255.0, ru.float() / 255.0, theta, go


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = case
    kind = case["kind"]
    if kind == "train":
        st.lu, st.ru, st.l, st.r, st.theta, st.go = _train_inputs(case, seed)
        for t in (st.l, st.r, st.theta):
            t.requires_grad_(True)
        st.ctx = Stereo(0, downscale=0)
        return st
    pairs = _pairs(case, seed)
    if kind == "pair":
        st.left, st.right = pairs[0]
        st.ctx = Stereo(0, downscale=case["downscale"], wx=case["wx"])
    elif kind == "host":
        st.left, st.right = (t.cpu().pin_memory() for t in pairs[0])
        st.disp = torch.empty(case["H"], case["W"], pin_memory=True)
        st.ctx = Stereo(0)
    else:
        st.pairs = pairs
        st.ctx = Stereo(0)
        st.disp = [torch.empty(p[0].shape[:2], device="cuda") for p in pairs]
        st.jobs = [_lib.stereo_job(p[0].data_ptr(), p[1].data_ptr(), W, H, d, o.data_ptr(), None, None, None)
                   for p, o, (W, H, d) in zip(pairs, st.disp, _frames(case))]
    return st


def run(st):
    case = st.case
    kind = case["kind"]
    if kind == "pair":
        o = st.ctx(st.left, st.right, case["dmax"], maps=case["maps"])
        return {"disp": o.disp, "dl": o.dl, "dr": o.dr, "gcp": o.gcp} if case["maps"] else {"disp": o.disp}
    if kind == "host":
        st.ctx.compute_host(st.left, st.right, case["dmax"], st.disp)
        return {"disp": st.disp}
    if kind == "batch":
        _lib.stereo_compute_batch(st.ctx.ctx, st.jobs, stream_handle(torch.cuda.current_stream()))
        return {"disp": st.disp}
    dhat = soft_argmin_disparity(st.l, st.r, st.theta, st.lu, st.ru, case["D"], 0.1, st.ctx)
    gl, gr, gt = torch.autograd.grad(dhat, (st.l, st.r, st.theta), st.go)
    return {"dhat": dhat.detach(), "grad_left": gl, "grad_right": gr, "grad_theta": gt}


def work(case):
    if case["kind"] == "train":
        n = case["B"] * case["W"] * case["H"]
        # in: two float and two uint8 RGB images and the loss gradient; out: the map and two image
        # gradients. A cell: 48 flops, 9 exponentials and six window sums of at least two terms
        return {"bytes": n * (2 * 12 + 2 * 3 + 4 + 4 + 2 * 12) + 32, "flops": n * case["D"] * 69}
    nbytes = cells = 0
    down = case.get("downscale", 1)
    for W, H, d in _frames(case):
        X, Y, D = (W // 2, H // 2, (d + 1) // 2) if down else (W, H, d)
        nbytes += 10 * W * H + (3 * X * Y if case.get("maps") else 0)
        cells += X * Y * D
    # a cell: 13 integer operations for the cost, both aggregations and the argmin of both bases
    return {"bytes": nbytes, "flops": 13 * cells}


# ------------------------------------------------------------------ the method in 64 bits

def _grey(rgb):
    c = rgb.long()
    return (77 * c[..., 0] + 150 * c[..., 1] + 29 * c[..., 2] + 128) >> 8


def _edge(t, dy, dx):
    """t(y + dy, x + dx) with coordinates clamped to the image."""
    H, W = t.shape
    y = (torch.arange(H, device=t.device) + dy).clamp(0, H - 1)
    x = (torch.arange(W, device=t.device) + dx).clamp(0, W - 1)
    return t[y][:, x]


def _halve(g):
    H, W = g.shape
    s = sum(_edge(g, j, i) for j in (-1, 0, 1) for i in (-1, 0, 1))
    return ((s + 4) // 9)[0:H // 2 * 2:2, 0:W // 2 * 2:2]


def _census(g):
    code = torch.zeros_like(g)
    for k, (dx, dy) in enumerate(((-1, -1), (1, -1), (-2, 0), (2, 0), (-1, 1), (1, 1))):
        code |= (_edge(g, dy, dx) < g).long() << k
    return code


def _arms(g, wx, wy, tc):
    """left, right, up and down arm lengths."""
    H, W = g.shape
    x, y = torch.arange(W, device=g.device)[None, :], torch.arange(H, device=g.device)[:, None]
    out = []
    for dy, dx, cap in ((0, -1, wx), (0, 1, wx), (-1, 0, wy), (1, 0, wy)):
        n, on = torch.zeros_like(g), torch.ones_like(g, dtype=torch.bool)
        for k in range(1, cap + 1):
            inside = (x + k * dx >= 0) & (x + k * dx < W) & (y + k * dy >= 0) & (y + k * dy < H)
            on = on & inside & ((_edge(g, k * dy, k * dx) - g).abs() < tc)
            n = n + on
        out.append(n)
    return out


def _popcount(v):
    return sum((v >> k) & 1 for k in range(6))


def _window(c, lo, hi, dim):
    """Sums of c from index lo to hi (both included) along dim, by differences of 64-bit prefixes."""
    pad = (1, 0) if dim == c.dim() - 1 else (0, 0, 1, 0)
    s = torch.nn.functional.pad(c.cumsum(dim), pad)
    return s.gather(dim, (hi + 1).expand_as(c)) - s.gather(dim, lo.expand_as(c))


def _exact_pair(left, right, dmax, downscale=1, wx=21, wy=31, tc=13, T=3, scale=512.0, lam=(0.3, 2.3)):
    dev = left.device
    full = _grey(left)
    gl, gr = full, _grey(right)
    D = dmax
    if downscale:
        gl, gr, D = _halve(gl), _halve(gr), (dmax + 1) // 2
    Y, X = gl.shape

    def table(n, f):
        return torch.tensor([math.floor(scale * (1 - math.exp(-f(i))) + 0.5) for i in range(n)], device=dev)
    ad, mc = table(256, lambda i: i / 255.0 / lam[0]), table(7, lambda i: i / lam[1])
    P = ad[255] + mc[6]
    cl, cr = _census(gl), _census(gr)
    x, y = torch.arange(X, device=dev)[None, :], torch.arange(Y, device=dev)[:, None]
    spans = []
    for g in (gl, gr):
        m, n, M, N = _arms(g, wx, wy, tc)
        spans.append((x - m, x + n, y - M, y + N))
    best = [torch.full((Y, X), 1 << 60, device=dev) for _ in range(2)]
    for d in range(D):
        C = P.expand(Y, X).clone()
        if d < X:
            C[:, d:] = ad[(gl[:, d:] - gr[:, :X - d]).abs()] + mc[_popcount(cl[:, d:] ^ cr[:, :X - d])]
        CR = P.expand(Y, X).clone()
        if d < X:
            CR[:, :X - d] = C[:, d:]
        for b, c in enumerate((C, CR)):
            x0, x1, y0, y1 = spans[b]
            best[b] = torch.minimum(best[b], (_window(_window(c, x0, x1, 1), y0, y1, 0) << 8) | d)
    dl, dr = best[0] & 255, best[1] & 255
    gcp = (x - dl >= 0) & (dr.gather(1, (x - dl).clamp(min=0)) == dl)
    med = torch.stack([_edge(dl, j, i) for j in (-1, 0, 1) for i in (-1, 0, 1)]).sort(0).values[4]
    # the nearest matched pixels on either side, then the fill
    xi = x.expand(Y, X)
    li = torch.where(gcp, xi, -1).cummax(1).values
    ri = torch.where(gcp, xi, X).flip(1).cummin(1).values.flip(1)
    hl, hr = li >= 0, ri < X
    lc, rc = li.clamp(min=0), ri.clamp(max=X - 1)
    a, b = med.gather(1, lc), med.gather(1, rc)
    i, j = (x - lc), (rc - x)
    lin = (a * j + b * i).double() / (i + j).clamp(min=1)
    edge = torch.where((gl.gather(1, lc) - gl).abs() < (gl.gather(1, rc) - gl).abs(), a, b).double()
    both = torch.where((a - b).abs() <= T, lin, edge)
    one = torch.where(hl, a, torch.where(hr, b, torch.zeros_like(a))).double()
    dp = torch.where(gcp, med.double(), torch.where(hl & hr, both, one))
    disp = dp
    if downscale:
        H, W = full.shape
        disp = torch.zeros(H, W, dtype=torch.float64, device=dev)
        e = 2 * dp
        nxt = dp[:, 1:]
        fo = full[0:2 * Y:2, 1:2 * X - 2:2]
        side = torch.where((gl[:, :-1] - fo).abs() < (gl[:, 1:] - fo).abs(), dp[:, :-1], nxt)
        o = torch.where((dp[:, :-1] - nxt).abs() <= T, dp[:, :-1] + nxt, 2 * side)
        row = torch.empty(Y, W, dtype=torch.float64, device=dev)
        row[:, 0:2 * X:2] = e
        row[:, 1:2 * X - 2:2] = o
        row[:, 2 * X - 1:] = e[:, -1:]
        disp[0:2 * Y:2] = row
        disp[1:2 * Y - 1:2] = 0.5 * (row[:-1] + row[1:])
        disp[2 * Y - 1:] = row[-1:]
    return disp, dl.to(torch.uint8), dr.to(torch.uint8), gcp.to(torch.uint8)


def _exact_train(case, seed):
    lu, ru, l, r, theta, go = _train_inputs(case, seed)
    B, D = case["B"], case["D"]
    l, r, th = (t.double().requires_grad_(True) for t in (l, r, theta))
    w = torch.tensor([77.0, 150.0, 29.0], dtype=torch.float64, device="cuda") / 256.0
    grads, dhats = [torch.zeros_like(l), torch.zeros_like(r), torch.zeros_like(th)], []
    for p in range(B):
        q = _grey(lu[p])
        cl, cr = _census(q), _census(_grey(ru[p]))
        m, n, M, N = _arms(q, 21, 31, 13)
        Y, X = q.shape
        x, y = torch.arange(X, device="cuda")[None, :], torch.arange(Y, device="cuda")[:, None]
        x0, x1, y0, y1 = x - m, x + n, y - M, y + N
        size = _window(_window(torch.ones(Y, X, dtype=torch.float64, device="cuda"), x0, x1, 1), y0, y1, 0)
        gl, gr = (l[p] * w).sum(-1), (r[p] * w).sum(-1)
        P = th[0] * (1 - torch.exp(-1 / th[2])) + th[1] * (1 - torch.exp(-6 / th[3]))
        z = []
        for d in range(D):
            C = P.expand(Y, X)
            if d < X:
                ham = _popcount(cl[:, d:] ^ cr[:, :X - d]).double()
                c = (th[0] * (1 - torch.exp(-(gl[:, d:] - gr[:, :X - d]).abs() / th[2]))
                     + th[1] * (1 - torch.exp(-ham / th[3])))
                C = torch.cat((P.expand(Y, d), c), 1)
            z.append(-_window(_window(C, x0, x1, 1), y0, y1, 0) / size / 0.1)
        soft = torch.softmax(torch.stack(z), 0)
        dhat = (soft * torch.arange(D, dtype=torch.float64, device="cuda")[:, None, None]).sum(0)
        for acc, g in zip(grads, torch.autograd.grad(dhat, (l, r, th), go[p].double())):
            acc += g
        dhats.append(dhat.detach())
    return {"dhat": torch.stack(dhats), "grad_left": grads[0], "grad_right": grads[1], "grad_theta": grads[2]}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    pairs = _pairs(case, seed)
    if case["kind"] == "batch":
        return {"disp": [_exact_pair(l, r, d)[0] for (l, r), (_, _, d) in zip(pairs, _frames(case))]}
    (l, r), d = pairs[0], case["dmax"]
    if case["kind"] == "host":
        return {"disp": _exact_pair(l, r, d)[0]}
    disp, dl, dr, gcp = _exact_pair(l, r, d, case["downscale"], case["wx"])
    return {"disp": disp, "dl": dl, "dr": dr, "gcp": gcp} if case["maps"] else {"disp": disp}
