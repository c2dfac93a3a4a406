"""The work that users of this framework have it do, as measurable cases.

Each case is one call (or one training step) through the package's public entry points on a
seeded synthetic scene of the kinds the framework is used for: random parallelograms in the
view frustum, stacked wavy transparent layers with shared vertices, and particle clouds.
Scenes are made on the GPU from the seed alone; `exact` composites the same scene in 64 bits
from its definition (integer coverage, the fp32 depth key's order, colours in fp64).
"""
import math

import torch

import paper_2405_13364_gb300 as lr

NEAR, FAR = 0.1, 100.0
SAMPLES4 = ((-32, -96), (96, -32), (-96, 32), (32, 96))   # default 4-sample pattern, 1/256 px
LIGHT = (0.4, 0.6, 1.0, 0.25)                             # direction toward the light, ambient
LAYERS = 32


# ---- cases ------------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one checked frame of a small flat scene with the default renderer;
        # launches and host work count
        dict(name="frustum 2k 256x256", kind="frustum", quads=2000, width=256, height=256, k=3, mode="frame",
             check=True),
        # a viewer's frame with odd sizes, an 8-bit image and the per-pixel overdraw count
        dict(name="frustum 100k 1021x767 rgba8", kind="frustum", quads=100_003, width=1021, height=767, k=3,
             mode="frame", check=True, rgba8=True, count=True),
        # an interactive loop: four small views captured once, replayed with new descriptors
        dict(name="graph 4 views 512x384", kind="mixed", quads=10_000, width=512, height=384, k=3, mode="graph",
             views=4),
        # an ordinary served request: indexed layers, per-vertex colours, default renderer
        dict(name="layers 250k 1024x768 k3", kind="layers", quads=250_000, width=1024, height=768, k=3, mode="frame",
             check=True),
        # the headline frame of the benchmark, in a frame loop, with the tuned sorter capacity
        dict(name="layers 1M 1920x1080", kind="layers", quads=1_048_576, width=1920, height=1080, k=1, mode="frame",
             check=False),
        # the same with normals and a light
        dict(name="lit 1M 1920x1080", kind="lit", quads=1_048_576, width=1920, height=1080, k=1, mode="frame",
             check=False),
        # a dense particle cloud, the benchmark's second frame
        dict(name="particles 2M 1920x1080", kind="particles", quads=2_000_000, width=1920, height=1080, k=1,
             mode="frame", check=False),
        # a particle cloud at the largest served resolution with the default renderer
        dict(name="particles 300k 2560x1440 k3", kind="particles", quads=300_000, width=2560, height=1440, k=3,
             mode="frame", check=True),
        # the opt-in early stop on the dense cloud
        dict(name="threshold 2M 1920x1080", kind="particles", quads=2_000_000, width=1920, height=1080, k=1,
             mode="threshold", check=False),
        # four samples per pixel
        dict(name="msaa4 1M 1920x1080", kind="layers", quads=1_048_576, width=1920, height=1080, k=1, mode="msaa"),
        # one batched launch over requests of different sizes and kinds (what the server issues)
        dict(name="batch 6 views 1920x1080", kind="mixed", quads=400_000, width=1920, height=1080, k=3, mode="batch",
             views=6),
        # a step of colour fitting: forward, squared loss, gradient of every quad's RGBA
        dict(name="train 512k 1024x1024", kind="layers_flat", quads=524_288, width=1024, height=1024, k=1,
             mode="train"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    mode, kind = rng.choice([("frame", "frustum"), ("frame", "layers"), ("frame", "lit"), ("frame", "particles"),
                             ("threshold", "particles"), ("threshold", "layers_flat"), ("msaa", "layers"),
                             ("graph", "mixed"), ("batch", "mixed"), ("train", "layers_flat")])
    w = _log(rng, 200, 1920)
    h = min(1080, max(96, int(w * rng.uniform(0.5, 1.0))))
    c = dict(kind=kind, width=w, height=h, k=rng.choice([1, 1, 2, 3, 3]), mode=mode)
    if mode == "graph":
        return dict(c, quads=_log(rng, 2000, 100_000), views=rng.choice([2, 3, 4, 6]))
    if mode == "batch":
        return dict(c, quads=_log(rng, 10_000, 400_000), views=rng.choice([2, 4, 6]))
    if mode == "train":
        return dict(c, quads=_log(rng, 10_000, 524_288), width=min(w, 1024), height=min(h, 1024))
    if mode == "msaa":
        return dict(c, quads=_log(rng, 10_000, 1_000_000))
    c = dict(c, quads=_log(rng, 2000, 1_000_000), check=rng.random() < 0.5)
    if mode == "frame" and kind in ("frustum", "particles") and rng.random() < 0.3:
        c = dict(c, rgba8=True, count=True)
    return c


# ---- scenes -----------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _perspective(w, h):
    f = 1.0 / math.tan(math.radians(30.0))
    return torch.tensor([[f * h / w, 0, 0, 0], [0, f, 0, 0],
                         [0, 0, -(FAR + NEAR) / (FAR - NEAR), -2 * FAR * NEAR / (FAR - NEAR)],
                         [0, 0, -1, 0]], dtype=torch.float32)


def _grid(quads, w, h):
    """Layer grid: quads per row and column of one of the 32 layers (2:1 on wide screens)."""
    per = max(1, quads // LAYERS)
    wide = w / h > 1.2
    ny = max(1, int(round(math.sqrt(per / 2.0 if wide else per))))
    return max(1, per // ny), ny, wide


def _scene(kind, quads, w, h, seed):
    """dict of positions f32[V][3], indices i32[Q][4] or None, colors, mode (0 flat, 1 per
    vertex, 2 lit), size."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 1009 + 17)

    def rand(*s, lo=0.0, hi=1.0):
        return torch.rand(*s, generator=g, device=dev, dtype=torch.float64) * (hi - lo) + lo

    def colors(n, a_lo, a_hi):
        return torch.cat([rand(n, 3), rand(n, 1, lo=a_lo, hi=a_hi)], 1).float()

    s = dict(indices=None, mode=0, width=w, height=h)
    if kind == "frustum":
        t = math.tan(math.radians(30.0))
        d = (NEAR ** 3 + rand(quads) * (FAR ** 3 - NEAR ** 3)).pow(1.0 / 3.0)
        c = torch.stack([rand(quads, lo=-1) * d * t * w / h, rand(quads, lo=-1) * d * t, -d], 1)
        e = []
        for _ in range(2):
            v = torch.randn(quads, 3, generator=g, device=dev, dtype=torch.float64)
            e.append(v / v.norm(dim=1, keepdim=True) * rand(quads, 1, lo=0.05, hi=1.5) / 2)
        p = torch.stack([c - e[0] - e[1], c + e[0] - e[1], c + e[0] + e[1], c - e[0] + e[1]], 1)
        return dict(s, positions=p.reshape(-1, 3).float(), colors=colors(quads, 0.2, 0.8))
    if kind == "particles":
        c = torch.randn(quads, 3, generator=g, device=dev, dtype=torch.float64) * 2.0
        c[:, 2] -= 10.0
        half = rand(quads, lo=2.0, hi=16.0) * -c[:, 2] * math.tan(math.radians(30.0)) / h
        o = torch.tensor([[-1, -1, 0], [1, -1, 0], [1, 1, 0], [-1, 1, 0]], device=dev, dtype=torch.float64)
        p = c[:, None] + half[:, None, None] * o
        return dict(s, positions=p.reshape(-1, 3).float(), colors=colors(quads, 0.02, 0.3))
    nx, ny, wide = _grid(quads, w, h)
    half_h = 5.09 if wide else 5.38
    xs = torch.linspace(-half_h * nx / ny, half_h * nx / ny, nx + 1, device=dev, dtype=torch.float64)
    ys = torch.linspace(-half_h, half_h, ny + 1, device=dev, dtype=torch.float64)
    gy, gx = (t[None] for t in torch.meshgrid(ys, xs, indexing="ij"))
    z = -(2.0 + 0.5 * torch.arange(LAYERS, device=dev, dtype=torch.float64))[:, None, None].expand(-1, ny + 1, nx + 1)
    dzx, dzy = torch.zeros_like(z), torch.zeros_like(z)
    for _ in range(4):
        km, an, ph = (rand(LAYERS, 1, 1, lo=lo, hi=hi) for lo, hi in ((0.5, 3.0), (0, 2 * math.pi), (0, 2 * math.pi)))
        kx, ky = km * an.cos(), km * an.sin()
        arg = kx * gx + ky * gy + ph
        z = z + 0.3 * arg.sin()
        dzx, dzy = dzx + 0.3 * kx * arg.cos(), dzy + 0.3 * ky * arg.cos()
    pos = torch.stack([gx.expand_as(z), gy.expand_as(z), z], -1).reshape(-1, 3).float()
    iy, ix = torch.meshgrid(torch.arange(ny, device=dev), torch.arange(nx, device=dev), indexing="ij")
    b = (iy * (nx + 1) + ix).reshape(-1)
    quad = torch.stack([b, b + 1, b + nx + 2, b + nx + 1], 1)
    idx = (quad[None] + (torch.arange(LAYERS, device=dev) * ((nx + 1) * (ny + 1)))[:, None, None]).reshape(-1, 4)
    s = dict(s, positions=pos, indices=idx.to(torch.int32))
    if kind == "layers_flat":
        return dict(s, colors=colors(idx.shape[0], 0.1, 0.5))
    col = colors(pos.shape[0], 0.1, 0.5)
    if kind == "layers":
        return dict(s, colors=col, mode=1)
    n = torch.stack([-dzx, -dzy, torch.ones_like(dzx)], -1).reshape(-1, 3)
    n = n / n.norm(dim=1, keepdim=True)
    return dict(s, colors=torch.cat([col, n.float(), torch.zeros_like(col[:, :1])], 1).contiguous(), mode=2)


def _scenes(case, seed):
    """The case's scenes: one, or for a mixed batch one per view, of cycling kind and size."""
    w, h, q = case["width"], case["height"], case["quads"]
    if case["kind"] != "mixed":
        return [_scene(case["kind"], q, w, h, seed)]
    out = []
    for i in range(case["views"]):
        kind = ("frustum", "layers", "particles")[i % 3]
        out.append(_scene(kind, max(64, q >> ((i + 1) % 3)), max(32, w >> (i % 2)), max(32, h >> (i % 2)),
                          seed * 31 + i))
    return out


# ---- the calls --------------------------------------------------------------------------

def prepare(case, seed):
    raw = _scenes(case, seed)
    scenes = [lr.DeviceScene.from_arrays(s["positions"], s["indices"], s["colors"], s["mode"],
                                         _perspective(s["width"], s["height"]), NEAR, FAR) for s in raw]
    r = lr.Renderer(sorter_k=case["k"], alpha_threshold=case["mode"] == "threshold")
    if case["kind"] == "lit":
        r.set_lighting(LIGHT[:3], LIGHT[3])
    st = dict(case=case, r=r, scene=scenes[0], items=[(d, s["width"], s["height"]) for d, s in zip(scenes, raw)])
    if case["mode"] in ("frame", "threshold"):
        st["opts"] = {o: True for o in ("rgba8", "count") if case.get(o)}
        if not case["check"]:   # a frame loop sizes its workspace with one checked frame
            r.render(scenes[0], case["width"], case["height"], **st["opts"])
    elif case["mode"] == "graph":
        st["graph"] = r.capture(st["items"])
    elif case["mode"] == "train":
        st["colors"] = scenes[0].colors.clone().requires_grad_(True)
        st["target"] = _target(case, seed)
    return st


def _target(case, seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) + 5)
    return torch.rand(case["height"], case["width"], 4, generator=g, device=_device())


def run(state):
    c, r = state["case"], state["r"]
    w, h = c["width"], c["height"]
    if c["mode"] in ("frame", "threshold"):
        return dict(r.render(state["scene"], w, h, check=c["check"], **state["opts"]))
    if c["mode"] == "graph":
        return [dict(o) for o in state["graph"].launch(state["items"])]
    if c["mode"] == "batch":
        return [dict(o) for o in r.render_batch(state["items"])]
    if c["mode"] == "msaa":
        return dict(rgba=r.render_msaa(state["scene"], w, h, samples=4))
    state["colors"].grad = None
    img = lr.composite(state["colors"], r, state["scene"], w, h)
    ((img - state["target"]) ** 2).sum().backward()
    return dict(rgba=img.detach(), grad=state["colors"].grad)


# ---- the work a pass cannot do without -----------------------------------------------------

def _fragments(kind, quads, w, h):
    """Expected fragments of a scene (the generators' mean depth complexity)."""
    if kind == "particles":
        # mean area of U[2, 16] px squares; the share of the cloud inside the view
        inside = 0.98 if w >= h else 0.9
        return quads * (16 ** 3 - 2 ** 3) / (3 * 14) * inside
    if kind == "frustum":
        return quads * 4.1 * (w * h) / 65536.0
    return 24.0 * w * h


def work(case):
    w, h, q = case["width"], case["height"], case["quads"]
    if case["kind"] == "mixed":
        parts = [(("frustum", "layers", "particles")[i % 3], max(64, q >> ((i + 1) % 3)), max(32, w >> (i % 2)),
                  max(32, h >> (i % 2))) for i in range(case["views"])]
    else:
        parts = [(case["kind"], q, w, h)]
    nbytes = flops = 0.0
    samples = 4 if case["mode"] == "msaa" else 1
    for kind, quads, pw, ph in parts:
        if kind in ("frustum", "particles"):
            nbytes += quads * (48 + 16)
        else:
            nx, ny, _ = _grid(quads, pw, ph)
            verts = LAYERS * (nx + 1) * (ny + 1)
            quads = LAYERS * nx * ny
            nbytes += quads * 16 + verts * 12
            nbytes += {"layers": verts * 16, "lit": verts * 32, "layers_flat": quads * 16}[kind]
        nbytes += pw * ph * (16 + 4 * bool(case.get("rgba8")) + 4 * bool(case.get("count")))
        # per vertex the transform (about 20), per fragment three edge tests, the depth key and
        # the blend (about 25), interpolated colours (20) and the light (20)
        frag = _fragments(kind, quads, pw, ph) * samples
        flops += quads * 4 * 20 + frag * (25 + (20 if kind in ("layers", "lit") else 0) + (20 if kind == "lit" else 0))
        if case["mode"] == "train":   # image and target read, gradients of image and colours
            nbytes += pw * ph * 48 + quads * 16
            flops += frag * 45
    return dict(bytes=nbytes, flops=flops)


# ---- 64-bit composite -------------------------------------------------------------------

def _snap(s, sub):
    """Snapped vertices i64[Q][4] x, y (1/256 px), fp32 1/w and the visible quads' indices.
    Coverage and depth order are defined on these fp32 and integer values."""
    m = _perspective(s["width"], s["height"]).to(s["positions"].device)
    x, y, z = s["positions"].unbind(1)
    row = lambda r: ((m[r, 0] * x + m[r, 1] * y) + m[r, 2] * z) + m[r, 3]  # noqa: E731
    cx, cy, cw = row(0), row(1), row(3)
    ok = (cw >= NEAR) & (cw <= FAR)
    safe = torch.where(ok, cw, torch.ones_like(cw))
    sx = (cx / safe + 1.0) * (0.5 * s["width"])
    sy = (1.0 - cy / safe) * (0.5 * s["height"])
    ok &= (sx.abs() <= 16384.0) & (sy.abs() <= 16384.0)
    vx = torch.round(sx.clamp(-20000, 20000) * 256.0).long() - sub[0]
    vy = torch.round(sy.clamp(-20000, 20000) * 256.0).long() - sub[1]
    idx = s["indices"].long() if s["indices"] is not None else \
        torch.arange(x.numel(), device=x.device).reshape(-1, 4)
    keep = ok[idx].all(1).nonzero().reshape(-1)
    idx = idx[keep]
    return vx[idx], vy[idx], (1.0 / safe)[idx], idx, keep


def _fragments64(s, sub=(0, 0)):
    """All covering fragments front to back per pixel: sorted pixel ids, quad ids and fp64
    straight RGBA."""
    X, Y, Q, vid, quad = _snap(s, sub)
    w, h, dev = s["width"], s["height"], X.device
    bx0 = ((X.amin(1) + 127) >> 8).clamp(min=0)
    bx1 = ((X.amax(1) - 128) >> 8).clamp(max=w - 1)
    by0 = ((Y.amin(1) + 127) >> 8).clamp(min=0)
    by1 = ((Y.amax(1) - 128) >> 8).clamp(max=h - 1)
    bw = (bx1 - bx0 + 1).clamp(min=0)
    area = bw * (by1 - by0 + 1).clamp(min=0)
    # per triangle: vertices oriented to a positive doubled area
    tri = []
    for t in (0, 1):
        a, b, c = 0, 1 + t, 2 + t
        A = (X[:, b] - X[:, a]) * (Y[:, c] - Y[:, a]) - (Y[:, b] - Y[:, a]) * (X[:, c] - X[:, a])
        sw = A < 0
        pick = lambda v, i, j: torch.stack([v[:, 0], torch.where(sw, v[:, j], v[:, i]),   # noqa: E731,B023
                                            torch.where(sw, v[:, i], v[:, j])], 1)
        tri.append((pick(X, b, c), pick(Y, b, c), pick(Q, b, c), A.abs(), pick(vid, b, c)))
    cum = area.cumsum(0)
    pixs, keys, quads, cols = [], [], [], []
    n, start = X.shape[0], 0
    while start < n:
        base = int(cum[start - 1]) if start else 0
        end = max(start + 1, int(torch.searchsorted(cum, base + 60_000_000, right=True)))
        own = torch.repeat_interleave(torch.arange(start, end, device=dev), area[start:end])
        o = torch.arange(own.numel(), device=dev) - (cum[own] - area[own] - base)
        px, py = bx0[own] + o % bw[own], by0[own] + o // bw[own]
        Px, Py = 256 * px + 128, 256 * py + 128
        cov = torch.zeros(own.numel(), 2, dtype=torch.bool, device=dev)
        for t in (0, 1):
            tx, ty, _, A, _ = tri[t]
            c = A[own] > 0
            for u, v in ((1, 2), (2, 0), (0, 1)):
                dx, dy = (tx[:, v] - tx[:, u])[own], (ty[:, v] - ty[:, u])[own]
                e = dx * (Py - ty[:, u][own]) - dy * (Px - tx[:, u][own])
                c &= (e > 0) | ((e == 0) & ((dy < 0) | ((dy == 0) & (dx > 0))))
            cov[:, t] = c
        hit = cov.reshape(-1).nonzero().reshape(-1)   # ascending (quad, pixel, triangle)
        del cov
        at, t = hit >> 1, (hit & 1).bool()
        qi = own[at]
        Px, Py, pix = Px[at], Py[at], py[at] * w + px[at]
        del own, o, px, py
        sel = lambda k: torch.where(t.reshape(-1, *[1] * (tri[0][k].dim() - 1)), tri[1][k][qi], tri[0][k][qi])  # noqa: E731,B023
        tx, ty, tq, A = sel(0), sel(1), sel(2), sel(3)
        edge = lambda u, v: (tx[:, v] - tx[:, u]) * (Py - ty[:, u]) - (ty[:, v] - ty[:, u]) * (Px - tx[:, u])  # noqa: E731,B023
        e1, e2 = edge(2, 0), edge(0, 1)
        inv = 1.0 / A.float()
        l1, l2 = e1.float() * inv, e2.float() * inv
        key = tq[:, 0] + (l1 * (tq[:, 1] - tq[:, 0]) + l2 * (tq[:, 2] - tq[:, 0]))
        if s["mode"] == 0:
            col = s["colors"][quad[qi]].double()
        else:
            wt = torch.stack([(A - e1 - e2).double(), e1.double(), e2.double()], 1) * tq.double()
            tv = sel(4)
            at3 = lambda lo, hi: sum(wt[:, k:k + 1] * s["colors"][tv[:, k], lo:hi].double() for k in range(3))  # noqa: E731,B023
            col = at3(0, 4) / wt.sum(1, keepdim=True)
            if s["mode"] == 2:
                nrm = at3(4, 7)
                L = torch.tensor(LIGHT[:3], dtype=torch.float64, device=dev)
                lam = (nrm @ (L / L.norm())).abs() / nrm.norm(dim=1)
                col[:, :3] *= (LIGHT[3] + (1 - LIGHT[3]) * lam)[:, None]
        pixs.append(pix)
        keys.append(key.view(torch.int32).long())
        quads.append(quad[qi])
        cols.append(col if s["mode"] else None)
        start = end
    if not pixs:
        z = torch.zeros(0, dtype=torch.long, device=dev)
        return z, z, torch.zeros(0, 4, dtype=torch.float64, device=dev)
    # front to back: larger key first, equal keys with the higher quad, then triangle, first
    pix, key, qd = (torch.cat(v).flip(0) for v in (pixs, keys, quads))
    order = torch.sort((pix << 32) | (0x7FFFFFFF - key), stable=True)[1]
    pix, qd = pix[order], qd[order]
    col = torch.cat(cols).flip(0)[order] if s["mode"] else s["colors"][qd].double()
    return pix, qd, col


def _composite64(s, sub=(0, 0), threshold=False, target=None):
    """fp64 image [H][W][4]; with a target also the gradient of the squared loss, f64[Q][4]."""
    pix, quad, col = _fragments64(s, sub)
    n, dev = s["width"] * s["height"], pix.device
    count = torch.bincount(pix, minlength=n)
    first = count.cumsum(0) - count
    by = torch.sort(count, descending=True)[1]         # pixels with more fragments first
    img = torch.zeros(n, 3, dtype=torch.float64, device=dev)
    T = torch.ones(n, dtype=torch.float64, device=dev)
    T32 = torch.ones(n, dtype=torch.float32, device=dev)
    most = int(count.max()) if n else 0
    alive = (n - torch.searchsorted(torch.sort(count)[0], torch.arange(most, device=dev), right=True)).tolist()
    front = torch.empty_like(col[:, 0]) if target is not None else None
    done = torch.empty_like(col[:, :3]) if target is not None else None
    for r in range(most):
        p = by[:alive[r]]
        f = first[p] + r
        if threshold:   # the stop is defined on the running fp32 product
            go = T32[p] > 1.0 / 128.0
            p, f = p[go], f[go]
        a = col[f, 3]
        img[p] += (T[p] * a)[:, None] * col[f, :3]
        if target is not None:
            front[f], done[f] = T[p], img[p]
        T[p] *= 1.0 - a
        if threshold:
            T32[p] *= 1.0 - a.float()
    out = torch.cat([img, (1.0 - T)[:, None]], 1)
    if target is None:
        return out.reshape(s["height"], s["width"], 4)
    g = 2.0 * (out - target.reshape(n, 4).double())
    gp, a = g[pix], col[:, 3]
    grad = torch.zeros(s["colors"].shape[0], 4, dtype=torch.float64, device=dev)
    da = (gp[:, :3] * (front[:, None] * col[:, :3] - (img[pix] - done) / (1.0 - a)[:, None])).sum(1)
    da += gp[:, 3] * T[pix] / (1.0 - a)
    grad.index_add_(0, quad, torch.cat([gp[:, :3] * (front * a)[:, None], da[:, None]], 1))
    return out.reshape(s["height"], s["width"], 4), grad


def exact(case, seed):
    scenes = _scenes(case, seed)
    if case["mode"] == "msaa":
        return dict(rgba=sum(_composite64(scenes[0], d) for d in SAMPLES4) / 4.0)
    if case["mode"] == "train":
        img, grad = _composite64(scenes[0], target=_target(case, seed))
        return dict(rgba=img, grad=grad)
    if case["mode"] in ("graph", "batch"):
        return [dict(rgba=_composite64(s)) for s in scenes]
    out = dict(rgba=_composite64(scenes[0], threshold=case["mode"] == "threshold"))
    return dict(out, **{o: None for o in ("rgba8", "count") if case.get(o)})
