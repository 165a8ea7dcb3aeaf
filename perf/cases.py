"""The framework's work, as cases to be timed: each kind of call that a user
of the renderer makes, over the range of sizes that the repository's own
configurations, tests and benchmark use.

Inputs are Zel'dovich lattices (the recipe of lt_inputs/zeldovich.py, drawn on
the GPU so that a 256^3 lattice takes milliseconds): n = -2.5, cut-off at 3/8
of the lattice's wavenumbers, growth set by the largest deformation eigenvalue
`lam` (above 1: shell crossing). `exact` evaluates the same quantities with
plain torch operations in FP64.
"""
from __future__ import annotations

import math

import torch

from paper_1208_3206_gb300 import Renderer
from paper_1208_3206_gb300.render import lt_render

# ---------------------------------------------------------------------------
# cases


def listed():
    return [
        # one frame of a small lattice: an interactive preview, bound by launches and latency
        dict(name="frame_small", kind="frame", N=32, W=256, H=256, view="z", lam=1.5, half=False, tile=0),
        # one frame of an ordinary snapshot over the periodic box window
        dict(name="frame_ortho", kind="frame", N=128, W=1024, H=1024, view="z", lam=3.0, half=False, tile=0),
        # one frame of the same snapshot from a perspective camera, at a screen's size
        dict(name="frame_persp", kind="frame", N=128, W=1920, H=1080, view="persp", lam=3.0, half=False, tile=0),
        # a large snapshot stored as half-precision offsets, seen obliquely at a size that no tile divides
        dict(name="frame_half", kind="frame", N=256, W=1501, H=1387, view="oblique", lam=4.0, half=True, tile=0),
        # a camera path over two large snapshots, replayed as one graph (the benchmark's workload, fewer frames)
        dict(name="movie", kind="movie", N=256, W=2048, H=2048, snaps=2, cams=4, lam=3.0, tile=64),
        # one step of fitting positions to an image: forward, loss and gradient
        dict(name="grad_step", kind="grad", N=64, W=512, H=512, view="z", lam=2.0, cams=1),
        # registering a new snapshot, with the density of every tetrahedron
        dict(name="build", kind="build", N=256, snaps=1, lam=3.0, half=False),
        # deposit onto a periodic grid
        dict(name="resample", kind="resample", N=128, n=512, lam=3.0, half=False, weight="density"),
        # a density slice through a large snapshot
        dict(name="slice", kind="slice", N=256, n=2048, lam=3.0, half=False, weight="density"),
        # the centroid splats of a snapshot
        dict(name="centroids", kind="centroids", N=128, W=1024, H=1024, view="z", lam=3.0),
        # near cubes exactly, far ones as splats
        dict(name="hybrid", kind="hybrid", N=128, W=1024, H=1024, lam=3.0, near=2.0),
        # area-averaged pixels
        dict(name="area", kind="area", N=128, W=1024, H=1024, view="z", lam=3.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "movie", "grad", "build", "resample", "slice", "centroids", "hybrid", "area"])
    top = {"frame": 256, "movie": 192, "build": 256, "slice": 256}.get(kind, 128)
    c = dict(kind=kind, N=_log_int(rng, 16, top), lam=round(rng.uniform(0.5, 3.0 if kind == "grad" else 4.0), 3),
             box=rng.choice([1.0, 1.0, 100.0]))
    if kind in ("build", "resample", "slice"):
        c["half"] = rng.random() < 0.3
    if kind == "build":
        c["snaps"] = rng.choice([1, 1, 2]) if c["N"] < 200 else 1
        return c
    if kind in ("resample", "slice"):
        c["n"] = _log_int(rng, 24, 512 if kind == "resample" else 2048)
        c["weight"] = rng.choice(["density", "streams"])
        return c
    most = {"frame": 2048, "movie": 1600}.get(kind, 1024)
    c["W"], c["H"] = _log_int(rng, 96, most), _log_int(rng, 96, most)
    if kind == "frame":
        c["view"] = rng.choice(["z", "oblique", "persp"])
        c["half"] = c["view"] != "z" and rng.random() < 0.4
        c["tile"] = rng.choice([0, 0, 8, 32, 64])
    elif kind == "movie":
        c["snaps"], c["cams"], c["tile"] = rng.choice([1, 2]), rng.choice([1, 2, 3]), rng.choice([0, 32, 64])
    elif kind == "grad":
        c["view"], c["cams"] = rng.choice(["z", "oblique"]), rng.choice([1, 2])
    elif kind == "hybrid":
        c["near"] = round(rng.uniform(1.3, 2.7), 3)
    else:
        c["view"] = rng.choice(["z", "oblique"])
    return c


# ---------------------------------------------------------------------------
# inputs


def _wave(N):
    k = torch.fft.fftfreq(N, d=1.0 / N, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    kx = torch.fft.rfftfreq(N, d=1.0 / N, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    return kx[None, None, :], k[None, :, None], k[:, None, None]


def _largest_eigenvalue(a, b, c, d, e, f):
    """The largest eigenvalue over all symmetric matrices ((a, d, e), (d, b, f), (e, f, c))."""
    q = (a + b + c) / 3.0
    p = torch.sqrt(((a - q) ** 2 + (b - q) ** 2 + (c - q) ** 2 + 2.0 * (d * d + e * e + f * f)) / 6.0).clamp_min(1e-300)
    a, b, c, d, e, f = (a - q) / p, (b - q) / p, (c - q) / p, d / p, e / p, f / p
    r = 0.5 * (a * (b * c - f * f) - d * (d * c - f * e) + e * (d * f - b * e))
    return float((q + 2.0 * p * torch.cos(torch.acos(r.clamp(-1.0, 1.0)) / 3.0)).max())


def _displacement(N, lam, seed):
    """Zel'dovich displacement of a unit box, [N^3][3] float64 in id order."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    white = torch.randn((N, N, N), generator=g, device="cuda", dtype=torch.float64)
    delta = torch.fft.rfftn(white)
    k = _wave(N)
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    inv = torch.where(k2 > 0, 1.0 / k2.clamp_min(1e-30), torch.zeros_like(k2))
    kc = 0.375 * N * 2.0 * math.pi
    delta = delta * torch.sqrt(torch.where(k2 > 0, k2.clamp_min(1e-30) ** -1.25 * torch.exp(-k2 / (kc * kc)), torch.zeros_like(k2)))
    if N % 2 == 0:
        delta[N // 2], delta[:, N // 2], delta[:, :, N // 2] = 0, 0, 0
    size = (N, N, N)
    t = [torch.fft.irfftn(k[a] * k[b] * delta * inv, s=size) for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
    grow = lam / _largest_eigenvalue(*t)
    del t
    return torch.stack([torch.fft.irfftn(1j * k[a] * delta * inv, s=size).reshape(-1) * grow for a in range(3)], dim=1)


def _lattice(N, box):
    h = float(torch.tensor(box, dtype=torch.float32)) / N
    i = torch.arange(N, device="cuda", dtype=torch.float64) * h
    z, y, x = torch.meshgrid(i, i, i, indexing="ij")
    return torch.stack([x, y, z], dim=-1).reshape(-1, 3)


def _positions(case, seed):
    """The snapshots of a case as the renderer takes them: [S][N^3][4]."""
    N, box, half = case["N"], case.get("box", 1.0), case.get("half", False)
    S = case.get("snaps", 1)
    out = torch.zeros((S, N ** 3, 4), dtype=torch.float16 if half else torch.float32, device="cuda")
    for s in range(S):
        lam = case["lam"] * (1.0 if s == 0 else 0.5)
        d = _displacement(N, lam, 1000 * int(seed) + 7 * s + 1)
        if half:
            out[s, :, :3] = (d * N).to(torch.float16)
        else:
            x = torch.remainder(_lattice(N, box) + d * box, box).to(torch.float32)
            out[s, :, :3] = torch.where(x >= box, torch.zeros_like(x), x)
    return out


def _unit(v):
    n = math.sqrt(sum(x * x for x in v))
    return [x / n for x in v]


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _dot(a, b):
    return sum(x * y for x, y in zip(a, b))


def _axes(cam):
    f = _unit(cam["fwd"])
    r = _unit(_cross(cam["up"], f))
    return r, _cross(f, r), f


def _cameras(case):
    """The views of a case, as dicts of the renderer's camera fields."""
    W, H, box = case["W"], case["H"], case.get("box", 1.0)
    view = case.get("view", "persp")
    n = case.get("cams", 1)
    if view == "z":
        # the periodic window of the box; further cameras look along the other axes
        axes = [((0, 0, 1), (0, 1, 0)), ((1, 0, 0), (0, 0, 1)), ((0, 1, 0), (1, 0, 0))]
        return [dict(type="ortho", W=W, H=H, fwd=f, up=u, lo=(0.0, 0.0), hi=(box, box), wrap=True) for f, u in axes[:n]]
    cams = []
    centre = [0.5 * box] * 3
    for i in range(n):
        if view == "oblique":
            cam = dict(type="ortho", W=W, H=H, fwd=(1.0 + 0.3 * i, 2.0, 2.5), up=(0.0, 0.0, 1.0), wrap=False)
            r, u, _ = _axes(cam)
            half = (0.55 * box, 0.6 * box)
            cam["lo"] = tuple(_dot(a, centre) - q for a, q in zip((r, u), half))
            cam["hi"] = tuple(_dot(a, centre) + q for a, q in zip((r, u), half))
        else:
            z = 1.0 - 2.0 * (i + 0.5) / max(4, n)
            rho, phi = math.sqrt(1.0 - z * z), math.pi * (3.0 - math.sqrt(5.0)) * i
            d = [rho * math.cos(phi), rho * math.sin(phi), z]
            cam = dict(type="persp", W=W, H=H, eye=tuple(c + 2.0 * box * x for c, x in zip(centre, d)),
                       fwd=tuple(-x for x in d), up=(0.0, 0.0, 1.0), fov_y_deg=60.0)
        cams.append(cam)
    return cams


def _frames(case):
    """Cameras and the snapshot of each: every camera over every snapshot."""
    cams, S = _cameras(case), case.get("snaps", 1)
    return [c for _ in range(S) for c in cams], [s for s in range(S) for _ in cams]


def prepare(case, seed):
    kind, N, box = case["kind"], case["N"], case.get("box", 1.0)
    pos = _positions(case, seed)
    state = dict(case=case, kind=kind, pos=pos)
    state["r"] = r = Renderer(tile=case.get("tile", 0))
    if kind == "grad":
        # the image to fit: another lattice's, as an observation would be
        r.build_tets(_positions(case, seed + 500009), N, box)
        state["cams"] = _cameras(case)
        r.project_bin(state["cams"])
        state["target"] = r.render_tiles().clone()
        state["pos"] = pos[0].requires_grad_(True)
        return state
    if kind == "build":
        state["rho"] = torch.empty((case["snaps"], 6 * N ** 3), dtype=torch.float32, device="cuda")
        return state
    r.build_tets(pos, N, box)
    if kind == "movie":
        state["cams"], snaps = _frames(case)
        state["image"] = torch.empty((len(snaps), case["H"], case["W"]), dtype=torch.float32, device="cuda")
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        r.graph_build(state["cams"], frame_snapshot=snaps, image=state["image"], stream=side)
        torch.cuda.current_stream().wait_stream(side)
    elif "W" in case:
        state["cams"] = _cameras(case)
    return state


def run(state):
    case, kind, r = state["case"], state["kind"], state["r"]
    if kind == "frame":
        r.project_bin(state["cams"])
        return r.render_tiles()
    if kind == "movie":
        r.graph_launch()
        return state["image"]
    if kind == "grad":
        img = lt_render(state["pos"], case["N"], state["cams"], renderer=r, box=case.get("box", 1.0))
        loss = ((img - state["target"]) ** 2).sum()
        (grad,) = torch.autograd.grad(loss, state["pos"])
        return {"image": img.detach(), "grad": grad}
    if kind == "build":
        r.build_tets(state["pos"], case["N"], case.get("box", 1.0), rho_out=state["rho"])
        return state["rho"]
    if kind == "resample":
        return r.resample(case["n"], weight=case["weight"])
    if kind == "slice":
        return r.slice(case["n"], _plane(case), weight=case["weight"])
    if kind == "centroids":
        return r.render_centroids(state["cams"][0])
    if kind == "hybrid":
        return r.render_hybrid(state["cams"][0], case["near"] * case.get("box", 1.0))
    return r.render_area(state["cams"][0])


def _plane(case):
    return 0.37 * case.get("box", 1.0)


# ---------------------------------------------------------------------------
# what a pass cannot do without


def work(case):
    """Positions read once and results written once; the operations of the
    fragments (tetrahedron, pixel): about 0.42 cell faces per tetrahedron in
    projection, 12 operations each seen orthographically, 22 in perspective."""
    kind, N, S = case["kind"], case["N"], case.get("snaps", 1)
    tets = 6 * N ** 3
    pos = N ** 3 * (8 if case.get("half", False) else 16) * S
    if kind == "build":
        return dict(bytes=pos + 4 * tets * S, flops=40 * tets * S)
    if kind == "resample":
        n = case["n"]
        return dict(bytes=pos + 4 * n ** 3, flops=24 * 0.33 * tets * (n / N) ** 2 + 5 * n ** 3)
    if kind == "slice":
        n = case["n"]
        return dict(bytes=pos + 4 * n * n, flops=6 * N ** 3 + 24 * 4 * n * n)
    px = case["W"] * case["H"]
    n_frames = case.get("cams", 1) * S
    view = case.get("view", "persp")
    cover = {"z": 1.0, "oblique": 0.76}.get(view, 0.25 * case["H"] / case["W"])  # pixels of a box face over all pixels
    frags = 0.42 * tets * max(px * cover / N ** 2, 0.1) * n_frames
    per = 22 if view == "persp" else 12
    nbytes = pos + 4 * px * n_frames
    if kind == "grad":
        return dict(bytes=2 * nbytes + 16 * N ** 3, flops=2 * per * frags)
    return dict(bytes=nbytes, flops=per * frags)


# ---------------------------------------------------------------------------
# the same quantities in FP64, with plain torch operations

# the six tetrahedra of a cube; corner n is (n & 1, n >> 1 & 1, n >> 2 & 1)
_TETS = ((1, 0, 2, 4), (3, 1, 2, 4), (3, 5, 1, 4), (3, 6, 5, 4), (3, 2, 6, 4), (3, 7, 5, 6))
_PAIRS = 1 << 24  # (tetrahedron, pixel) pairs at a time


def _displacements(pos, N, box):
    """FP64 displacements from the lattice points of one snapshot, [N^3][3]."""
    boxf = float(torch.tensor(box, dtype=torch.float32))
    if pos.dtype == torch.float16:
        # the offsets times the cell edge, which the renderer keeps in FP32
        hf = torch.tensor(box, dtype=torch.float32) / N
        return (pos[:, :3].to(torch.float32) * hf.to(pos.device)).to(torch.float64)
    d = pos[:, :3].to(torch.float64) - _lattice(N, box)
    return torch.where(d > 0.5 * boxf, d - boxf, torch.where(d < -0.5 * boxf, d + boxf, d))


def _cube_chunks(N, size=1 << 18):
    for a in range(0, N ** 3, size):
        yield torch.arange(a, min(a + size, N ** 3), device="cuda")


def _corner_ids(cubes, N):
    i, j, k = cubes % N, (cubes // N) % N, cubes // (N * N)
    ids, offs = [], []
    for n in range(8):
        a, b, c = n & 1, (n >> 1) & 1, (n >> 2) & 1
        ids.append((i + a) % N + N * ((j + b) % N + N * ((k + c) % N)))
        offs.append(torch.stack([i + a, j + b, k + c], dim=-1))
    return torch.stack(ids, dim=1), torch.stack(offs, dim=1)


def _vertices(disp, cubes, N, box):
    """Unwrapped vertices of the cubes' tetrahedra, [6 C][4][3], in id order."""
    h = float(torch.tensor(box, dtype=torch.float32)) / N
    ids, offs = _corner_ids(cubes, N)
    corners = offs.to(torch.float64) * h + disp[ids]
    table = torch.tensor(_TETS, device=corners.device)
    return corners[:, table].reshape(-1, 4, 3)


def _volume(v):
    a, b, c = v[:, 1] - v[:, 0], v[:, 2] - v[:, 0], v[:, 3] - v[:, 0]
    return (a * torch.linalg.cross(b, c)).sum(-1) / 6.0


def _faces(v):
    """Outward normals and a point of each face, [T][4][3]."""
    n, p = [], []
    for f in range(4):
        a, b, c = v[:, (f + 1) & 3], v[:, (f + 2) & 3], v[:, (f + 3) & 3]
        m = torch.linalg.cross(b - a, c - a)
        side = (m * (v[:, f] - a)).sum(-1, keepdim=True)
        n.append(torch.where(side > 0, -m, m))
        p.append(a)
    return torch.stack(n, dim=1), torch.stack(p, dim=1)


def _t(v):
    return torch.tensor(v, dtype=torch.float64, device="cuda")


def _pixels(lo, hi, size, wrap):
    a, b = torch.ceil(lo), torch.floor(hi)
    if not wrap:
        a, b = a.clamp(0, size), b.clamp(-1, size - 1)
    return a.to(torch.int64), b.to(torch.int64)


def _expand(x0, x1, y0, y1, weight=1):
    """(tetrahedron, x, y) for every pixel of every rectangle, at most about _PAIRS at a time."""
    wx, wy = (x1 - x0 + 1).clamp_min(0), (y1 - y0 + 1).clamp_min(0)
    count = wx * wy
    keep = torch.nonzero(count).reshape(-1)
    total = torch.cumsum(count[keep], 0)
    at, done = 0, 0
    while at < keep.numel():
        end = int(torch.searchsorted(total, done + _PAIRS // weight, right=True))
        end = min(max(end, at + 1), keep.numel())
        ids = keep[at:end]
        c = count[ids]
        t = torch.repeat_interleave(ids, c)
        first = torch.cumsum(c, 0) - c
        q = torch.arange(t.numel(), device=t.device) - torch.repeat_interleave(first, c)
        w = wx[t]
        yield t, x0[t] + q % w, y0[t] + q // w
        done = int(total[end - 1])
        at = end


def _add(image, x, y, val):
    H, W = image.shape
    image.reshape(-1).index_add_(0, (y % H) * W + x % W, val)


def _view(cam, box):
    r, u, f = _axes(cam)
    if cam["type"] == "ortho":
        px = [(cam["hi"][q] - cam["lo"][q]) / (cam["W"], cam["H"])[q] for q in range(2)]
        return dict(persp=False, r=_t(r), u=_t(u), f=_t(f), lo=cam["lo"], px=px, wrap=bool(cam.get("wrap", False)))
    ty = math.tan(0.5 * cam["fov_y_deg"] * math.pi / 180.0)
    return dict(persp=True, r=_t(r), u=_t(u), f=_t(f), eye=_t(cam["eye"]), tan=(ty * cam["W"] / cam["H"], ty), wrap=False)


def _project(V, p, W, H):
    """Pixel coordinates (a pixel's centre at its whole number) and depth of points [..][3]."""
    if not V["persp"]:
        return (p @ V["r"] - V["lo"][0]) / V["px"][0] - 0.5, (p @ V["u"] - V["lo"][1]) / V["px"][1] - 0.5, None
    e = p - V["eye"]
    z = e @ V["f"]
    return (e @ V["r"] / z / V["tan"][0] + 1.0) * 0.5 * W - 0.5, (e @ V["u"] / z / V["tan"][1] + 1.0) * 0.5 * H - 0.5, z


def _face_lines(V, v, x0, y0, W, H):
    """Entry and exit parameters along the ray of pixel (x0 + i, y0 + j): for
    face f, num (affine in the pixel) over den; [T][4] each of the
    coefficients (num0, numx, numy, den0, denx, deny)."""
    n, a = _faces(v)
    nr, nu, nf = n @ V["r"], n @ V["u"], n @ V["f"]
    zero = torch.zeros_like(nr)
    if not V["persp"]:
        wa = V["lo"][0] + (x0.to(torch.float64) + 0.5) * V["px"][0]
        wb = V["lo"][1] + (y0.to(torch.float64) + 0.5) * V["px"][1]
        o = wa[:, None] * V["r"] + wb[:, None] * V["u"]
        num = (n * (a - o[:, None])).sum(-1)
        return num, -nr * V["px"][0], -nu * V["px"][1], nf, zero, zero
    sx, sy = 2.0 * V["tan"][0] / W, 2.0 * V["tan"][1] / H
    xt = (x0.to(torch.float64) + 0.5) * sx - V["tan"][0]
    yt = (y0.to(torch.float64) + 0.5) * sy - V["tan"][1]
    den = nf + nr * xt[:, None] + nu * yt[:, None]
    return (n * (a - V["eye"])).sum(-1), zero, zero, den, nr * sx, nu * sy


def _chords(L, t, i, j, persp):
    """Ray parameter where pixel (x0 + i, y0 + j) enters and leaves tetrahedron t, and the faces."""
    big = 1e300
    t_in = torch.full(t.shape, 0.0 if persp else -big, dtype=torch.float64, device=t.device)
    t_out = torch.full_like(t_in, big)
    f_in, f_out = torch.zeros_like(t), torch.zeros_like(t)
    for f in range(4):
        num, den = L[0][t, f], L[3][t, f]
        if persp:
            den = den + L[4][t, f] * i + L[5][t, f] * j
        else:
            num = num + L[1][t, f] * i + L[2][t, f] * j
        s = num / den
        out = (den > 0) & (s < t_out)
        inn = (den < 0) & (s > t_in)
        t_out, f_out = torch.where(out, s, t_out), torch.where(out, torch.full_like(t, f), f_out)
        t_in, f_in = torch.where(inn, s, t_in), torch.where(inn, torch.full_like(t, f), f_in)
        t_out = torch.where((den == 0) & (num < 0), torch.full_like(t_out, -big), t_out)
    return t_in, t_out, f_in, f_out


def _render(case, pos, cam, near=None):
    """Column density at the pixel centres, [H][W] float64; with `near` only the cubes within it of the eye."""
    N, box, W, H = case["N"], case.get("box", 1.0), cam["W"], cam["H"]
    V = _view(cam, box)
    disp = _displacements(pos, N, box)
    image = torch.zeros((H, W), dtype=torch.float64, device="cuda")
    m = 1.0 / (6.0 * N ** 3)
    for cubes in _cube_chunks(N):
        if near is not None:
            cubes = cubes[_near(case, disp, cubes, V, near)]
            if not cubes.numel():
                continue
        v = _vertices(disp, cubes, N, box)
        vol = _volume(v).abs()
        rho = torch.where(vol > 0, m / vol, torch.zeros_like(vol))
        x, y, _ = _project(V, v, W, H)
        x0, x1 = _pixels(x.amin(1), x.amax(1), W, V["wrap"])
        y0, y1 = _pixels(y.amin(1), y.amax(1), H, V["wrap"])
        L = _face_lines(V, v, x0, y0, W, H)
        for t, px, py in _expand(x0, x1, y0, y1):
            t_in, t_out, _, _ = _chords(L, t, px - x0[t], py - y0[t], V["persp"])
            _add(image, px, py, rho[t] * (t_out - t_in).clamp_min(0.0))
    return image * _ray_length(V, W, H) if V["persp"] else image


def _ray_length(V, W, H):
    xt = V["tan"][0] * (2.0 * (torch.arange(W, device="cuda", dtype=torch.float64) + 0.5) / W - 1.0)
    yt = V["tan"][1] * (2.0 * (torch.arange(H, device="cuda", dtype=torch.float64) + 0.5) / H - 1.0)
    return torch.sqrt(1.0 + xt[None, :] ** 2 + yt[:, None] ** 2)


def _near(case, disp, cubes, V, near):
    p = _lattice(case["N"], case.get("box", 1.0))[cubes] + disp[cubes]
    return ((p - V["eye"]) ** 2).sum(-1) < near * near


def _splats(case, pos, cam, near=None):
    """Centroid splats, [H][W] float64; with `near` only the cubes beyond it."""
    N, box, W, H = case["N"], case.get("box", 1.0), cam["W"], cam["H"]
    V = _view(cam, box)
    disp = _displacements(pos, N, box)
    image = torch.zeros((H, W), dtype=torch.float64, device="cuda")
    m = 1.0 / (6.0 * N ** 3)
    for cubes in _cube_chunks(N):
        if near is not None:
            cubes = cubes[~_near(case, disp, cubes, V, near)]
            if not cubes.numel():
                continue
        v = _vertices(disp, cubes, N, box)
        vol = _volume(v).abs()
        h = vol ** (1.0 / 3.0)
        x, y, z = _project(V, v.mean(1), W, H)
        if V["persp"]:
            sx, sy = z * (2.0 * V["tan"][0] / W), z * (2.0 * V["tan"][1] / H)
        else:
            sx, sy = torch.full_like(h, V["px"][0]), torch.full_like(h, V["px"][1])
        x0, x1 = _pixels(x - 2.0 * h / sx, x + 2.0 * h / sx, W, V["wrap"])
        y0, y1 = _pixels(y - 2.0 * h / sy, y + 2.0 * h / sy, H, V["wrap"])
        x1 = torch.where(vol > 0, x1, x0 - 1)
        for t, px, py in _expand(x0, x1, y0, y1):
            q = torch.sqrt(((px - x[t]) * sx[t]) ** 2 + ((py - y[t]) * sy[t]) ** 2) / h[t]
            w = torch.where(q < 1.0, 1.0 - 1.5 * q * q + 0.75 * q ** 3, 0.25 * (2.0 - q).clamp_min(0.0) ** 3)
            _add(image, px, py, m * 10.0 / (7.0 * math.pi) * w / h[t] ** 2)
    return image * _ray_length(V, W, H) if V["persp"] else image


def _gradient(case, pos, cam, g):
    """d (sum g I) / d position of one orthographic view, [N^3][3] float64.
    The chord of a ray is the difference of two functions affine in the pixel
    (exit and entry face), so the pixels enter through three moments per face."""
    N, box, W, H = case["N"], case.get("box", 1.0), cam["W"], cam["H"]
    V = _view(cam, box)
    disp = _displacements(pos, N, box)
    grad = torch.zeros((N ** 3, 3), dtype=torch.float64, device="cuda")
    m = 1.0 / (6.0 * N ** 3)
    h = float(torch.tensor(box, dtype=torch.float32)) / N
    table = torch.tensor(_TETS, device="cuda")
    for cubes in _cube_chunks(N):
        ids, offs = _corner_ids(cubes, N)
        corners = (offs.to(torch.float64) * h + disp[ids]).requires_grad_(True)
        with torch.enable_grad():
            v = corners[:, table].reshape(-1, 4, 3)
            rho = m / _volume(v).abs()
            x, y, _ = _project(V, v.detach(), W, H)
            x0, x1 = _pixels(x.amin(1), x.amax(1), W, V["wrap"])
            y0, y1 = _pixels(y.amin(1), y.amax(1), H, V["wrap"])
            L = _face_lines(V, v, x0, y0, W, H)
        D = [q.detach() for q in L]
        mom = torch.zeros((3, v.shape[0] * 4), dtype=torch.float64, device="cuda")
        for t, px, py in _expand(x0, x1, y0, y1):
            i, j = px - x0[t], py - y0[t]
            t_in, t_out, f_in, f_out = _chords(D, t, i, j, False)
            gv = torch.where(t_out > t_in, g[py % H, px % W], torch.zeros_like(t_in))
            for q, w in enumerate((gv, gv * i, gv * j)):
                mom[q].index_add_(0, t * 4 + f_out, w)
                mom[q].index_add_(0, t * 4 + f_in, -w)
        mom = mom.reshape(3, -1, 4)
        with torch.enable_grad():
            ok = D[3] != 0
            den = torch.where(ok, L[3], torch.ones_like(L[3]))
            total = (rho[:, None] * torch.where(ok, (L[0] * mom[0] + L[1] * mom[1] + L[2] * mom[2]) / den, torch.zeros_like(den))).sum()
            (gc,) = torch.autograd.grad(total, corners)
        grad.index_add_(0, ids.reshape(-1), gc.reshape(-1, 3))
    return grad


def _hull(x, y):
    """Hull vertices [T][4] (counter-clockwise; a triangle's last one twice)
    and the apex of projected tetrahedra."""
    def orient(a, b, c):
        return (x[:, b] - x[:, a]) * (y[:, c] - y[:, a]) - (y[:, b] - y[:, a]) * (x[:, c] - x[:, a])

    s = torch.stack([orient(1, 2, 3), -orient(0, 2, 3), orient(0, 1, 3), -orient(0, 1, 2)], dim=1) > 0
    pos = s.sum(1)
    # a lone sign: that vertex lies inside the triangle of the others
    lone = torch.where((pos == 1)[:, None], s, ~s).to(torch.int64).argmax(1)
    other = torch.tensor([[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]], device=x.device)[lone]
    tri = torch.cat([other, other[:, 2:]], dim=1)
    # two of each: vertices of one sign are the ends of a diagonal
    order = torch.argsort(s.to(torch.int64), dim=1, stable=True)
    quad = order[:, [0, 2, 1, 3]]
    two = pos == 2
    idx = torch.where(two[:, None], quad, tri)
    hx, hy = torch.gather(x, 1, idx), torch.gather(y, 1, idx)
    # the crossing of the diagonals (0, 2) and (1, 3)
    dx, dy = hx[:, 2] - hx[:, 0], hy[:, 2] - hy[:, 0]
    ex, ey = hx[:, 3] - hx[:, 1], hy[:, 3] - hy[:, 1]
    den = dx * ey - dy * ex
    q = ((hx[:, 1] - hx[:, 0]) * ey - (hy[:, 1] - hy[:, 0]) * ex) / torch.where(den == 0, torch.ones_like(den), den)
    ax = torch.where(two, hx[:, 0] + q * dx, torch.gather(x, 1, lone[:, None])[:, 0])
    ay = torch.where(two, hy[:, 0] + q * dy, torch.gather(y, 1, lone[:, None])[:, 0])
    nx, ny = torch.roll(hx, -1, 1), torch.roll(hy, -1, 1)
    area2 = (hx * ny - hy * nx).sum(1)
    return hx, hy, ax, ay, area2


def _beside(xa, ya, xb, yb, a, b, c):
    """The integral of a x + b y + c over the part of the unit square to the
    right of the edge (xa, ya) -> (xb, yb), signed by its direction in y. The
    inner integral is cubic in y on each stretch between the edge's crossings
    of x = 0 and x = 1, so two Gauss points are exact."""
    lo, hi = torch.minimum(ya, yb).clamp(0, 1), torch.maximum(ya, yb).clamp(0, 1)
    dy = yb - ya
    slope = (xb - xa) / torch.where(dy == 0, torch.ones_like(dy), dy)
    back = dy / torch.where(xb == xa, torch.ones_like(dy), xb - xa)
    cut = [torch.where(xb == xa, lo, ya + (e - xa) * back) for e in (0.0, 1.0)]
    y1, y2 = torch.minimum(*cut).clamp_min(lo).clamp_max(hi), torch.maximum(*cut).clamp_min(lo).clamp_max(hi)
    total = torch.zeros_like(xa)
    for p, q in ((lo, y1), (y1, y2), (y2, hi)):
        mid, half = 0.5 * (p + q), 0.5 * (q - p)
        for s in (-1.0, 1.0):
            yy = mid + s * half / math.sqrt(3.0)
            xx = (xa + (yy - ya) * slope).clamp(0, 1)
            total = total + half * ((b * yy + c) * (1.0 - xx) + 0.5 * a * (1.0 - xx * xx))
    return torch.where(dy > 0, total, torch.where(dy < 0, -total, torch.zeros_like(total)))


def _area(case, pos, cam):
    """Mean column density over each pixel's square, [H][W] float64."""
    N, box, W, H = case["N"], case.get("box", 1.0), cam["W"], cam["H"]
    V = _view(cam, box)
    disp = _displacements(pos, N, box)
    image = torch.zeros((H, W), dtype=torch.float64, device="cuda")
    m = 1.0 / (6.0 * N ** 3)
    for cubes in _cube_chunks(N):
        v = _vertices(disp, cubes, N, box)
        x, y, _ = _project(V, v, W, H)
        x, y = x + 0.5, y + 0.5  # pixel p covers [p, p + 1]
        bx, by = torch.floor(x[:, :1]), torch.floor(y[:, :1])
        hx, hy, ax, ay, area2 = _hull(x - bx, y - by)
        x0, x1 = torch.floor(x.amin(1)), torch.floor(x.amax(1))
        y0, y1 = torch.floor(y.amin(1)), torch.floor(y.amax(1))
        if not V["wrap"]:
            x0, x1, y0, y1 = x0.clamp_min(0), x1.clamp_max(W - 1), y0.clamp_min(0), y1.clamp_max(H - 1)
        top = 3.0 * m / (0.5 * area2.abs() * V["px"][0] * V["px"][1])
        # the linear function of each sector: `top` at the apex, 0 along the hull edge
        ex, ey = torch.roll(hx, -1, 1) - hx, torch.roll(hy, -1, 1) - hy
        d = ex * (ay[:, None] - hy) - ey * (ax[:, None] - hx)
        ok = (d != 0) & (_volume(v) != 0)[:, None]
        k = torch.where(ok, top[:, None] / torch.where(ok, d, torch.ones_like(d)), torch.zeros_like(d))
        a, b, c = -ey * k, ex * k, (ey * hx - ex * hy) * k
        sign = torch.where(d > 0, 1.0, -1.0).to(torch.float64)  # the sector's sense of rotation
        for t, px, py in _expand(*(q.to(torch.int64) for q in (x0, x1, y0, y1)), weight=4):
            ox, oy = px - bx[t, 0], py - by[t, 0]
            val = torch.zeros_like(ox)
            for e in range(4):
                f = (e + 1) & 3
                cc = c[t, e] + a[t, e] * ox + b[t, e] * oy
                P = [(ax[t] - ox, ay[t] - oy), (hx[t, e] - ox, hy[t, e] - oy), (hx[t, f] - ox, hy[t, f] - oy)]
                s = 0.0
                for q in range(3):
                    s = s - _beside(*P[q], *P[(q + 1) % 3], a[t, e], b[t, e], cc)
                val = val + sign[t, e] * s
            _add(image, px.to(torch.int64), py.to(torch.int64), val)
    return image


def _resample(case, pos):
    N, box, n = case["N"], case.get("box", 1.0), case["n"]
    g = float(torch.tensor(box, dtype=torch.float32)) / n
    cam = dict(type="ortho", W=n, H=n, fwd=(0, 0, 1), up=(0, 1, 0), lo=(0.0, 0.0), hi=(g * n, g * n), wrap=True)
    V = _view(cam, box)
    disp = _displacements(pos, N, box)
    grid = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    m = 1.0 / (6.0 * N ** 3)
    for cubes in _cube_chunks(N):
        v = _vertices(disp, cubes, N, box)
        vol = _volume(v).abs()
        w = torch.where(vol > 0, m / vol if case["weight"] == "density" else torch.ones_like(vol), torch.zeros_like(vol))
        x, y, _ = _project(V, v, n, n)
        x0, x1 = _pixels(x.amin(1), x.amax(1), n, True)
        y0, y1 = _pixels(y.amin(1), y.amax(1), n, True)
        L = _face_lines(V, v, x0, y0, n, n)
        for t, px, py in _expand(x0, x1, y0, y1):
            z_in, z_out, _, _ = _chords(L, t, px - x0[t], py - y0[t], False)
            some = torch.nonzero((z_out > z_in) & (w[t] > 0)).reshape(-1)
            t, px, py, z_in, z_out = t[some], px[some] % n, py[some] % n, z_in[some], z_out[some]
            c = torch.floor(z_in / g)
            while t.numel():
                part = (torch.minimum(z_out, (c + 1) * g) - torch.maximum(z_in, c * g)).clamp_min(0.0)
                grid.index_add_(0, ((c.to(torch.int64) % n) * n + py) * n + px, w[t] * part)
                more = torch.nonzero((c + 1) * g < z_out).reshape(-1)
                t, px, py, z_in, z_out, c = t[more], px[more], py[more], z_in[more], z_out[more], c[more] + 1
    return grid.reshape(n, n, n)


def _slice(case, pos):
    N, box, n = case["N"], case.get("box", 1.0), case["n"]
    boxf = float(torch.tensor(box, dtype=torch.float32))
    g = boxf / n
    disp = _displacements(pos, N, box)
    image = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    m = 1.0 / (6.0 * N ** 3)
    for cubes in _cube_chunks(N):
        v = _vertices(disp, cubes, N, box)
        for copy in (-1, 0, 1):
            z0 = _plane(case) + copy * boxf
            hit = (v[..., 2].amin(1) <= z0) & (v[..., 2].amax(1) >= z0)
            if not bool(hit.any()):
                continue
            u = v[hit]
            vol = _volume(u).abs()
            w = torch.where(vol > 0, m / vol if case["weight"] == "density" else torch.ones_like(vol), torch.zeros_like(vol))
            x0, x1 = _pixels(u[..., 0].amin(1) / g - 0.5, u[..., 0].amax(1) / g - 0.5, n, True)
            y0, y1 = _pixels(u[..., 1].amin(1) / g - 0.5, u[..., 1].amax(1) / g - 0.5, n, True)
            nrm, pt = _faces(u)
            off = (nrm * pt).sum(-1)
            for t, px, py in _expand(x0, x1, y0, y1):
                p = torch.stack([(px + 0.5) * g, (py + 0.5) * g, torch.full_like(px, 1, dtype=torch.float64) * z0], dim=-1)
                inside = torch.ones_like(t, dtype=torch.bool)
                for f in range(4):
                    inside &= (nrm[t, f] * p).sum(-1) <= off[t, f]
                _add(image, px, py, torch.where(inside, w[t], torch.zeros_like(w[t])))
    return image


@torch.no_grad()
def exact(case, seed):
    kind, N, box = case["kind"], case["N"], case.get("box", 1.0)
    pos = _positions(case, seed)
    if kind == "build":
        out = torch.empty((case["snaps"], 6 * N ** 3), dtype=torch.float64, device="cuda")
        for s in range(case["snaps"]):
            disp = _displacements(pos[s], N, box)
            for cubes in _cube_chunks(N):
                vol = _volume(_vertices(disp, cubes, N, box)).abs()
                out[s, 6 * int(cubes[0]):6 * int(cubes[-1]) + 6] = torch.where(vol > 0, 1.0 / (6.0 * N ** 3) / vol, torch.zeros_like(vol))
        return out
    if kind == "resample":
        return _resample(case, pos[0])
    if kind == "slice":
        return _slice(case, pos[0])
    cams = _cameras(case)
    if kind == "grad":
        target = _positions(case, seed + 500009)
        images = [_render(case, pos[0], c) for c in cams]
        # the target is what prepare() hands over: its pixels in FP32
        grad = sum(_gradient(case, pos[0], c, 2.0 * (im - _render(case, target[0], c))) for c, im in zip(cams, images))
        return {"image": torch.stack(images), "grad": torch.cat([grad, torch.zeros_like(grad[:, :1])], dim=1)}
    if kind == "centroids":
        return _splats(case, pos[0], cams[0])
    if kind == "hybrid":
        near = case["near"] * box
        return _render(case, pos[0], cams[0], near) + _splats(case, pos[0], cams[0], near)
    if kind == "area":
        return _area(case, pos[0], cams[0])
    cams, snaps = _frames(case)
    return torch.stack([_render(case, pos[s], c) for c, s in zip(cams, snaps)])
