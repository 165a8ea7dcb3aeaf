"""The kernels at the sizes where their work split can go wrong: lattices that
do not fill a warp, a block or a group of blocks, odd snapshot strides, boxes
whose cell edge rounds, tetrahedra of zero volume, and the smallest and
odd-sized grids, against FP64 (numpy or the oracle).
"""
import numpy as np
import pytest

import oracle
from lt_inputs import ZeldovichField, fp16_offsets

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TETS = np.array([[1, 0, 2, 4], [3, 1, 2, 4], [3, 5, 1, 4], [3, 6, 5, 4], [3, 2, 6, 4], [3, 7, 5, 6]])


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    return Renderer()


def lattice(N, lam, seed, box=1.0):
    if N < 4:  # too small for the generator's spectrum
        rng = np.random.default_rng(seed)
        d = rng.uniform(-0.2, 0.2, (N ** 3, 3)) * lam / N
    else:
        d = ZeldovichField.generate(N, -2.0, 0.375 * N, seed).displacement(lam)
    return d  # in units of a unit box, [N^3][3]


def wrapped(d, N, box):
    i = np.arange(N ** 3)
    q = np.stack([i % N, (i // N) % N, i // (N * N)], axis=1) * (box / N)
    x = np.mod(q + d * box, box).astype(np.float32)
    out = np.zeros((N ** 3, 4), dtype=np.float32)
    out[:, :3] = np.where(x >= np.float32(box), np.float32(0), x)
    return out


def volumes(disp, N, h):
    """Signed volumes [6 N^3] from FP64 displacements and the cell edge h."""
    c = np.arange(N ** 3)
    i, j, k = c % N, (c // N) % N, c // (N * N)
    corner = []
    for n in range(8):
        a, b, e = n & 1, (n >> 1) & 1, n >> 2
        idx = (i + a) % N + N * ((j + b) % N + N * ((k + e) % N))
        corner.append(disp[idx] + np.array([a, b, e]) * h)
    v = np.stack(corner, axis=1)[:, TETS]  # [N^3][6][4][3]
    e = v[:, :, 1:] - v[:, :, :1]
    return (np.einsum("tsa,tsa->ts", e[:, :, 0], np.cross(e[:, :, 1], e[:, :, 2])) / 6.0).reshape(-1)


def unwrapped(pos, N, box):
    i = np.arange(N ** 3)
    q = np.stack([i % N, (i // N) % N, i // (N * N)], axis=1) * (box / N)
    d = pos[:, :3].astype(np.float64) - q
    return d - box * np.round(d / box)


def decoded(off, N):
    """The positions that FP16 offsets stand for in a unit box: the offset
    times the cell edge as the renderer holds it, in FP32."""
    i = np.arange(N ** 3)
    q = np.stack([i % N, (i // N) % N, i // (N * N)], axis=1) / N
    return np.mod(q + (off[:, :3].astype(np.float32) * (np.float32(1) / np.float32(N))).astype(np.float64), 1.0)


@pytest.mark.parametrize("N,box,half,snaps", [(1, 1.0, False, 1), (2, 1.0, False, 3), (3, 1.0, False, 2), (7, 100.0, False, 3),
                                              (8, 1.0, True, 1), (16, 1.0, False, 2), (33, 1.0, False, 1),
                                              (33, 40.0, True, 2), (64, 1.0, False, 1)])
def test_densities(R, N, box, half, snaps):
    """Densities of every tetrahedron. The FP32 determinant of a volume above
    0.1 h^3 is off by a few 2^-24 of the product of its edges (here below
    4^3 h^3): 1e-4 relative. Smaller volumes come from exact edges: FP32's
    rounding of the density (2^-24) and what h = box / N, a rounded number
    off a power of two, moves the edges that wrap by (2^-24 N h each). Both
    sides' FP64 determinants round by 64 h^3 2^-49, which hides the density's
    last bit below 2^-20 h^3; whether a volume is zero is compared where the
    products are exact in FP64 (11-bit offsets)."""
    pos, ref, zero = [], [], 0
    hf = np.float32(box) / np.float32(N)
    for s in range(snaps):
        d = lattice(N, 2.5, 11 + s)
        # tetrahedra of exactly zero volume (N >= 8): a particle on its neighbour
        if half:
            p = fp16_offsets(d, N)
            if N >= 8:
                p[6] = (0.25, -0.5, 0.125, 0)
                p[5] = (1.25, -0.5, 0.125, 0)
            disp = (p[:, :3].astype(np.float32) * hf).astype(np.float64)
            h = float(hf)
        else:
            p = wrapped(d, N, box)
            if N >= 8:
                p[5] = p[6]
            disp, h = unwrapped(p, N, box), box / N
        v = volumes(disp, N, h)
        pos.append(p)
        ref.append(v)
        zero += int((v == 0).sum())
    pos, v = np.stack(pos), np.stack(ref)
    out = torch.full((snaps, 6 * N ** 3), -1.0, dtype=torch.float32, device="cuda")
    R.build_tets(torch.from_numpy(pos).cuda(), N, box, rho_out=out)
    st = R.get_stats()
    got = out.cpu().numpy().astype(np.float64)
    with np.errstate(divide="ignore"):
        rho = 1.0 / (6.0 * N ** 3) / np.abs(v)
    h3 = (box / N) ** 3
    small = np.abs(v) < 0.0999 * h3
    exact = (N & (N - 1)) == 0
    tol = np.where(small, 2.0 ** -23, 1e-4) + (0.0 if exact else 1.0) * 64 * 2.0 ** -24 * N * h3 / np.maximum(np.abs(v), 1e-300)
    ok = np.abs(v) > (2.0 ** -20 if exact else 1e-3) * h3
    assert np.all(np.abs(got - rho)[ok] <= (tol * rho)[ok])
    if exact and half:
        assert zero > 0
        assert st["degenerate"] == zero
        assert np.all(got[v == 0] == 0)
        assert st["inverted"] == int((v > 0).sum())


@pytest.mark.parametrize("N,n,z0,half", [(1, 3, 0.3, False), (2, 1, 0.4, False), (5, 33, -0.21, False), (9, 31, 7.77, False),
                                         (16, 200, 0.999, True), (11, 64, 0.013, False)])
@pytest.mark.parametrize("weight", ["streams", "density"])
def test_slices(R, N, n, z0, half, weight):
    """Slice points against the oracle: counts equal, densities to 1e-5 (FP64
    volumes on both sides, sums of 2^-28 of the mean and FP32's rounding)."""
    d = lattice(N, 1.7, 5)
    if half:
        p = fp16_offsets(d, N)
        ref_pos = decoded(p, N)
    else:
        p = ref_pos = wrapped(d, N, 1.0)
    R.build_tets(torch.from_numpy(p).cuda(), N)
    got = R.slice(n, z0, weight).cpu().numpy().astype(np.float64).ravel()
    R.sync()
    a = (np.arange(n) + 0.5) / n
    X, Y = np.meshgrid(a, a)
    pts = np.stack([X.ravel(), Y.ravel(), np.full(n * n, z0 - np.floor(z0))], axis=1)
    ref = oracle.point_density(ref_pos, N, pts, weight)
    if weight == "streams":
        assert np.array_equal(got, ref)
    else:
        assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(ref, 1.0))


def view(W, H, kind):
    if kind == "persp":
        return dict(type="persp", W=W, H=H, eye=(1.9, -0.8, 1.4), fwd=(-1.4, 1.3, -0.9), up=(0, 0, 1), fov_y_deg=50.0)
    return dict(type="ortho", W=W, H=H, fwd=(0, 0, 1), up=(0, 1, 0), lo=(0.0, 0.0), hi=(1.0, 1.0), wrap=True)


@pytest.mark.parametrize("kind", ["z", "persp"])
@pytest.mark.parametrize("N,W,H,tile,frac_bits", [(40, 33, 29, 64, 0), (40, 33, 29, 16, 0), (24, 130, 65, 32, 0), (24, 16, 16, 8, 0),
                                                  (12, 200, 3, 64, 0), (24, 70, 50, 16, 44), (5, 1, 1, 32, 0)])
def test_raster_items(kind, N, W, H, tile, frac_bits):
    """Tiles whose lists are split into several work items (a 33 x 29 frame of
    64000 cubes: 500 of them for one tile), ragged ones, one-pixel ones, and
    pixel sums past their low 32-bit word (44 fraction bits). Against the
    oracle at the raster's own bound (fragments beyond 1e-5 of max(value, mean)
    are exact; their sum stays within 1e-4), and twice bit for bit."""
    from paper_1208_3206_gb300.render import Renderer
    r = Renderer(tile=tile, frac_bits=frac_bits)
    p = wrapped(lattice(N, 2.0, 3), N, 1.0)
    cam = view(W, H, kind)
    r.build_tets(torch.from_numpy(p).cuda(), N)
    r.project_bin([cam, cam])
    img, mass = r.render_tiles(with_mass=True)
    again = r.render_tiles()
    r.sync()
    ref = oracle.render(p, N, cam)
    mean = ref[ref > 0].mean() if (ref > 0).any() else 1.0
    for f in range(2):
        got = img[f].cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - ref) <= 1e-4 * np.maximum(ref, mean))
    assert torch.equal(img, again) and torch.equal(img[0], img[1])
    area = 1.0 / (W * H) if kind == "z" else (2.0 * np.tan(np.radians(25.0)) / H) ** 2
    assert abs(float(mass[0]) - ref.sum() * area) <= 1e-5 * ref.sum() * area
    r.project_bin([cam])  # fewer tiles in the same buffers
    assert torch.equal(r.render_tiles()[0], img[0])


@pytest.mark.parametrize("W,H,tile", [(1024, 1024, 16), (1040, 1024, 16), (512, 512, 8), (64, 64, 64)])
def test_worklist_forms(W, H, tile):
    """4096 tiles (the work list of one block), more, and as many frames as make
    more; lists that grow from nothing, from those of fewer frames and of a
    smaller lattice, and that are too large. Sums are fixed-point: bit for bit."""
    from paper_1208_3206_gb300.render import Renderer
    cam = view(W, H, "persp")
    small, large = wrapped(lattice(8, 1.0, 5), 8, 1.0), wrapped(lattice(24, 2.0, 3), 24, 1.0)
    images = []
    for order in ([1], [1, 3], [3, 1], [0, 1]):
        r = Renderer(tile=tile)
        for frames in order:
            r.build_tets(torch.from_numpy(large if frames else small).cuda(), 24 if frames else 8)
            r.project_bin([cam] * max(frames, 1))
            img = r.render_tiles()
        r.sync()
        images += [x for x in img] if frames else []
    assert images[0].sum() > 0
    for x in images[1:]:
        assert torch.equal(x, images[0])


@pytest.mark.parametrize("N,W,H,kind,lam,half", [(1, 9, 7, "z", 0.5, False), (3, 40, 33, "z", 1.0, False), (13, 300, 7, "z", 2.0, False),
                                                 (49, 61, 50, "z", 3.0, False), (50, 64, 48, "persp", 2.0, False),
                                                 (16, 256, 256, "persp", 4.0, False), (20, 90, 80, "z", 6.0, True)])
def test_centroid_blocks(N, W, H, kind, lam, half):
    """Splats by blocks of the lattice: blocks that the lattice does not fill,
    several windows per block (splats of 100 pixels and more), blocks strewn by
    strong displacement, both block sizes, periodic copies. A pixel's sum is
    off by the FP32 spline (a few 2^-24 each) and 2^-28 of the mean: 1e-5."""
    from paper_1208_3206_gb300.render import Renderer
    r = Renderer()
    d = lattice(N, lam, 9)
    if half:
        p = fp16_offsets(d, N)
        ref_pos = decoded(p, N)
    else:
        p = ref_pos = wrapped(d, N, 1.0)
    cam = view(W, H, kind)
    r.build_tets(torch.from_numpy(p).cuda(), N)
    img = r.render_centroids(cam)
    again = r.render_centroids(cam)
    r.sync()
    ref = oracle.centroids(ref_pos, N, cam)
    got = img.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(ref, 1.0))
    assert torch.equal(img, again)


@pytest.mark.parametrize("frac_bits", [31, 34, 40])
def test_centroid_peaks(frac_bits):
    """Pixel sums of finer units than a window's 32-bit words hold: a few of
    the splats, most and all of them go to the image directly. Against the sums
    at the default 28 bits: a unit is 2^-28 of the mean, and half units of either
    sign from 10^5 splats in a pixel make 6e-7 of it (the FP32 values are the
    same on both routes); 1e-5 leaves a factor for the fullest pixel."""
    from paper_1208_3206_gb300.render import Renderer
    p = torch.from_numpy(wrapped(lattice(49, 3.0, 9), 49, 1.0)).cuda()
    images = []
    for bits in (0, frac_bits):
        r = Renderer(frac_bits=bits)
        r.build_tets(p, 49)
        images.append(r.render_centroids(view(150, 131, "z")))
        r.sync()
    assert (images[0] - images[1]).abs().max() <= 1e-5 * images[0].mean()


@pytest.mark.parametrize("N,n,lam,half", [(1, 4, 0.5, False), (2, 33, 1.0, False), (5, 1, 1.0, False), (6, 70, 2.0, False),
                                          (11, 24, 3.0, False), (33, 8, 3.0, False), (16, 40, 4.0, True), (12, 31, 0.0, False)])
@pytest.mark.parametrize("weight", ["density", "streams"])
def test_resample_forms(N, n, lam, half, weight):
    """Cells against the oracle: columns past the periodic edge, tetrahedra of
    hundreds of columns and cells and of fractions of one, the undeformed
    lattice (every face vertical or level) and FP16 lattices, whose flat
    tetrahedra take FP64. A cell's parts are rounded to 2^-28 of the mean cell
    and come from heights good to 2^-40: 1e-5 of max(cell, mean)."""
    from paper_1208_3206_gb300.render import Renderer
    r = Renderer()
    d = lattice(N, lam, 4) if lam > 0 else np.zeros((N ** 3, 3))
    if half:
        p = fp16_offsets(d, N)
        ref_pos = decoded(p, N)
    else:
        if lam == 0:
            d = d + np.array([0.0123, 0.0077, 0.0031])  # columns off the faces
        p = ref_pos = wrapped(d, N, 1.0)
    r.build_tets(torch.from_numpy(p).cuda(), N)
    grid = r.resample(n, weight)
    again = r.resample(n, weight)
    r.sync()
    ref = oracle.resample(ref_pos, N, n, weight)
    got = grid.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(ref, 1.0 / n))
    assert torch.equal(grid, again)


def test_resample_between_bin_and_render():
    """A grid needs no bins, but as ever the frames are binned again before they
    are rendered or counted; the adjoint of the binned frames stands."""
    from paper_1208_3206_gb300.render import Renderer
    N, cam = 8, view(32, 24, "z")
    r = Renderer()
    r.build_tets(torch.from_numpy(wrapped(lattice(N, 1.0, 2), N, 1.0)).cuda(), N)
    r.project_bin([cam])
    img = r.render_tiles()
    grad = r.render_backward(2.0 * img).clone()
    r.resample(16, "density")
    with pytest.raises(Exception):
        r.render_tiles(img)
    assert r._lib.lt_render_tiles(r._h, img.data_ptr(), None, None) != 0
    assert torch.equal(r.render_backward(2.0 * img), grad)
    r.project_bin([cam])
    assert torch.equal(r.render_tiles(), img)


@pytest.mark.parametrize("N,W,H,kind,lam", [(1, 5, 9, "z", 0.5), (2, 64, 64, "z", 1.0), (4, 300, 210, "z", 2.0), (9, 31, 3, "z", 3.0),
                                            (24, 20, 20, "z", 3.0), (16, 90, 70, "oblique", 4.0), (6, 41, 37, "z", 0.0)])
def test_area_stages(N, W, H, kind, lam):
    """Area-averaged pixels: tetrahedra of thousands of pixels and of fractions
    of one (squares that hold a whole hull, over several rays, over one, inside
    one sector), the undeformed lattice (apexes on hull vertices and edges).
    Lines are good to 2^-24 of a pixel and hulls are 0.05 pixels wide at least
    in FP32, so a tetrahedron's share is good to about 1e-5 and the pixel to
    1e-5 of max(pixel, mean)."""
    from paper_1208_3206_gb300.render import Renderer
    r = Renderer()
    d = lattice(N, lam, 6) if lam > 0 else np.zeros((N ** 3, 3))
    p = wrapped(d, N, 1.0)
    cam = view(W, H, "z")
    if kind == "oblique":
        cam = dict(type="ortho", W=W, H=H, fwd=(1.0, 2.0, 2.5), up=(0, 0, 1), lo=(-0.4, -0.6), hi=(0.8, 0.7), wrap=False)
    r.build_tets(torch.from_numpy(p).cuda(), N)
    img = r.render_area(cam)
    again = r.render_area(cam)
    r.sync()
    ref = oracle.render_area(p, N, cam)
    got = img.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(ref, 1.0))
    assert torch.equal(img, again)


@pytest.mark.parametrize("N,W,H,snaps", [(1, 9, 9, 1), (3, 33, 20, 2), (7, 64, 50, 2), (18, 40, 61, 1)])
def test_backward_blocks(R, N, W, H, snaps):
    """The adjoint over lattices that do not fill a block of 32 cubes, several
    snapshots and frames (one snapshot seen twice, periodic and oblique): the
    repository's bound for gradients, 1e-3 of the oracle's in the 2-norm."""
    p = [wrapped(lattice(N, 1.2, 20 + s), N, 1.0) for s in range(snaps)]
    cams = [view(W, H, "z")] * snaps
    cams.append(dict(type="ortho", W=W, H=H, fwd=(1.0, 2.0, 2.5), up=(0, 0, 1), lo=(-0.4, -0.6), hi=(0.8, 0.7), wrap=False))
    of = list(range(snaps)) + [snaps - 1]
    R.build_tets(torch.from_numpy(np.stack(p)).cuda(), N)
    R.project_bin(cams, of)
    g = np.random.default_rng(N).normal(size=(len(cams), H, W)).astype(np.float32)
    got = R.render_backward(torch.from_numpy(g).cuda()).cpu().numpy().astype(np.float64)
    R.sync()
    for s in range(snaps):
        ref = sum(oracle.gradient(p[s], N, cams[f], g[f].astype(np.float64)) for f in range(len(cams)) if of[f] == s)
        assert np.linalg.norm(got[s] - ref) <= 1e-3 * max(np.linalg.norm(ref), 1e-30)
