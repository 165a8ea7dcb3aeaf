"""Area-averaged pixels where hull edges and rays run along the pixels' sides.

Lattices seen along an axis whose pixel edges lie on lattice planes: the lines
of a tetrahedron are parallel to a pixel's sides and pass them at the rounding
of the positions (1e-16 to 1e-7 of a pixel), on either side. The share of a
tetrahedron in a pixel must not depend on which side that is. Against the FP64
oracle: lines are good to 2^-24 of a pixel and a hull's function to 2^-24 of
its largest value, over sectors at least a pixel long here, so a pixel is good
to 1e-5 of max(pixel, mean); the periodic frame holds the mass to 1e-6.
"""
import numpy as np
import pytest

import oracle
from lt_inputs import ortho_z

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    return Renderer()


def lattice(N):
    i = np.arange(N ** 3)
    return np.stack([i % N, (i // N) % N, i // (N * N)], axis=1)


def displaced(N, kind):
    """Displacements in cells: none; a plane wave along an axis; two axes
    random (multiples of 2^-10 of a cell) and the third not displaced."""
    d = np.zeros((N ** 3, 3))
    if kind.startswith("wave"):
        a = "xyz".index(kind[-1])
        d[:, a] = 0.9 * np.sin(2.0 * np.pi * lattice(N)[:, a] / N) * N / (2.0 * np.pi)
    elif kind.startswith("still"):
        d = np.random.default_rng(N).integers(-614, 615, (N ** 3, 3)) / 1024.0
        d[:, "xyz".index(kind[-1])] = 0.0
    return d


def particles(N, kind, half):
    """What the renderer takes, and the positions it stands for."""
    d = displaced(N, kind)
    p = np.zeros((N ** 3, 4), dtype=np.float16 if half else np.float32)
    if half:
        p[:, :3] = d
        off = p[:, :3].astype(np.float32) * (np.float32(1) / np.float32(N))
        return p, np.mod(lattice(N) / N + off.astype(np.float64), 1.0)
    x = np.mod((lattice(N) + d) / N, 1.0).astype(np.float32)
    p[:, :3] = np.where(x >= 1, np.float32(0), x)
    return p, p


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("N,W,H,kind", [(10, 10, 10, "none"), (40, 40, 40, "none"), (20, 60, 80, "none"), (50, 200, 200, "none"),
                                        (18, 36, 36, "none"), (18, 36, 36, "wave x"), (18, 36, 36, "wave y"),
                                        (18, 36, 36, "wave z"), (20, 60, 80, "still y"), (12, 36, 24, "still z")])
def test_pixel_edges_on_lattice_planes(R, N, W, H, kind, half):
    p, x = particles(N, kind, half)
    R.build_tets(torch.from_numpy(p).cuda(), N)
    got = R.render_area(ortho_z(W, H)).cpu().numpy().astype(np.float64)
    R.sync()
    ref = np.ones((H, W)) if kind == "none" else oracle.render_area(x, N, ortho_z(W, H))
    assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(ref, 1.0))
    assert abs(got.mean() - 1.0) <= 1e-6


@pytest.mark.parametrize("shift", [0.0, 1e-15, 1e-12, 1e-9, 1e-8, 3e-8, 1e-7, 1e-6])
@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("N", [6, 10, 16])
def test_lattice_planes_beside_pixel_edges(R, N, sign, shift):
    """The undeformed lattice behind a window that begins `shift` pixels off a
    lattice plane (the pixels are then 1e-6 / W smaller or larger at most)."""
    W = 4 * N
    p, x = particles(N, "none", False)
    lo = np.float32(sign * shift / W)
    cam = dict(type="ortho", W=W, H=W, fwd=(0, 0, 1), up=(0, 1, 0), lo=(lo, lo), hi=(1.0, 1.0), wrap=False)
    R.build_tets(torch.from_numpy(p).cuda(), N)
    got = R.render_area(cam).cpu().numpy().astype(np.float64)
    R.sync()
    # (a window that begins before the box loses `shift` of its first row and column)
    assert np.all(np.abs(got - 1.0) <= 1e-5)
    assert abs(got.mean() - 1.0) <= 1e-6


@pytest.mark.parametrize("N,W,H,kind", [(5, 20, 15, "still x"), (7, 21, 35, "still x"), (9, 36, 45, "still y"),
                                        (11, 22, 33, "still x"), (13, 52, 39, "still y"), (20, 60, 60, "still x")])
def test_projections_that_nearly_coincide(R, N, W, H, kind):
    """FP16 lattices with an axis at rest: vertices of a tetrahedron that project
    onto one line, or onto one point, but for the rounding of their FP64
    coordinates (box / N is not a power of two)."""
    p, x = particles(N, kind, True)
    R.build_tets(torch.from_numpy(p).cuda(), N)
    got = R.render_area(ortho_z(W, H)).cpu().numpy().astype(np.float64)
    R.sync()
    ref = oracle.render_area(x, N, ortho_z(W, H))
    assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(ref, 1.0))
    assert abs(got.mean() - 1.0) <= 1e-6
