"""Resampling where the grid's columns run along faces of the tessellation: the
lattice at rest, or at rest along one axis, with columns on lattice planes and
on the diagonals between them. A column on a face belongs to one side of it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    return Renderer()


def particles(N, d, half):
    i = np.arange(N ** 3)
    q = np.stack([i % N, (i // N) % N, i // (N * N)], axis=1)
    p = np.zeros((N ** 3, 4), dtype=np.float16 if half else np.float32)
    x = np.mod((q + d) / N, 1.0).astype(np.float32)
    p[:, :3] = d if half else np.where(x >= 1, np.float32(0), x)
    return torch.from_numpy(p).cuda()


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("weight", ["density", "streams"])
@pytest.mark.parametrize("N,n", [(2, 5), (2, 21), (4, 2), (6, 15), (6, 31), (8, 20), (10, 9), (12, 15), (12, 30), (16, 8), (16, 16),
                                 (7, 7), (5, 25)])
def test_lattice_at_rest(R, N, n, weight, half):
    """Every cell holds the mean (its edge 1 / n times density 1, or one stream)
    to FP32's rounding and the FP32 positions' (2^-24 of the box, over a
    cell of the lattice: 2^-24 N)."""
    R.build_tets(particles(N, np.zeros((N ** 3, 3)), half), N)
    g = R.resample(n, weight=weight).cpu().numpy().astype(np.float64) * n
    R.sync()
    assert np.abs(g - 1.0).max() <= 2.0 ** -23 * (1 + N)


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("N,n,at_rest", [(8, 20, 0), (8, 20, 1), (6, 15, 0), (10, 9, 1), (4, 2, 0)])
def test_mass_with_an_axis_at_rest(R, N, n, at_rest, half):
    """Columns on lattice planes of the axis at rest, the others random: the mass
    of a plane's columns is that of the columns 1e-5 of a cell beside it, on one
    side or the other (to 1e-3: the lattice does not fold)."""
    d = np.random.default_rng(N).integers(-200, 201, (N ** 3, 3)) / 1024.0  # (below a quarter of a cell)
    d[:, at_rest] = 0.0
    on_plane = (2 * np.arange(n) + 1) * N % (2 * n) == 0
    assert on_plane.any()

    def planes(shift):
        moved = d.copy()
        moved[:, at_rest] = shift
        R.build_tets(particles(N, moved, half and shift == 0.0), N)  # (such offsets are not in FP16)
        g = R.resample(n, weight="density").cpu().numpy().astype(np.float64).sum(0)
        R.sync()
        return (g.sum(0) if at_rest == 0 else g.sum(1))[on_plane]

    here, right, left = planes(0.0), planes(1e-5), planes(-1e-5)
    assert np.all(np.minimum(np.abs(here - right), np.abs(here - left)) <= 1e-3 * here)


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("N,n", [(6, 15), (7, 21), (9, 27), (10, 9), (12, 30), (13, 39)])
def test_particles_that_coincide(R, N, n, axis):
    """A seventh of a lattice's particles moved onto their neighbours: tetrahedra
    flat in the vertical planes that columns run along, with volumes of rounding's
    size. A cell's line crosses the tetrahedra of a few cubes, no more."""
    p = particles(N, np.zeros((N ** 3, 3)), False)
    i = np.arange(N ** 3)
    a, b, c = i % N, (i // N) % N, i // (N * N)
    onto = i[((a + 2 * b + 3 * c) % 7 == 3) & (np.maximum(a, b) < N - 2) & (c < N - 1)]
    for q in onto:
        p[int(q) + (1, N)[axis]] = p[int(q)]
    R.build_tets(p, N)
    streams = R.resample(n, weight="streams").cpu().numpy().astype(np.float64) * n
    R.sync()
    assert 0.0 <= streams.min() and streams.max() <= 24.0
    assert 0.9 <= streams.mean() <= 1.1
    assert bool(torch.isfinite(R.resample(n, weight="density")).all())
    R.sync()
