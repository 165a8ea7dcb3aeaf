"""What the tile size may and may not change in a frame.

A tetrahedron's edge functions are formed relative to its box in the tile, so
the tile size decides how they round, and with it which fragments of very flat
tetrahedra are evaluated exactly. Frames of a given tile size therefore keep
their values, and a size that nobody chose is the documented 16 for every frame.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Renderer():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    return Renderer


def sheets(N, seed):
    """A unit box's lattice whose planes lie together in pairs (within 2^-18),
    strewn over half a cell in them: half of the tetrahedra are nearly flat.
    Coordinates are multiples of 2^-24, the same on every machine."""
    rng = np.random.default_rng(seed)
    i = np.arange(N ** 3)
    q = np.stack([i % N, (i // N) % N, i // (N * N)], axis=1).astype(np.int64)
    q[:, 2] &= ~1
    one = 1 << 24
    x = (q * one) // N + rng.integers(-one // (2 * N), one // (2 * N), q.shape)
    x[:, 2] = (q[:, 2] * one) // N + rng.integers(0, 64, N ** 3)
    pos = np.zeros((N ** 3, 4), dtype=np.float32)
    pos[:, :3] = (x % one).astype(np.float32) / np.float32(one)
    return torch.from_numpy(pos).cuda()


OBLIQUE = dict(type="ortho", W=300, H=280, fwd=(1.0, 2.0, 0.4), up=(0, 0, 1), lo=(-0.6, -0.4), hi=(0.9, 1.0), wrap=False)

# pixels of sheets(24, 2) that moved by 3e-6 to 8e-6 of their value with
# coordinates taken from the anchor in one step (the same as before that)
PIXELS = {
    64: {(50, 69): "0x1.5f6b420p-2", (47, 137): "0x1.65fa2a0p-2", (57, 171): "0x1.8e84520p-2",
         (56, 117): "0x1.c11fa60p-2", (45, 31): "0x1.b895ca0p-2", (50, 68): "0x1.9e56ac0p-2"},
    32: {(52, 174): "0x1.505fca0p-2", (52, 172): "0x1.6235460p-2", (52, 171): "0x1.71c0ac0p-2",
         (50, 69): "0x1.5f6c400p-2", (221, 161): "0x1.205c540p-1", (215, 193): "0x1.df81d20p-2"},
}


@pytest.mark.parametrize("tile", sorted(PIXELS))
def test_values_of_a_tile_size(Renderer, tile):
    """Two roundings of a pixel (its exact fragments' conversion and its own) may differ."""
    R = Renderer(tile=tile)
    R.build_tets(sheets(24, 2), 24)
    R.project_bin(OBLIQUE)
    img = R.render_tiles().cpu().numpy().reshape(280, 300).astype(np.float64)
    for (y, x), v in PIXELS[tile].items():
        assert abs(img[y, x] - float.fromhex(v)) <= 2.0 ** -23 * float.fromhex(v), (y, x)


def test_values_in_perspective(Renderer):
    """The same in perspective at 64-pixel tiles, where the pixels moved by 7e-6
    to 1.1e-5; approximate reciprocals in the projection leave 2e-6."""
    R = Renderer(tile=64)
    R.build_tets(sheets(24, 2), 24)
    R.project_bin(dict(type="persp", W=300, H=280, eye=(0.5, -1.4, 0.9), fwd=(0.0, 1.0, -0.21), up=(0, 0, 1), fov_y_deg=50.0))
    img = R.render_tiles().cpu().numpy().reshape(280, 300).astype(np.float64)
    for (y, x), v in {(191, 128): 1.7096133, (191, 66): 1.8924608, (105, 190): 1.1309264}.items():
        assert abs(img[y, x] - v) <= 2e-6 * v, (y, x)


@pytest.mark.parametrize("W,H", [(300, 280), (1040, 1024)])
def test_tile_left_open(Renderer, W, H):
    """The default tile is 16 pixels whatever the frame's size, and writing back
    the configuration that was read changes nothing."""
    view = dict(OBLIQUE, W=W, H=H)
    pos = sheets(16, 3)

    def frame(R):
        R.build_tets(pos, 16)
        R.project_bin(view)
        return R.render_tiles().clone(), R.get_stats()["tile"]

    want, _ = frame(Renderer(tile=16))
    R = Renderer()
    for _ in range(2):
        img, tile = frame(R)
        assert tile == 16
        assert torch.equal(img, want)
        R.set_config(**R.get_config())
