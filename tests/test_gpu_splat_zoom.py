"""Centroid splats seen through windows so small that a splat reaches further
than FP32 counts pixels (2^24), to beyond 10^9 pixels, and beside splats that do
not, against the kernel in FP64 (numpy)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TETS = np.array([[1, 0, 2, 4], [3, 1, 2, 4], [3, 5, 1, 4], [3, 6, 5, 4], [3, 2, 6, 4], [3, 7, 5, 6]])
BITS = 62


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    return Renderer(frac_bits=BITS)


def tetrahedra(d, N):
    """Vertices [6 N^3][4][3] from displacements in cells (unit box)."""
    c = np.arange(N ** 3)
    i, j, k = c % N, (c // N) % N, c // (N * N)
    corner = []
    for n in range(8):
        a, b, e = n & 1, (n >> 1) & 1, n >> 2
        idx = (i + a) % N + N * ((j + b) % N + N * ((k + e) % N))
        corner.append((np.stack([i + a, j + b, k + e], axis=1) + d[idx]) / N)
    return np.stack(corner, axis=1)[:, TETS].reshape(-1, 4, 3)


def splats(v, lo, hi, W, H):
    e = v[:, 1:] - v[:, :1]
    h = np.cbrt(np.abs(np.einsum("ta,ta->t", e[:, 0], np.cross(e[:, 1], e[:, 2])) / 6.0))
    x = lo[0] + (np.arange(W) + 0.5) * ((hi[0] - lo[0]) / W)
    y = lo[1] + (np.arange(H) + 0.5) * ((hi[1] - lo[1]) / H)
    out = np.zeros((H, W))
    for c, s in zip(v.mean(1), h):
        q = np.sqrt((x[None, :] - c[0]) ** 2 + (y[:, None] - c[1]) ** 2) / s
        out += np.where(q < 1, 1 - 1.5 * q * q + 0.75 * q ** 3, 0.25 * np.maximum(2 - q, 0) ** 3) * 10 / (7 * np.pi * s * s)
    return out / len(v), len(v)


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("N,W,H,size", [(2, 77, 23, 1e-4), (2, 77, 23, 1.6e-6), (3, 34, 92, 4e-7), (1, 64, 64, 1e-7), (4, 9, 9, 1e-7),
                                        (2, 64, 30, 3e-8), (1, 40, 40, 1e-8), (1, 90, 5, 2e-8)])
def test_splats_of_a_far_zoom(R, N, W, H, size, half):
    """A splat's value is good to 3e-6 of it in FP32 (its place, over its size,
    to a few 2^-24), and is rounded to a unit: the fraction bits count from the
    mean of the window, which is 1 / size^2 of the box's."""
    rng = np.random.default_rng(N + W)
    d = rng.integers(-512, 513, (N ** 3, 3)) / 2048.0  # (exact in both formats)
    lo = np.array([0.43, 0.38])
    hi = lo + size * np.array([1.0, H / W])
    p = np.zeros((N ** 3, 4), dtype=np.float16 if half else np.float32)
    c = np.arange(N ** 3)
    q = np.stack([c % N, (c // N) % N, c // (N * N)], axis=1)
    if half:
        p[:, :3] = d
        d = (p[:, :3].astype(np.float32) * (np.float32(1) / np.float32(N))).astype(np.float64) * N
    else:
        p[:, :3] = np.mod((q + d) / N, 1.0)
        d = p[:, :3].astype(np.float64) * N - q
        d -= N * np.round(d / N)
    R.build_tets(torch.from_numpy(p).cuda(), N)
    got = R.render_centroids(dict(type="ortho", W=W, H=H, fwd=(0, 0, 1), up=(0, 1, 0), lo=tuple(lo), hi=tuple(hi), wrap=False))
    R.sync()
    ref, n = splats(tetrahedra(d, N), lo, hi, W, H)
    unit = 2.0 ** -BITS / ((hi[0] - lo[0]) * (hi[1] - lo[1]))
    assert np.all(np.abs(got.cpu().numpy() - ref) <= 3e-6 * ref + n * unit)
