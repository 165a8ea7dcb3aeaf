"""Densities of tetrahedra whose volume leaves FP32's range (particles far
outside the box): m over an infinite volume is 0."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TETS = np.array([[1, 0, 2, 4], [3, 1, 2, 4], [3, 5, 1, 4], [3, 6, 5, 4], [3, 2, 6, 4], [3, 7, 5, 6]])


@pytest.mark.parametrize("far", [1e12, 1e16, 3e19, 1e25])
def test_density_of_a_volume_out_of_range(far):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    N = 4
    i = np.arange(N ** 3)
    q = np.stack([i % N, (i // N) % N, i // (N * N)], axis=1)
    p = np.zeros((N ** 3, 4), dtype=np.float32)
    p[:, :3] = q / N
    p[21, 0] = far  # two neighbours, far off in x and in y
    p[22, 1] = far
    rho = torch.full((1, 6 * N ** 3), -1.0, device="cuda")
    R = Renderer()
    R.build_tets(torch.from_numpy(p).cuda(), N, rho_out=rho)
    R.sync()
    # the six products of a determinant in FP32: infinite where their sum is not
    # a number (an infinity of each sign), which is left out
    d = p[:, :3] - (q / N).astype(np.float32)
    c = np.stack([np.stack([(q[:, k] + o[k]) % N for k in range(3)], axis=1) @ np.array([1, N, N * N])
                  for o in [(n & 1, (n >> 1) & 1, n >> 2) for n in range(8)]], axis=1)
    off = np.array([(n & 1, (n >> 1) & 1, n >> 2) for n in range(8)], dtype=np.float32) / N
    v = (off[None] + d[c])[:, TETS].reshape(-1, 4, 3)
    a, b, e = (v[:, k] - v[:, 0] for k in (1, 2, 3))
    with np.errstate(over="ignore", invalid="ignore"):
        V = (a[:, 0] * (b[:, 1] * e[:, 2] - b[:, 2] * e[:, 1]) + a[:, 1] * (b[:, 2] * e[:, 0] - b[:, 0] * e[:, 2])
             + a[:, 2] * (b[:, 0] * e[:, 1] - b[:, 1] * e[:, 0]))
    assert V.dtype == np.float32
    got = rho.cpu().numpy()[0]
    assert np.isinf(V).any() == (far > 1e18)
    assert np.all(got[np.isinf(V)] == 0.0)
    assert np.all(np.isfinite(got[np.isfinite(V)]))
