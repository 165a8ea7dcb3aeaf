"""Cubes with a corner that is not finite are drawn by no projection, so they
are in no gradient and no grid either. In a lattice of 2^3 particles every
particle is a corner of all eight cubes: one bad particle leaves nothing."""
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


def bad_lattice(R, N, bad, value, half):
    rng = np.random.default_rng(N)
    i = np.arange(N ** 3)
    q = np.stack([i % N, (i // N) % N, i // (N * N)], axis=1)
    d = rng.uniform(-0.3, 0.3, (N ** 3, 3))
    p = np.zeros((N ** 3, 4), dtype=np.float16 if half else np.float32)
    p[:, :3] = d if half else np.mod((q + d) / N, 1.0)
    good = torch.from_numpy(p.copy()).cuda()
    p[bad, 1] = value
    pos = torch.from_numpy(p).cuda()
    return good, pos


def latched(R):
    from paper_1208_3206_gb300._lib import LtError
    with pytest.raises(LtError) as e:
        R.sync()
    return e.value.name == "LT_ERR_NONFINITE"


VIEW = dict(type="ortho", W=24, H=20, fwd=(0, 0, 1), up=(0, 1, 0), lo=(0, 0), hi=(1, 1), wrap=True)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("half", [False, True])
def test_gradient_of_bad_cubes(R, half, value):
    good, pos = bad_lattice(R, 2, 3, value, half)
    R.build_tets(pos, 2)
    assert latched(R)
    R.project_bin([VIEW])
    assert float(R.render_tiles().abs().max()) == 0.0
    assert float(R.render_backward(torch.ones((1, 20, 24), device="cuda")).abs().max()) == 0.0
    assert latched(R)  # (by the bin pass)
    # 5^3: the particles that share no cube with the bad one are not touched
    good, pos = bad_lattice(R, 5, 31, value, half)
    g = torch.rand((1, 20, 24), generator=torch.Generator("cuda").manual_seed(1), device="cuda")
    grads = []
    for p in (good, pos):
        R.build_tets(p, 5)
        R.project_bin([VIEW])
        grads.append(R.render_backward(g).reshape(125, -1).clone())
    assert latched(R)
    i = np.arange(125)
    q = np.stack([i % 5, (i // 5) % 5, i // 25], axis=1)
    far = (np.abs((q - q[31] + 2) % 5 - 2) >= 2).any(1)
    assert far.sum() == 98
    assert torch.equal(grads[0][far], grads[1][far])
    assert bool(torch.isfinite(grads[1]).all())
    assert float(grads[1][31].abs().max()) == 0.0


@pytest.mark.parametrize("weight", ["density", "streams"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("half", [False, True])
def test_grid_of_bad_cubes(R, half, value, weight):
    _, pos = bad_lattice(R, 2, 3, value, half)
    R.build_tets(pos, 2)
    assert latched(R)
    assert float(R.resample(12, weight=weight).abs().max()) == 0.0
    assert latched(R)
