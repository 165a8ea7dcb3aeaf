"""The rounding of area-averaged pixels against the FP64 oracle, where hulls are
long and flat: sectors a few hundredths of a pixel wide and tens long, whose
function rises a hundred times faster than the mean pixel's."""
import numpy as np
import pytest

import oracle
from lt_inputs import ZeldovichField

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    return Renderer()


@pytest.mark.parametrize("N,W,H,lam,seed", [(16, 700, 150, 3.5, 7), (16, 700, 150, 3.5, 8), (24, 640, 640, 2.5, 7)])
def test_long_flat_sectors(R, N, W, H, lam, seed):
    """Rounding a pixel to FP32 moves it by 2^-24 / sqrt(3) at most in the
    root mean square; its tetrahedra's parts, each rounded like a vertex's place
    (2^-24 of a pixel) and of both signs, add less than that again: 5e-8 of the
    image's norm together."""
    pos = ZeldovichField.generate(N, -2.5, 0.375 * N, seed).positions(lam)
    cam = dict(type="ortho", W=W, H=H, fwd=(1.0, 2.0, 2.5), up=(0, 0, 1), lo=(-0.95, -0.55), hi=(0.35, 0.75), wrap=False)
    R.build_tets(torch.from_numpy(pos).cuda(), N)
    got = R.render_area(cam).cpu().numpy().astype(np.float64)
    R.sync()
    ref = oracle.render_area(pos, N, cam)
    assert np.linalg.norm(got - ref) <= 5e-8 * np.linalg.norm(ref)
