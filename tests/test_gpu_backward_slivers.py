"""The adjoint's row spans where an edge function's slope nears FP32's range:
cells squeezed to slivers, seen along an axis at which their vertices coincide,
at many fraction bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def squeezed(delta):
    """4^3 particles at rest but for two planes `delta` on either side of x = 5/16."""
    i = np.arange(64)
    q = np.stack([i % 4, (i // 4) % 4, i // 16], axis=1)
    x = q / 4.0
    x[:, 0] = np.where(q[:, 0] == 0, 0.3125 - delta, np.where(q[:, 0] == 1, 0.3125 + delta, x[:, 0]))
    p = np.zeros((64, 4), dtype=np.float32)
    p[:, :3] = x
    return torch.from_numpy(p).cuda()


@pytest.mark.parametrize("delta,bits", [(1.25 * 2.0 ** -18, 62), (1.25 * 2.0 ** -19, 60), (1.25 * 2.0 ** -20, 58),
                                        (1.25 * 2.0 ** -21, 56)])
def test_steep_edges(delta, bits):
    """Slopes between 2^126 and 2^128: the fraction bits scale every edge
    function by a power of two, exactly, so the gradient does not depend on them."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3206_gb300.render import Renderer
    view = dict(type="ortho", W=8, H=8, fwd=(0, 0, 1), up=(0, 1, 0), lo=(0, 0), hi=(1, 1), wrap=True)
    g = torch.rand((1, 8, 8), generator=torch.Generator("cuda").manual_seed(2), device="cuda")

    def gradient(frac_bits):
        R = Renderer(frac_bits=frac_bits)
        R.build_tets(squeezed(delta), 4)
        R.project_bin([view])
        return R.render_backward(g).clone()

    assert torch.equal(gradient(bits), gradient(40))
