"""An upstream gradient that is not finite at one pixel reaches only the
Gaussians that pixel composites: the adjoints take skipped pixels along with a
zero weight, which must not meet the infinity."""
import numpy as np
import pytest

from paper_2412_20720_gb300 import synthetic as sy
from paper_2412_20720_gb300.render import PARAM_KEYS, RenderConfig, Renderer
from helpers import to_device

pytestmark = pytest.mark.gpu


def _case(tile, ppt):
    params = sy.make_scene(1500, 23, (-1, -1, -1), (1, 1, 1), sh_degree=1, t_order=1).as_dict()
    cfg = RenderConfig(sh_degree=1, t_order=1, inst_capacity=1 << 18, tile=tile, pixels_per_thread=ppt)
    return to_device(params), Renderer(1500, [sy.tiny_view(96, 72)], cfg)


def _check(run, value, scale_tol):
    """run(v, s) -> gradient rows with the pixel's upstream gradient v and the others' scaled by s."""
    others, one, bad = run(0.0, 1.0), run(1.0, 0.0), run(value, 1.0)
    touched = (one != 0).any(1)
    wrong = ~np.isfinite(bad).all(1)
    assert touched.any() and wrong.any() and not (wrong & ~touched).any()
    assert np.abs(bad[~touched] - others[~touched]).max() <= scale_tol * np.abs(others).max()


# 1e-4 of the largest gradient: atomics add in another order from run to run
@pytest.mark.parametrize("tile,ppt", [(16, 2), (16, 4), (16, 8), (8, 1), (8, 2)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_colour_gradients(tile, ppt, value):
    import torch
    p, r = _case(tile, ppt)
    gen = torch.Generator(device="cuda").manual_seed(1)
    base = torch.randn(3 * r.total_pixels, device="cuda", generator=gen)

    def run(v, s):
        r.forward(p)
        d = base * s
        d[[37 * 96 + 51, 72 * 96 + 37 * 96 + 51]] = v  # red and green of pixel (51, 37)
        grads = {k: torch.zeros_like(p[k]) for k in PARAM_KEYS}
        r.backward(p, d, grads)
        return torch.cat([grads[k].reshape(1500, -1) for k in PARAM_KEYS], 1).cpu().numpy()

    _check(run, value, 1e-4)
