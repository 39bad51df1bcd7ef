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


@pytest.mark.parametrize("D,tile", [(8, 16), (16, 8), (32, 16)])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_feature_gradients(D, tile, value):
    import torch
    p, r = _case(tile, 0)
    gen = torch.Generator(device="cuda").manual_seed(2)
    feats = torch.randn((1500, D), device="cuda", generator=gen)
    gate = torch.rand((D,), device="cuda", generator=gen)
    base = torch.randn(D * r.total_pixels, device="cuda", generator=gen)

    def run(v, s):
        r.forward_features(p, feats, gate)
        d = base * s
        d[3 * 72 * 96 + 37 * 96 + 51] = v  # component 3 of pixel (51, 37)
        g = torch.zeros_like(feats)
        r.backward_features(feats, gate, d, g)
        return g.cpu().numpy()

    _check(run, value, 1e-4)


@pytest.mark.parametrize("D", [8, 16, 32])
def test_feature_map_of_a_feature_that_is_not_finite(D):
    """NaN in one Gaussian's feature reaches only the pixels that composite it,
    and only its component."""
    import torch
    p, r = _case(16, 0)
    gen = torch.Generator(device="cuda").manual_seed(3)
    feats = torch.randn((1500, D), device="cuda", generator=gen)
    ref = r.forward_features(p, feats).view(D, -1).cpu().numpy()
    # a Gaussian that the view shows: the one with the largest gradient
    grad = torch.zeros_like(feats)
    r.backward_features(feats, None, torch.ones(D * r.total_pixels, device="cuda"), grad)
    g = int(grad.abs().sum(1).argmax())
    alone = torch.zeros_like(feats)
    alone[g] = 1.0
    hit = r.forward_features(p, alone).view(D, -1)[5].cpu().numpy() != 0  # the pixels that composite it
    bad = feats.clone()
    bad[g, 5] = float("nan")
    got = r.forward_features(p, bad).view(D, -1).cpu().numpy()
    assert hit.any()
    np.testing.assert_array_equal(np.isnan(got[5]), hit)
    assert np.isfinite(got[np.arange(D) != 5]).all()
    np.testing.assert_array_equal(got[:, ~hit], ref[:, ~hit])


@pytest.mark.parametrize("tile,ppt", [(16, 2), (16, 4), (16, 8), (8, 1), (8, 2)])
def test_products_that_overflow_stay_with_their_pixel(tile, ppt):
    """A finite gradient so large that its products with the colours overflow
    reaches only the Gaussians its pixel composites."""
    import torch
    p, r = _case(tile, ppt)
    gen = torch.Generator(device="cuda").manual_seed(1)
    base = torch.randn(3 * r.total_pixels, device="cuda", generator=gen)

    def run(v, s):
        r.forward(p)
        d = base * s
        d[[c * 72 * 96 + 37 * 96 + 51 for c in range(3)]] = v  # all channels of pixel (51, 37)
        grads = {k: torch.zeros_like(p[k]) for k in PARAM_KEYS}
        r.backward(p, d, grads)
        return torch.cat([grads[k].reshape(1500, -1) for k in PARAM_KEYS], 1).cpu().numpy()

    _check(run, 3.4e38, 1e-4)


@pytest.mark.parametrize("tile,ppt", [(16, 2), (16, 4), (16, 8), (8, 1), (8, 2)])
def test_a_colour_near_the_largest_float_stays_with_its_pixels(tile, ppt):
    """One Gaussian's colour of 8e37 makes the products with ordinary gradients
    overflow at the pixels that composite it and nowhere else."""
    import torch
    p, r = _case(tile, ppt)
    gen = torch.Generator(device="cuda").manual_seed(4)
    base = 8.0 * torch.randn(3 * r.total_pixels, device="cuda", generator=gen)

    def run(q, d):
        img = r.forward(q).clone()
        grads = {k: torch.zeros_like(p[k]) for k in PARAM_KEYS}
        r.backward(q, d, grads)
        return img, torch.cat([grads[k].reshape(1500, -1) for k in PARAM_KEYS], 1).cpu().numpy()

    img, ref = run(p, base)
    g = int(np.argsort(np.abs(ref).sum(1))[-100])  # a Gaussian that the view shows
    q = {k: v.clone() for k, v in p.items()}
    q["sh"][g] = 0.0
    q["sh"][g, 0] = 3e38  # times Y_00: colour 8.5e37 in every channel
    hit = (r.forward(q) != img).view(3, -1).any(0).repeat(3)
    touched = (run(p, base * hit)[1] != 0).any(1)
    bad = run(q, base)[1]
    assert touched[g] and not touched.all() and not np.isfinite(bad).all()
    assert np.isfinite(bad[~touched]).all()
    assert np.abs(bad[~touched] - ref[~touched]).max() <= 1e-4 * np.abs(ref).max()


def test_depth_that_overflows_stays_with_its_pixels():
    """A Gaussian whose camera depth overflows to infinity reaches the depth
    plane of the pixels that composite it and no other."""
    import torch
    params = sy.make_scene(1500, 23, (-1, -1, -1), (1, 1, 1), sh_degree=1, t_order=1).as_dict()
    p = to_device(params)
    # looking along (1, 1, 1): a mean of 3.4e38 in all coordinates has depth 5.9e38 and projects to the image centre
    view = sy.look_at((-2.0, -2.0, -2.0), (0, 0, 0), (0, -1, 0), 96, 72, 0.5)
    p["opacity_logit"] -= 3.0  # faint: the last Gaussian still shows
    p["mean"][7] = torch.tensor([3.4e38, 3.4e38, 3.4e38, 0.5], device="cuda")
    p["opacity_logit"][7] = 3.0
    for tile, ppt in ((16, 2), (16, 4), (16, 8), (8, 1), (8, 2)):
        r = Renderer(1500, [view], RenderConfig(sh_degree=1, t_order=1, inst_capacity=1 << 18, tile=tile,
                                                pixels_per_thread=ppt))
        rgb, aux = r.forward_aux(p, 0.1)
        q = dict(p, opacity_logit=p["opacity_logit"].clone())
        q["opacity_logit"][7] = -30.0
        rgb0, aux0 = r.forward_aux(q, 0.1)
        d, d0 = aux.view(4, -1)[0], aux0.view(4, -1)[0]
        hit = (aux.view(4, -1)[1] != aux0.view(4, -1)[1]) | (rgb != rgb0).view(3, -1).any(0)
        assert 0 < int(hit.sum()) < 100 and torch.isfinite(d0).all()
        assert torch.isinf(d[hit]).all()
        assert torch.equal(d[~hit], d0[~hit])


@pytest.mark.parametrize("D,tile", [(8, 16), (16, 8), (32, 16)])
def test_feature_gradients_near_the_largest_float(D, tile):
    """The adjoint is linear in the upstream gradient up to the largest floats:
    a component of 3.4025e38 (which rounds to infinity with 11 significant
    bits) gives that multiple of the gradient of 1, to 1e-3."""
    import torch
    p, r = _case(tile, 0)
    gen = torch.Generator(device="cuda").manual_seed(2)
    feats = torch.randn((1500, D), device="cuda", generator=gen)

    def run(v):
        r.forward_features(p, feats)
        d = torch.zeros(D * r.total_pixels, device="cuda")
        d[3 * 72 * 96 + 37 * 96 + 51] = v
        g = torch.zeros_like(feats)
        r.backward_features(feats, None, d, g)
        return g.cpu().numpy().astype(np.float64)

    one, big = run(1.0) * 3.4025e38, run(3.4025e38)
    below = np.abs(one).max(1) < 3e38  # the others may overflow
    assert (one[below] != 0).any()
    assert np.isfinite(big[below]).all()
    assert np.abs(big[below] - one[below]).max() <= 1e-3 * np.abs(one[below]).max()
