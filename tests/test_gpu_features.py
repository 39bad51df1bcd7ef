"""Parity of the scale-gated feature rendering (Sec. 7) and its backward
(geometry fixed) with the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2412_20720_gb300 import synthetic as sy
from paper_2412_20720_gb300.render import RenderConfig, Renderer

from helpers import (check_pixels, compare_group, loss_gradient_at_settled_pixels, oracle_flags, oracle_proj,
                     oracle_settings, to_device)

pytestmark = pytest.mark.gpu


def feat_case(D, ts=(0.5,), seed=17, n=1500, tile=16):
    sc = sy.make_scene(n, seed, (-1, -1, -1), (1, 1, 1), sh_degree=1, t_order=1)
    views = [sy.tiny_view(96, 72, t=t) for t in ts]
    cfg = RenderConfig(sh_degree=1, t_order=1, inst_capacity=1 << 18, tile=tile)
    params = sc.as_dict()
    rng = np.random.default_rng(seed)
    feats = rng.standard_normal((params["mean"].shape[0], D)).astype(np.float32)
    gate = rng.uniform(0.0, 1.0, D).astype(np.float32)
    return params, views, cfg, feats, gate


@pytest.mark.parametrize("D,ts", [(32, (0.5,)), (8, (0.4, 0.6)), (16, (0.5,))])
def test_feature_map_matches_oracle(D, ts):
    import torch
    params, views, cfg, feats, gate = feat_case(D, ts)
    r = Renderer(params["mean"].shape[0], views, cfg)
    p = to_device(params)
    out = r.forward_features(p, torch.from_numpy(feats).cuda(), torch.from_numpy(gate).cuda())
    r.check()
    got = [x.cpu().numpy() for x in r.split(out, D)]
    img = [x.cpu().numpy() for x in r.split(r.forward(p))]
    T = r.workspace_view(r.layout.pix_T, torch.float32, r.total_pixels).cpu().numpy()
    r.check()
    fhat = oracle.gated_features(feats, gate)
    off = 0
    for k, v in enumerate(views):
        H, W = int(v["height"]), int(v["width"])
        pr = oracle_proj(params, v, cfg)
        # the admissible results carry the features composited with the
        # colour weights as extra channels; the matched one is checked
        flags, chosen = check_pixels(pr, v, cfg, np.arange(W * H), img[k].reshape(3, -1).T, T[off:off + H * W],
                                     extra=fhat)
        off += H * W
        assert np.abs(chosen[:, 5:]).max() > 0.3
        assert np.abs(got[k].reshape(D, -1).T - chosen[:, 5:]).max() <= 2e-4


# The adjoint takes 4-pixel strips for D <= 16 on 16-pixel tiles, 2-pixel
# strips otherwise.
@pytest.mark.parametrize("D,tile", [(32, 16), (16, 16), (8, 16), (8, 8)])
def test_feature_backward_matches_oracle(D, tile):
    import torch
    params, views, cfg, feats, gate = feat_case(D, seed=18, tile=tile)
    view = views[0]
    st = oracle_settings(cfg)
    flags = oracle_flags(oracle_proj(params, view, cfg), view, cfg)
    pr = oracle.preprocess(params, view, st)
    F, mg = oracle.render_features(pr, view, st, feats, gate)
    dF = loss_gradient_at_settled_pixels(np.random.default_rng(19), flags, F.shape)
    gf, gg = oracle.render_features_backward(pr, view, st, feats, gate, dF)
    r = Renderer(params["mean"].shape[0], views, cfg)
    f_d, g_d = torch.from_numpy(feats).cuda(), torch.from_numpy(gate).cuda()
    r.forward_features(to_device(params), f_d, g_d)
    grad_f = torch.zeros_like(f_d)
    grad_g = torch.zeros_like(g_d)
    r.backward_features(f_d, g_d, torch.from_numpy(dF.reshape(-1).astype(np.float32)).cuda(), grad_f, grad_g)
    r.check()
    compare_group("dL/df", grad_f.cpu().numpy().astype(np.float64), gf, 1e-3, 1e-4)
    compare_group("dL/dgate", grad_g.cpu().numpy().astype(np.float64), gg, 1e-3, 1e-4)


@pytest.mark.parametrize("D,tile", [(8, 16), (16, 16), (32, 16), (16, 8), (32, 8)])
def test_short_list_kernels_match_the_matrix_kernels(D, tile):
    """The same calls by both routes (an instance capacity of fewer and of more
    than 40 instances a tile, 4225 tiles).  Map: weights add up to at most 1,
    so the split products stay within 2^-21 and up to 150 roundings of 2^-24;
    gradients: 1e-4 of the largest, as atomics add in another order."""
    import torch
    params = to_device(sy.make_scene(3000, 21, (-1, -1, -1), (1, 1, 1), sh_degree=1, t_order=1).as_dict())
    W, H = 65 * tile, 65 * tile - 9
    gen = torch.Generator(device="cuda").manual_seed(5)
    feats, gate = torch.randn((3000, D), device="cuda", generator=gen), torch.rand((D,), device="cuda", generator=gen)
    up = torch.randn(D * W * H, device="cuda", generator=gen)
    got = []
    for cap in (39 * 4225, 1 << 21):
        r = Renderer(3000, [sy.tiny_view(W, H)], RenderConfig(sh_degree=1, t_order=1, inst_capacity=cap, tile=tile))
        out = r.forward_features(params, feats, gate)
        assert r.check()[1] > 20_000
        gf, gg = torch.zeros_like(feats), torch.zeros_like(gate)
        r.backward_features(feats, gate, up, gf, gg)
        got.append((out, gf, gg))
    (ma, fa, ga), (mb, fb, gb) = got
    assert float(ma.abs().max()) > 0.3
    assert float((ma - mb).abs().max()) <= 2.0 ** -21 + 150 * 2.0 ** -24
    assert float((fa - fb).abs().max()) <= 1e-4 * float(fa.abs().max())
    assert float((ga - gb).abs().max()) <= 1e-4 * float(ga.abs().max())


def _eleven_bits(x):
    """x rounded to 11 significant bits."""
    m, e = np.frexp(x)
    return np.ldexp(np.round(m * 2048) / 2048, e)


def test_split_products_keep_their_bits():
    """The matrix kernels' sums against FP64 sums of the same weights, which
    one-hot features give exactly.  A product is within 2^-21 of itself and the
    accumulation within some roundings of 2^-24, so 2^-19 of the sum of the
    magnitudes bounds the error; operands of 11 bits miss it."""
    import torch
    n, W, H, tol = 32, 48, 40, 2.0 ** -19
    params = to_device(sy.make_scene(n, 4, (-0.7, -0.7, -0.7), (0.7, 0.7, 0.7), sh_degree=1, t_order=1).as_dict())
    params["opacity_logit"] += 1.5
    r = Renderer(n, [sy.tiny_view(W, H)], RenderConfig(sh_degree=1, t_order=1, inst_capacity=1 << 16))
    rng = np.random.default_rng(6)
    w = r.forward_features(params, torch.eye(n, device="cuda")).view(n, -1).cpu().numpy().astype(np.float64)
    assert (w.max(1) > 0.05).sum() >= 8
    for D in (32, 16, 8):
        f = rng.standard_normal((n, D)).astype(np.float32)
        g = rng.standard_normal((D, H * W)).astype(np.float32)
        norm = np.sqrt((f.astype(np.float64) ** 2).sum(1, keepdims=True))
        fhat = f / norm
        feats = torch.from_numpy(f).cuda()
        out = r.forward_features(params, feats).view(D, -1).cpu().numpy()
        want, size = fhat.T @ w, np.abs(fhat).T @ w
        assert np.all(np.abs(out - want) <= tol * size)
        if D == 32:
            assert np.any(np.abs(fhat.T @ _eleven_bits(w) - want) > 4 * tol * size)
        gf = torch.zeros_like(feats)
        r.backward_features(feats, None, torch.from_numpy(g.reshape(-1)).cuda(), gf)
        jac = lambda v: (v - fhat * (fhat * v).sum(1, keepdims=True)) / norm
        want, mag = jac(w @ g.T.astype(np.float64)), w @ np.abs(g.T)
        size = (mag + np.abs(fhat) * (np.abs(fhat) * mag).sum(1, keepdims=True)) / norm
        assert np.all(np.abs(gf.cpu().numpy() - want) <= tol * size)
        assert np.any(np.abs(jac(_eleven_bits(w) @ g.T) - want) > 4 * tol * size)
        assert np.any(np.abs(jac(w @ _eleven_bits(g).T) - want) > 4 * tol * size)
    r.check()
