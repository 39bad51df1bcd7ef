"""Preprocess through the staging area (many logical blocks, large instance
buffers) against the look-back form (small instance buffers): the same slots,
records and counts bit for bit."""
import numpy as np
import pytest

from paper_2412_20720_gb300 import fgs4d
from paper_2412_20720_gb300 import synthetic as sy
from paper_2412_20720_gb300.render import RenderConfig, Renderer
from helpers import to_device

pytestmark = pytest.mark.gpu


# 608 logical blocks of 256 (the smallest count staged), a ragged last block,
# several views, lean grids; a visible capacity below the need
@pytest.mark.parametrize("n,nviews,stage_blocks,vis_cap", [
    (155_393, 1, 0, 0), (155_648, 1, 1, 0), (60_001, 3, 0, 0), (60_001, 3, 2, 0), (200_000, 1, 0, 20_000)])
def test_same_records_as_with_the_look_back(n, nviews, stage_blocks, vis_cap):
    import torch
    params = to_device(sy.make_scene(n, 31, (-2, -2, -2), (2, 2, 2), sh_degree=1, t_order=1).as_dict())
    views = [sy.tiny_view(400, 300, t=0.2 + 0.3 * k) for k in range(nviews)]
    got = []
    for inst_cap in (1 << 22, 1000):
        r = Renderer(n, views, RenderConfig(sh_degree=1, t_order=1, inst_capacity=inst_cap, vis_capacity=vis_cap,
                                            stage_blocks_per_sm=stage_blocks))
        fgs4d.preprocess(r.gaussians(params), r.views, r.nviews, r.settings, r.ws.data_ptr(), r.ws_bytes, r.stream())
        code, counts = r.status()
        assert code == (fgs4d.ERR_CAPACITY if vis_cap else fgs4d.OK)
        v, L = counts[0], r.layout
        got.append([np.array(counts)] + [r.workspace_view(off, torch.int32, k * v).cpu().numpy()
                                         for off, k in ((L.rec_geom, 4), (L.rec_color, 4), (L.rec_blue, 1), (L.rec_tau, 1),
                                                        (L.rec_meta, 4), (L.depth_key, 1))])
    assert got[0][0][0] > 10_000
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


# one view and several; capacities that stage the records (two kernels)
@pytest.mark.parametrize("n,nviews,inst_cap", [(155_648, 1, 1 << 20), (60_001, 3, 1 << 20)])
def test_a_second_preprocess_keeps_the_lists(n, nviews, inst_cap):
    """Preprocess with other colours leaves the sorted lists in place: the
    compositor then gives the image of a whole render with them."""
    import torch
    params = to_device(sy.make_scene(n, 31, (-2, -2, -2), (2, 2, 2), sh_degree=1, t_order=1).as_dict())
    views = [sy.tiny_view(400, 300, t=0.2 + 0.3 * k) for k in range(nviews)]
    r = Renderer(n, views, RenderConfig(sh_degree=1, t_order=1, inst_capacity=inst_cap))
    assert fgs4d.preprocess_kernels(n, r.views, r.nviews, r.settings) == 2
    other = dict(params, sh=params["sh"].flip(0).contiguous())
    want = r.forward(other).clone()
    first = r.forward(params).clone()
    ws = r.ws.data_ptr()
    fgs4d.preprocess(r.gaussians(other), r.views, r.nviews, r.settings, ws, r.ws_bytes, r.stream())
    got = torch.empty_like(want)
    fgs4d.render_fwd(n, r.views, r.nviews, r.settings, ws, r.ws_bytes, got.data_ptr(), None, r.stream())
    assert not torch.equal(first, want) and torch.equal(got, want)


def test_adjoint_of_records_the_caller_filled():
    """Records copied into a workspace that no preprocess ran on give the
    gradients of the workspace they came from (several views, SH rows that
    make the adjoint take groups of Gaussians)."""
    import torch
    n, nviews = 100_003, 4  # 115 MB of SH rows and gradients, 461 MB by slots
    params = to_device(sy.make_scene(n, 7, (-2, -2, -2), (2, 2, 2), sh_degree=3, t_order=2).as_dict())
    views = [sy.tiny_view(400, 300, t=0.2 + 0.2 * k) for k in range(nviews)]
    cfg = RenderConfig(sh_degree=3, t_order=2, inst_capacity=1 << 22)
    a, b = Renderer(n, views, cfg), Renderer(n, views, cfg)
    gen = torch.Generator(device="cuda").manual_seed(1)
    d = torch.randn(3 * a.total_pixels, device="cuda", generator=gen)
    a.forward(params)
    v, L = a.check()[0], a.layout
    b.ws.fill_(0x7f)
    b.ws[L.counters:L.counters + 256] = 0
    b.workspace_view(L.counters, torch.int32, 1).fill_(v)
    for off, words in ((L.rec_geom, 4), (L.rec_color, 4), (L.rec_blue, 1), (L.rec_tau, 1), (L.rec_meta, 4), (L.depth_key, 1)):
        b.workspace_view(off, torch.int32, words * v).copy_(a.workspace_view(off, torch.int32, words * v))
    ws = b.ws.data_ptr()
    img = torch.empty(3 * b.total_pixels, device="cuda")
    fgs4d.bin_sort(n, b.views, b.nviews, b.settings, ws, b.ws_bytes, b.stream())
    fgs4d.render_fwd(n, b.views, b.nviews, b.settings, ws, b.ws_bytes, img.data_ptr(), None, b.stream())
    got = []
    for r in (a, b):
        grads = {k: torch.zeros_like(x) for k, x in params.items()}
        r.backward(params, d, grads)
        r.check()
        got.append(grads)
    for k, want in got[0].items():  # atomics add in another order from run to run
        assert float(want.abs().max()) > 0
        assert float((got[1][k] - want).abs().max()) <= 1e-4 * float(want.abs().max()), k
