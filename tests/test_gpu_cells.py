"""Two-level binning (cells of 8x8 tiles): instance lists and ranges against
the oracle's sort on records written straight into the workspace, at the
visible capacities that take it (65,536, and 1,024 per cell)."""
import numpy as np
import pytest

import oracle
from paper_2412_20720_gb300 import fgs4d
from paper_2412_20720_gb300 import synthetic as sy
from paper_2412_20720_gb300.render import RenderConfig
from helpers import canonical_ranges
from test_gpu_parity import KEEP_ALL, _min_q_over_tile, _read_instances, _synthetic_records, _write_records

pytestmark = pytest.mark.gpu


def _run(rec, views, tile, inst_cap, view_of_slot=0, stage_blocks=0, vis_cap=1 << 19):
    from paper_2412_20720_gb300.render import Renderer
    n = rec["rect"].shape[0]
    cfg = RenderConfig(sh_degree=0, t_order=0, inst_capacity=inst_cap, tile=tile, vis_capacity=vis_cap,
                       stage_blocks_per_sm=stage_blocks)
    r = Renderer(n, views, cfg)
    _write_records(r, rec, view_of_slot)
    fgs4d.bin_sort(n, r.views, r.nviews, r.settings, r.ws.data_ptr(), r.ws_bytes, r.stream())
    return r, r.status()


# one cell; ragged grids whose last cells hold one tile row
# or column; 8-pixel tiles with 352 cells (two cell-sort passes); lean grids;
# rects that span up to 5 x 5 cells
@pytest.mark.parametrize("n,W,H,tile,extent,stage_blocks", [
    (3, 16, 16, 16, 2, 0), (16_384, 257, 257, 16, 6, 0), (20_001, 1157, 643, 16, 17, 1), (30_011, 1352, 1014, 8, 6, 0),
    (16_385, 1013, 619, 8, 34, 2), (16_384, 4112, 16, 16, 40, 0)])
def test_lists_equal_the_oracles(n, W, H, tile, extent, stage_blocks):
    rng = np.random.default_rng(n + tile)
    gw, gh = (W + tile - 1) // tile, (H + tile - 1) // tile
    rec = _synthetic_records(rng, n, W, H, extent, tile=tile, tau=KEEP_ALL)
    keys, vals, ranges = oracle.sort_instances(rec["rect"], rec["depth"], gw, gh)
    m = keys.shape[0]
    r, (code, counts) = _run(rec, [sy.tiny_view(W, H)], tile, m, stage_blocks=stage_blocks)  # exactly the capacity
    assert code == fgs4d.OK and counts[1] == m and counts[3] == m
    tiles, slots, gr = _read_instances(r, m, gw * gh)
    np.testing.assert_array_equal(tiles, (keys >> np.uint64(32)).astype(np.int64))
    np.testing.assert_array_equal(slots, vals)
    np.testing.assert_array_equal(canonical_ranges(gr), ranges)


def test_capacity_overflow_reports_the_need():
    n, W, H = 16_384, 640, 480
    rng = np.random.default_rng(3)
    rec = _synthetic_records(rng, n, W, H, 9, tau=KEEP_ALL)
    m = oracle.sort_instances(rec["rect"], rec["depth"], 40, 30)[0].shape[0]
    for cap in (m - 1, m // 3, n // 2):  # the last holds fewer instances than there are pairs
        _, (code, counts) = _run(rec, [sy.tiny_view(W, H)], 16, cap)
        assert code == fgs4d.ERR_CAPACITY and counts[1] == cap and counts[3] == m


def test_views_of_mixed_size():
    sizes, ns = [(200, 150), (64, 48), (1014, 1352), (17, 700)], [5000, 500, 9000, 3000]
    rng = np.random.default_rng(5)
    recs = [_synthetic_records(rng, n, w, h, 9, tau=KEEP_ALL) for n, (w, h) in zip(ns, sizes)]
    rec = {k: np.concatenate([x[k] for x in recs]) for k in recs[0]}
    tiles_e, slots_e, ranges_e, tb, sb, ib = [], [], [], 0, 0, 0
    for x, n, (w, h) in zip(recs, ns, sizes):
        gw, gh = (w + 15) // 16, (h + 15) // 16
        keys, vals, ranges = oracle.sort_instances(x["rect"], x["depth"], gw, gh)
        tiles_e.append((keys >> np.uint64(32)).astype(np.int64) + tb)
        slots_e.append(vals + sb)
        ranges_e.append(np.where(ranges[:, 1:] > ranges[:, :1], ranges + ib, ranges))
        tb, sb, ib = tb + gw * gh, sb + n, ib + keys.shape[0]
    r, (code, counts) = _run(rec, [sy.tiny_view(w, h) for w, h in sizes], 16, ib,
                             np.concatenate([np.full(n, k) for k, n in enumerate(ns)]))
    assert code == fgs4d.OK and counts[1] == ib
    tiles, slots, gr = _read_instances(r, ib, tb)
    np.testing.assert_array_equal(tiles, np.concatenate(tiles_e))
    np.testing.assert_array_equal(slots, np.concatenate(slots_e))
    np.testing.assert_array_equal(canonical_ranges(gr), np.concatenate(ranges_e))


@pytest.mark.parametrize("tile", [16, 8])
def test_left_out_tiles_are_skipped_by_every_pixel(tile):
    """With finite ellipses (round and elongated, up to 60:1) the list is an
    order-preserving part of the rect membership, and a left-out pair has q >
    tau - 4e-3 in FP64 at every pixel centre (4e-3: the margin of the records'
    tau), so alpha < 1/255 there."""
    n, W, H = 16_384, 45 * tile + 3, 37 * tile + 5
    rng = np.random.default_rng(11 + tile)
    gw, gh = (W + tile - 1) // tile, (H + tile - 1) // tile
    rec = _synthetic_records(rng, n, W, H, 12, tile=tile)
    keys, vals, _ = oracle.sort_instances(rec["rect"], rec["depth"], gw, gh)
    r, (code, counts) = _run(rec, [sy.tiny_view(W, H)], tile, keys.shape[0])
    assert code == fgs4d.OK
    tiles, slots, _ = _read_instances(r, counts[1], gw * gh)
    full = (keys >> np.uint64(32)).astype(np.int64) * n + vals
    pos = {int(p): j for j, p in enumerate(full)}
    jj = np.array([pos[int(p)] for p in tiles * n + slots])
    assert np.all(np.diff(jj) > 0)
    left = np.setdiff1d(np.arange(full.size), jj)
    assert 0.2 * full.size < left.size < full.size
    for j in rng.choice(left, 6000, replace=False):
        t, i = divmod(int(full[j]), n)
        assert _min_q_over_tile(rec, i, t % gw, t // gw, W, H, tile) > float(rec["tau"][i]) - 4e-3, (t, i)


# one key; a group of 32 less and more one; the last count ranked by counting
# and the first sorted by passes
@pytest.mark.parametrize("n", [1, 31, 32, 33, 257, 4095, 4096, 4097, 8193])
def test_depth_order_of_few_slots(n):
    import torch
    rng = np.random.default_rng(n)
    rec = _synthetic_records(rng, n, 320, 240, 3, tau=KEEP_ALL)
    for cap in (n, 100_000):  # the count, not the capacity, decides
        r, (code, _) = _run(rec, [sy.tiny_view(320, 240)], 16, 20 * n + 16, vis_cap=cap)
        assert code == fgs4d.OK
        got = r.workspace_view(r.layout.sorted_slots, torch.int32, n).cpu().numpy()
        np.testing.assert_array_equal(got, np.argsort(rec["depth"], kind="stable"))


def _lists(r, counts, ntiles):
    tiles, slots, gr = _read_instances(r, counts[1], ntiles)
    return tiles, slots, canonical_ranges(gr)


@pytest.mark.parametrize("n,cap", [(16_384, 8192), (16_385, 300)])
def test_pair_overflow_reports_a_need_that_fits(n, cap):
    """More candidate (slot, cell) pairs than 8 x inst_capacity: the reported
    need is the tiles of the rects (here each holds an instance), and a call
    with that capacity succeeds."""
    W, H, gw, gh = 640, 480, 40, 30
    rec = _synthetic_records(np.random.default_rng(n), n, W, H, 34, tau=KEEP_ALL)
    r0 = rec["rect"].astype(np.int64)
    cells = (((r0[:, 2] - 1) >> 3) - (r0[:, 0] >> 3) + 1) * (((r0[:, 3] - 1) >> 3) - (r0[:, 1] >> 3) + 1)
    cells[(r0[:, 2] <= r0[:, 0]) | (r0[:, 3] <= r0[:, 1])] = 0
    assert cells.sum() > 8 * cap
    keys, vals, ranges = oracle.sort_instances(rec["rect"], rec["depth"], gw, gh)
    m = keys.shape[0]
    _, (code, counts) = _run(rec, [sy.tiny_view(W, H)], 16, cap)
    assert code == fgs4d.ERR_CAPACITY and counts[1] == cap and counts[3] == m
    r, (code, counts) = _run(rec, [sy.tiny_view(W, H)], 16, counts[3])
    assert code == fgs4d.OK and counts[1] == m and counts[3] == m
    tiles, slots, gr = _lists(r, counts, gw * gh)
    np.testing.assert_array_equal(tiles, (keys >> np.uint64(32)).astype(np.int64))
    np.testing.assert_array_equal(slots, vals)
    np.testing.assert_array_equal(gr, ranges)


def _stretched(rec, rng, lo, hi):
    """Ellipses of widths lo..hi along one axis and 0.55..hi along the other."""
    n = rec["rect"].shape[0]
    ang = rng.uniform(0, np.pi, n)
    ang[::9] = rng.integers(0, 4, ang[::9].size) * (np.pi / 4)
    s1 = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    s2 = np.exp(rng.uniform(np.log(0.55), np.log(hi), n))
    c, s, k = np.cos(ang), np.sin(ang), 0.5 * np.log2(np.e)
    rec["conic2"] = np.stack([k * (c * c / s1 ** 2 + s * s / s2 ** 2), k * 2 * c * s * (1 / s1 ** 2 - 1 / s2 ** 2),
                              k * (s * s / s1 ** 2 + c * c / s2 ** 2)], 1)


# round and elongated ellipses of many sizes, on both tile edges; needles (their q is a difference of terms 1e4
# times as large); centres on pixel centres
@pytest.mark.parametrize("tile,W,H,lo,hi", [(16, 723, 597, 0.55, 30.0), (8, 363, 301, 0.55, 30.0),
                                            (16, 1352, 1014, 20.0, 500.0), (16, 1280, 720, 1e3, 1e5),
                                            (8, 640, 480, 100.0, 1e4)])
def test_lists_equal_the_instance_sorts(tile, W, H, lo, hi):
    """The same list, counts and ranges by both routes (visible capacity below
    and above 65,536), at a capacity of exactly the instances."""
    n, ntiles = 30_000, ((W + tile - 1) // tile) * ((H + tile - 1) // tile)
    rng = np.random.default_rng(W + tile)
    rec = _synthetic_records(rng, n, W, H, 24, tile=tile)
    _stretched(rec, rng, lo, hi)
    rec["uv"][::5] = np.floor(rec["uv"][::5]) + np.float32(0.5)
    views = [sy.tiny_view(W, H)]
    a, (code, want) = _run(rec, views, tile, 1 << 23, vis_cap=n)
    assert code == fgs4d.OK and want[1] > n
    b, (code, got) = _run(rec, views, tile, want[1])
    assert code == fgs4d.OK and got == want
    for x, y in zip(_lists(a, want, ntiles), _lists(b, got, ntiles)):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("stage_blocks", [0, 1])
def test_pairs_beyond_the_capacity_whose_masks_are_empty(stage_blocks):
    """Circles of radius 4 px centred (3, 3) px from the corner of four cells:
    four candidate pairs, three with a tile.  At a capacity of exactly the
    instances (fewer than the candidates) the pairs are compacted."""
    n, W, H = 16_384, 640, 512
    rng = np.random.default_rng(9)
    rec = _synthetic_records(rng, n, W, H, 2)
    cx, cy = rng.integers(1, 5, n) * 128.0, rng.integers(1, 4, n) * 128.0
    sx, sy_ = rng.choice([-1.0, 1.0], n), rng.choice([-1.0, 1.0], n)
    rec["uv"] = np.stack([cx + 3 * sx, cy + 3 * sy_], 1).astype(np.float32)
    rec["rect"] = np.stack([cx / 16 - 1, cy / 16 - 1, cx / 16 + 1, cy / 16 + 1], 1).astype(np.int32)
    rec["tau"][:] = 8.0
    k = 8.0 / 4.0 ** 2
    rec["conic2"] = np.tile(np.float32([k, 0.0, k]), (n, 1))
    views, ntiles = [sy.tiny_view(W, H)], 40 * 32
    a, (code, want) = _run(rec, views, 16, 1 << 20, vis_cap=n)
    assert code == fgs4d.OK and want[1] == 3 * n  # of the 4 n candidate pairs
    b, (code, got) = _run(rec, views, 16, want[1], stage_blocks=stage_blocks)
    assert code == fgs4d.OK and got == want
    for x, y in zip(_lists(a, want, ntiles), _lists(b, got, ntiles)):
        np.testing.assert_array_equal(x, y)


def test_lists_do_not_depend_on_the_capacities():
    """The same list at both sides of every line that the capacities draw: the
    binning's route, four slots a thread in the pair scan (2^19), eight keys a
    thread in the depth sort (2^20), three sub-tiles a ticket in the instance
    sort (2^26)."""
    n, W, H = 30_000, 640, 480
    rng = np.random.default_rng(12)
    rec = _synthetic_records(rng, n, W, H, 20)
    _stretched(rec, rng, 2.0, 60.0)
    views, ntiles, want = [sy.tiny_view(W, H)], 40 * 30, None
    for vis_cap, inst_cap in ((n, 1 << 22), (n, 1 << 26), (65_535, 1 << 26), (65_536, 1 << 22), ((1 << 19) - 1, 1 << 22),
                              (1 << 19, 1 << 22), ((1 << 20) - 1, 1 << 22), (1 << 20, 1 << 22)):
        r, (code, counts) = _run(rec, views, 16, inst_cap, vis_cap=vis_cap)
        assert code == fgs4d.OK and counts[1] > 10 * n
        got = [np.array(counts)] + list(_lists(r, counts, ntiles))
        want = want or got
        for x, y in zip(want, got):
            np.testing.assert_array_equal(x, y)
