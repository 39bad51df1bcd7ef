"""Instance emission where most depth-sorted positions hold no pair, so that
one chunk of 2048 pairs spans more positions than its caches hold."""
import numpy as np
import pytest

import oracle
from paper_2412_20720_gb300 import fgs4d
from paper_2412_20720_gb300 import synthetic as sy
from paper_2412_20720_gb300.render import RenderConfig, Renderer
from helpers import canonical_ranges
from test_gpu_parity import KEEP_ALL, _read_instances, _synthetic_records, _write_records

pytestmark = pytest.mark.gpu


# 2048 positions of a chunk fit the cache, 2049 do not
@pytest.mark.parametrize("n,every", [(2048, 2048), (2049, 2049), (9001, 8), (30_001, 40)])
def test_positions_without_pairs(n, every):
    W, H = 320, 240
    rng = np.random.default_rng(n)
    rec = _synthetic_records(rng, n, W, H, 3, tau=KEEP_ALL)
    rank = np.argsort(np.argsort(rec["depth"], kind="stable"))
    keep = (rank % every == 0) | (rank == n - 1)  # the first and last position of the order hold pairs
    rec["rect"][:, 2:] = np.where(keep[:, None], np.minimum(rec["rect"][:, :2] + 2, [W // 16, H // 16]), rec["rect"][:, :2])
    keys, vals, ranges = oracle.sort_instances(rec["rect"], rec["depth"], W // 16, H // 16)
    m = keys.shape[0]
    r = Renderer(n, [sy.tiny_view(W, H)], RenderConfig(sh_degree=0, t_order=0, inst_capacity=m))
    _write_records(r, rec, 0)
    fgs4d.bin_sort(n, r.views, r.nviews, r.settings, r.ws.data_ptr(), r.ws_bytes, r.stream())
    code, counts = r.status()
    assert code == fgs4d.OK and counts[1] == m
    tiles, slots, gr = _read_instances(r, m, (W // 16) * (H // 16))
    np.testing.assert_array_equal(tiles, (keys >> np.uint64(32)).astype(np.int64))
    np.testing.assert_array_equal(slots, vals)
    np.testing.assert_array_equal(canonical_ranges(gr), ranges)
