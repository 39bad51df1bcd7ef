"""fgs4d_zero_set clears every element of its tensors and nothing beside them."""
import pytest

from paper_2412_20720_gb300 import fgs4d


def test_rejects_bad_tables():
    for bad in ([(0, 4)], [(4096 + 4, 4)], [(4096, -1)], [(4096, 1)] * (fgs4d.ADAM_MAX_TENSORS + 1)):
        with pytest.raises(fgs4d.Fgs4dError):
            fgs4d.zero_set(bad, 0)


# empty, below and above one unit of four, a ragged tail
@pytest.mark.gpu
def test_clears_exactly_the_set():
    import torch
    sizes = (0, 1, 3, 4, 5, 1_000_003)
    bufs = [torch.ones(n + 8, device="cuda") for n in sizes]
    fgs4d.zero_set([(b.data_ptr(), n) for b, n in zip(bufs, sizes)], torch.cuda.current_stream().cuda_stream)
    for b, n in zip(bufs, sizes):
        assert not b[:n].any() and bool((b[n:] == 1).all())
