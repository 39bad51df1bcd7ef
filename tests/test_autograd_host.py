"""The autograd backward on the host, with the library's calls recorded instead
of made: tensors that saved-tensor hooks hand back in another form are refused
before a kernel writes to the gradients shaped like them."""
import types

import pytest
import torch

from paper_2412_20720_gb300 import fgs4d
from paper_2412_20720_gb300 import render as R


def _renderer(n, monkeypatch, calls):
    r = R.Renderer.__new__(R.Renderer)
    r.n, r.device, r.config = n, torch.device("cpu"), R.RenderConfig()
    r.views, r.nviews, r.settings, r.ws, r.ws_bytes = None, 1, None, torch.zeros(1), 0
    r.stream = lambda: 0
    monkeypatch.setattr(fgs4d, "zero_set", lambda tensors, stream: calls.append(("zero", list(tensors))))
    monkeypatch.setattr(fgs4d, "render_bwd", lambda *a: calls.append(("bwd",)))
    return r


def _params(n):
    return [torch.zeros(s) for s in ((n, 4), (n, 4), (n, 4), (n, 4), (n,), (n, 8, 3))]


def _backward(r, saved):
    return R.Render4DGS.backward(types.SimpleNamespace(renderer=r, saved_tensors=saved), torch.zeros(12))


# other element size (a clear of 4 bytes an element would leave the array), other strides, other device
@pytest.mark.parametrize("change", [lambda t: t.half(), lambda t: t.double(),
                                    lambda t: t.transpose(0, -1).contiguous().transpose(0, -1),
                                    lambda t: t.to("meta")])
def test_nothing_is_cleared_before_the_check(monkeypatch, change):
    calls = []
    r = _renderer(5, monkeypatch, calls)
    saved = _params(5)
    saved[5] = change(saved[5])
    with pytest.raises(ValueError):
        _backward(r, saved)
    assert calls == []


def test_every_gradient_is_cleared_before_the_adjoint(monkeypatch):
    calls = []
    r = _renderer(5, monkeypatch, calls)
    out = _backward(r, _params(5))
    assert [c[0] for c in calls] == ["zero", "bwd"]
    assert calls[0][1] == [(g.data_ptr(), g.numel()) for g in out[1:]]
