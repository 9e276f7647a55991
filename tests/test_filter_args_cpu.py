"""What the spectral filter refuses, and the buffers that it hands to the
library: the C calls are replaced by recorders, so nothing needs a GPU."""
import types

import pytest

torch = pytest.importorskip("torch")

import paper_2603_27569_gb300 as fg
from paper_2603_27569_gb300 import torch_api

N, ROWS = 256, 3


@pytest.fixture
def calls(monkeypatch):
    """(name, grad_H buffer or None) of every library call."""
    log = []
    at = {"fft_filter_forward_packed": None, "fft_filter_backward_packed": 5, "fft_filter_step": 6,
          "fft_filter_apply": None, "fft_filter_grad_h": 2}
    for name, i in at.items():
        monkeypatch.setattr(torch_api.B, name, lambda *a, name=name, i=i: log.append(
            (name, None if i is None else a[i])))
    monkeypatch.setattr(torch_api, "_filter_plan", lambda *a: types.SimpleNamespace(handle=1))
    monkeypatch.setattr(torch_api, "_raw_stream", lambda index: 0)
    monkeypatch.setattr(torch_api, "_raw", lambda x, *a, **k: log.append(("raw", None)) or x)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: None)
    return log


def c64(*shape, **kw):
    return torch.ones(shape, dtype=torch.complex64, **kw)


BAD_H = {
    "half as long": (c64(N // 2), ValueError),
    "real": (torch.ones(N), TypeError),
    "real, interleaved": (torch.ones(N, 2), TypeError),
    "double": (torch.ones(N, dtype=torch.complex128), TypeError),
    "two filters": (c64(2, N), ValueError),
    "no dimension": (c64(), ValueError),
    "elsewhere": (c64(N, device="meta"), ValueError),
}


@pytest.mark.parametrize("which", list(BAD_H))
@pytest.mark.parametrize("call", ["fused", "separate", "step"])
def test_unusable_filters_are_refused_before_any_launch(calls, call, which):
    H, error = BAD_H[which]
    x = c64(ROWS, N)
    with pytest.raises(error):
        if call == "step":
            fg.spectral_filter_step(x, H, torch.ones(ROWS, N))
        else:
            fg.spectral_filter(x, H, fused=call == "fused")
    assert not calls


@pytest.mark.parametrize("x", [torch.ones(ROWS, N), torch.ones(ROWS, N, dtype=torch.complex128)])
def test_rows_of_another_type_are_refused(calls, x):
    for f in (lambda: fg.spectral_filter(x, c64(N)),
              lambda: fg.spectral_filter_step(x, c64(N), torch.ones(ROWS, N))):
        with pytest.raises(TypeError):
            f()
    assert not calls


def test_a_mask_elsewhere_is_refused(calls):
    with pytest.raises(ValueError):
        fg.spectral_filter_step(c64(ROWS, N), c64(N), torch.ones(ROWS, N, device="meta"))
    assert not calls


@pytest.mark.parametrize("shape", [(N,), (1, N)])
def test_grad_h_buffer_is_n_points(calls, shape):
    x, H = c64(ROWS, N), c64(*shape, requires_grad=True)
    y = fg.spectral_filter(x, H)
    if shape == (N,):
        y.backward(torch.ones_like(y))
        assert H.grad.shape == (N,)
    else:  # the gradient is the [N] filter's: autograd refuses it for another shape
        with pytest.raises(RuntimeError, match="shape"):
            y.backward(torch.ones_like(y))
    assert fg.spectral_filter_step(x, H, torch.ones(ROWS, N))[3].shape == (N,)
    sums = [b for _, b in calls if b is not None]
    assert len(sums) == 2
    for b in sums:
        assert b.shape == (N,) and b.dtype == torch.complex64 and b.device == x.device
