"""fft_filter_step with grad_H in memory that it also reads: grad_H is the last
buffer written, so H, a row of x or the mask may hold it."""
import numpy as np
import pytest

import paper_2603_27569_gb300 as fg
from paper_2603_27569_gb300 import synth
from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2603_27569_gb300 import build

    build.build()


# 400 rows: several per CTA at 8192; 37: one ragged tile of several rows at 1024
@pytest.mark.parametrize("N,rows", [(1024, 37), (8192, 400)])
@pytest.mark.parametrize("where", ["H", "x", "mask"])
def test_grad_h_in_an_input(N, rows, where):
    def run(alias):
        x, H = to_dev(synth.gaussian((rows, N), seed=1)), to_dev(synth.gaussian(N, seed=2))
        m = to_dev(synth.real_mask((rows, N), seed=3))
        y, gx = torch.empty_like(x), torch.empty_like(x)
        loss = torch.empty((), device="cuda")
        gH = {"H": H, "x": x[rows // 2], "mask": m[4:6].view(torch.complex64).view(N),
              None: torch.empty_like(H)}[alias]
        plan = fg.fft_filter_plan(N, rows)
        fg.fft_filter_step(plan, x, H, m, y, gx, gH, loss, torch.cuda.current_stream())
        out = [to_host(t) for t in (y, gx, gH, loss)]
        fg.fft_destroy(plan)
        return out

    for a, b in zip(run(None), run(where)):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))


@pytest.mark.parametrize("N,rows", [(1024, 6001), (16384, 160)])
def test_one_grad_h_buffer_for_calls_back_to_back(N, rows):
    # the buffer holds each call's packed H, then its result, with no host
    # synchronisation in between
    x, m = to_dev(synth.gaussian((rows, N), seed=1)), to_dev(synth.real_mask((rows, N), seed=3))
    Hs = [to_dev(synth.gaussian(N, seed=10 + i)) for i in range(6)]
    loss = torch.empty((), device="cuda")
    st = torch.cuda.current_stream()
    plan = fg.fft_filter_plan(N, rows)
    gH = torch.empty_like(Hs[0])
    got = []
    for H in Hs:
        y, gx = torch.empty_like(x), torch.empty_like(x)
        fg.fft_filter_step(plan, x, H, m, y, gx, gH, loss, st)
        got.append((y, gx, gH.clone()))
    fg.fft_destroy(plan)
    for H, outs in zip(Hs, got):
        torch.cuda.synchronize()
        want = fg.spectral_filter_step(x, H, m)
        for a, b in zip(outs, (want[0], want[2], want[3])):
            assert np.array_equal(to_host(a).view(np.uint32), to_host(b).view(np.uint32))
