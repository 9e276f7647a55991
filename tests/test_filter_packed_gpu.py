"""The filter plan's forward and backward with the saved spectrum in natural
and in packed order, at every length: batches that give some CTAs a second
tile and end in a ragged one.  The two orders hold the same numbers, so every
result agrees bit for bit; the natural one is checked against the oracle."""
import numpy as np
import pytest

import oracle
import paper_2603_27569_gb300 as fg
from paper_2603_27569_gb300 import synth
from gpu_util import NTHREADS, TOL_FP32, TOL_GRAD, rel_l2_rows, to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2603_27569_gb300 import build

    build.build()


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# rows: one more than whole rounds of resident CTAs (608 of 4096 / N rows, 304
# at 8192, 152 at 16384), and a single row
@pytest.mark.parametrize("N,rows", [(256, 9729), (512, 4865), (1024, 2433), (2048, 1217),
                                    (4096, 609), (8192, 305), (16384, 153), (256, 1), (1024, 1),
                                    (8192, 1)])
@pytest.mark.parametrize("conj_h", [False, True])
def test_natural_and_packed_spectrum_agree(N, rows, conj_h):
    x = synth.gaussian((rows, N), seed=N)
    H = synth.gaussian(N, seed=N + 1)
    g = synth.gaussian((rows, N), seed=N + 2)
    xd, Hd, gd = to_dev(x), to_dev(H), to_dev(g)
    st = torch.cuda.current_stream()
    plan = fg.fft_filter_plan(N, rows)
    out = []
    for fwd, bwd in ((fg.fft_filter_forward, fg.fft_filter_backward),
                     (fg.fft_filter_forward_packed, fg.fft_filter_backward_packed)):
        y, X, gx = (torch.full_like(xd, float("nan")) for _ in range(3))
        gH = torch.full_like(Hd, float("nan"))
        fwd(plan, xd, Hd, y, X, conj_h, st)
        bwd(plan, gd, Hd, X, gx, gH, st)
        out.append([to_host(t) for t in (y, X, gx, gH)])
    y0 = torch.full_like(xd, float("nan"))
    fg.fft_filter_forward(plan, xd, Hd, y0, None, conj_h, st)
    out[1].append(to_host(y0))
    fg.fft_destroy(plan)
    (y, X, gx, gH), (yp, Xp, gxp, gHp, yn) = out
    for a, b in ((y, yp), (y, yn), (gx, gxp), (gH, gHp)):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    order = lambda r: np.sort(r.view(np.uint64))  # a permutation of each row
    assert np.array_equal(order(X[-1]), order(Xp[-1]))
    pick = np.unique(np.r_[0, rows // 2, rows - 1])
    wantX = oracle.fft(x, nthreads=NTHREADS)
    assert rel_l2_rows(X, wantX).max() <= TOL_FP32
    Hw = np.conj(H) if conj_h else H
    want_y = oracle.ifft(wantX[pick] * Hw.astype(np.complex128))
    assert rel_l2_rows(y[pick], want_y).max() <= 2 * TOL_FP32
    gz = oracle.fft(g, nthreads=NTHREADS) / N
    assert rel(gH, (np.conj(wantX) * gz).sum(0)) <= TOL_GRAD
    want_gx = N * oracle.ifft(np.conj(H.astype(np.complex128)) * gz[pick])
    assert rel(gx[pick], want_gx) <= TOL_GRAD
