"""grad_H of batches with hundreds of rows per row slot.  Every row is the same,
so a sum in row order adds the same rounding error again and again, while a
pairwise sum of equal terms is exact: the error says how long the ordered sums
are.  Below 8192 points they run over at most 32 rows."""
import numpy as np
import pytest

import oracle
import paper_2603_27569_gb300 as fg
from paper_2603_27569_gb300 import synth
from gpu_util import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RUN = 32         # rows added in order
U = 2.0 ** -24   # one FP32 rounding
# Two roundings per row, each at most U of the sum so far, which is half the
# whole on average: RUN U.  The ragged tail adds a few levels of the tree (8 U),
# the two transforms 2e-7 each.  640 rows in order come to about 1e-5.
TOL = (RUN + 8) * U + 4e-7


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2603_27569_gb300 import build

    build.build()


@pytest.mark.parametrize("N", [256, 1024, 4096])
def test_ordered_sums_stay_short(N):
    rows = 640 * 456 * 4096 // N + 3  # 640 rounds of three CTAs per SM, 4096 points each
    x, g, H = (synth.gaussian((1, N), seed=N + i) for i in range(3))
    row = fg.fft(to_dev(x))
    X = row.expand(rows, N).contiguous()
    gy = to_dev(g).expand(rows, N).contiguous()
    gx, gH = torch.empty_like(gy), torch.full((N,), float("nan"), dtype=torch.complex64, device="cuda")
    plan = fg.fft_filter_plan(N, rows)
    fg.fft_filter_backward(plan, gy, to_dev(H[0]), X, gx, gH, torch.cuda.current_stream())
    got = to_host(gH).astype(np.complex128)
    fg.fft_destroy(plan)
    G = oracle.fft(g)[0] / N
    want = rows * np.conj(oracle.fft(x)[0]) * G
    assert np.linalg.norm(got - want) <= TOL * np.linalg.norm(want)
    # each launch's rows were transformed: the first, the last, and all equal
    want_gx = N * oracle.ifft(np.conj(H.astype(np.complex128)) * G)
    for r in (0, rows // 2, rows - 1):
        one = to_host(gx[r])
        assert np.linalg.norm(one - want_gx[0]) <= 1e-6 * np.linalg.norm(want_gx)
    assert bool((gx.view(torch.int64) == gx[0].view(torch.int64)).all())
