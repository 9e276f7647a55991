"""Tensors that torch conjugates or negates lazily (x.conj(), z.conj().imag):
every public function takes the values, not the memory behind them."""
import pytest

import paper_2603_27569_gb300 as fg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS, N = 5, 1024


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2603_27569_gb300 import build

    build.build()


def noise(*shape, seed=0):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, dtype=torch.complex64, generator=g).cuda()


def lazy(t):
    v = t.conj()
    assert v.is_conj()
    return v, v.resolve_conj()


@pytest.mark.parametrize("f", [fg.fft, fg.ifft, fg.fft_columns], ids=["fft", "ifft", "columns"])
def test_transforms(f):
    v, x = lazy(noise(ROWS, 16, N) if f is fg.fft_columns else noise(ROWS, N))
    assert torch.equal(f(v), f(x))


def test_host_buffers():
    v, x = lazy(noise(ROWS, N).cpu())
    assert torch.equal(fg.fft_host(v), fg.fft_host(x))


def test_gradient_of_a_transform():
    v, g = lazy(noise(ROWS, N, seed=1))
    grads = [torch.autograd.grad(fg.fft(x), x, w)[0]
             for w in (v, g) for x in [noise(ROWS, N).requires_grad_(True)]]
    assert torch.equal(*grads)


@pytest.mark.parametrize("fused", [True, False])
def test_filter(fused):
    (xv, x), (Hv, H), (gv, g) = (lazy(noise(*s, seed=i)) for i, s in enumerate([(ROWS, N), (N,), (ROWS, N)]))

    def run(x, H, g):
        x, H = x.detach().requires_grad_(True), H.detach().requires_grad_(True)
        y = fg.spectral_filter(x, H, fused)
        return (y.detach(),) + torch.autograd.grad(y, (x, H), g)

    for a, b in zip(run(xv, Hv, gv), run(x, H, g)):
        assert torch.equal(a, b)


def test_step():
    (xv, x), (Hv, H) = lazy(noise(ROWS, N)), lazy(noise(N, seed=1))
    mv = noise(ROWS, N, seed=2).conj().imag
    assert mv.is_neg()
    for a, b in zip(fg.spectral_filter_step(xv, Hv, mv), fg.spectral_filter_step(x, H, mv.resolve_neg())):
        assert torch.equal(a, b)
