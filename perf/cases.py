"""The workloads by which this library's speed is measured.

Each case is one call (or one differentiable forward and backward) through the
public entry points, over the ranges the library is built for: rows of 256 to
2^20 points, columns of 64 to 2^16 points, the spectral filter and its training
step, 16-bit storage, the split-precision transform and ragged batches.
"""
import math

import numpy as np
import torch

import paper_2603_27569_gb300 as fg
from paper_2603_27569_gb300 import synth

POINTS = 1 << 25  # the largest call: 256 MiB of complex64


def listed():
    return [
        # A small burst of short lines: launch and host latency.
        {"name": "burst_256", "kind": "fft", "N": 256, "rows": 256, "inverse": False},
        # One coherent processing block of long range lines: fewer rows than SMs.
        {"name": "block_16384", "kind": "fft", "N": 16384, "rows": 32, "inverse": False},
        # Ordinary bulk range processing, an odd number of lines, back to time.
        {"name": "bulk_4096_odd", "kind": "fft", "N": 4096, "rows": 8191, "inverse": True},
        # The largest one-CTA size at full load.
        {"name": "bulk_16384", "kind": "fft", "N": 16384, "rows": 2048, "inverse": False},
        # Long dwell lines beyond one SM's reach (four-step).
        {"name": "long_131072", "kind": "fft", "N": 131072, "rows": 256, "inverse": False},
        # Azimuth pass of an image: columns of a row-major matrix, no transpose.
        {"name": "azimuth_2048", "kind": "columns", "L": 2048, "cols": 16384, "mats": 1, "inverse": False},
        # Learning a matched filter with any loss: forward and backward through autograd.
        {"name": "train_8192", "kind": "train", "N": 8192, "rows": 4096},
        # The same on short lines and a batch of no special size.
        {"name": "train_1024_odd", "kind": "train", "N": 1024, "rows": 6001},
        # The fused training step for the masked-energy loss.
        {"name": "step_8192", "kind": "step", "N": 8192, "rows": 4096},
        # Archived 16-bit samples transformed in place of a widened copy.
        {"name": "half_4096", "kind": "half", "N": 4096, "rows": 8192, "inverse": False},
        # Split-precision tensor-core transform.
        {"name": "split_4096", "kind": "split", "N": 4096, "rows": 8192, "inverse": False},
        # A mixed batch of sizes and directions in one launch.
        {"name": "ragged_20000", "kind": "ragged", "count": 20000},
    ]


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def _rows(rng, N, most=POINTS):
    return _log_int(rng, max(1, (1 << 16) // N), most // N)


def draw(rng):
    kind = rng.choice(["fft", "fft", "fft", "long", "columns", "columns", "train", "step", "half", "split", "ragged"])
    inverse = rng.random() < 0.5
    if kind == "fft":
        N = 1 << rng.randint(8, 14)
        return {"kind": "fft", "N": N, "rows": _rows(rng, N), "inverse": inverse}
    if kind == "long":
        N = 1 << rng.randint(15, 20)
        return {"kind": "fft", "N": N, "rows": _rows(rng, N), "inverse": inverse}
    if kind == "columns":
        L = 1 << rng.randint(6, 16)
        mats = rng.randint(1, 3)
        tiles = _log_int(rng, 1, max(1, POINTS // (L * 16 * mats)))  # 16 columns each
        return {"kind": "columns", "L": L, "cols": 16 * tiles, "mats": mats, "inverse": inverse}
    if kind in ("train", "step"):
        N = 1 << rng.randint(8, 14)
        return {"kind": kind, "N": N, "rows": _rows(rng, N)}
    if kind == "half":
        N = 1 << rng.randint(8, 14)
        return {"kind": "half", "N": N, "rows": _rows(rng, N), "inverse": inverse}
    if kind == "split":
        N = rng.choice([256, 4096, 16384])
        return {"kind": "split", "N": N, "rows": _rows(rng, N), "inverse": inverse}
    return {"kind": "ragged", "count": _log_int(rng, 100, 20000)}


class _Ragged:
    """A ragged plan that is given back with its owner."""

    def __init__(self, d):
        self.handle = fg.fft_ragged_plan(d["N"], d["direction"], d["offset"], d["offset"])

    def __del__(self):
        fg.fft_destroy(self.handle)


def _noise(shape, g):
    return torch.randn(shape, dtype=torch.complex64, device="cuda", generator=g)


def _pulse(N):
    """A linear-FM pulse of N / 4 samples, -0.4 to +0.4 cycles per sample, zero-padded to N."""
    n = torch.arange(N // 4, dtype=torch.float64, device="cuda")
    phase = 2 * math.pi * (-0.4 * n + 0.4 * n * n / (N // 4))
    p = torch.zeros(N, dtype=torch.complex64, device="cuda")
    p[: N // 4] = torch.polar(torch.ones_like(phase), phase).to(torch.complex64)
    return p


def _echoes(rows, N, g):
    """Range lines: delayed echoes of the pulse with random complex amplitudes, noise 10 dB below."""
    p = _pulse(N)
    x = _noise((rows, N), g) * 0.3
    for _ in range(2):
        delay = int(torch.randint(0, N // 2, (), device="cuda", generator=g))
        x += torch.roll(p, delay) * _noise((rows, 1), g)
    return x, p


def _inputs(case, seed):
    """The tensors of one call, from the seed alone."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    if kind in ("fft", "split"):
        return {"x": _noise((case["rows"], case["N"]), g)}
    if kind == "half":
        x = torch.view_as_real(_noise((case["rows"], case["N"]), g)).to(torch.float16)
        return {"x": torch.view_as_complex(x)}
    if kind == "columns":
        return {"x": _noise((case["mats"], case["L"], case["cols"]), g)}
    if kind in ("train", "step"):
        rows, N = case["rows"], case["N"]
        x, p = _echoes(rows, N, g)
        # a filter some steps into training: the matched filter, perturbed
        H = torch.fft.fft(p).conj() * (1 + 0.1 * _noise((N,), g))
        if kind == "train":
            return {"x": x, "H": H, "gy": _noise((rows, N), g)}
        return {"x": x, "H": H, "mask": torch.rand((rows, N), device="cuda", generator=g)}
    d = synth.ragged_draw(case["count"], seed=case["count"])  # one mix of sizes per case, new data per seed
    return {"d": d, "x": _noise((d["total"],), g)}


def prepare(case, seed):
    s = dict(_inputs(case, seed), case=case)
    if case["kind"] == "train":
        s["layer"] = fg.SpectralFilter(s["H"])
        s["x"].requires_grad_(True)
    elif case["kind"] == "ragged":
        s["plan"] = _Ragged(s["d"])
        s["y"] = torch.empty_like(s["x"])
    return s


def run(s):
    case, x = s["case"], s["x"]
    kind = case["kind"]
    if kind == "fft":
        return fg.fft(x, inverse=case["inverse"])
    if kind == "half":
        return fg.fft(x, inverse=case["inverse"], precision="fp16_storage")
    if kind == "split":
        return fg.fft(x, inverse=case["inverse"], precision="fp16x2")
    if kind == "columns":
        return fg.fft_columns(x, inverse=case["inverse"])
    if kind == "train":
        y = s["layer"](x)
        gx, gH = torch.autograd.grad(y, (x, s["layer"].H), s["gy"])
        return [y.detach(), gx, gH]
    if kind == "step":
        return list(fg.spectral_filter_step(x, s["H"], s["mask"]))
    fg.fft_exec(s["plan"].handle, x, s["y"], torch.cuda.current_stream())
    return s["y"]


def _transform_flops(points, N):
    return 5.0 * points * math.log2(N)


def work(case):
    kind = case["kind"]
    if kind == "ragged":
        d = synth.ragged_draw(case["count"], seed=case["count"])
        return {"bytes": 16 * d["total"], "flops": sum(_transform_flops(int(N), int(N)) for N in d["N"])}
    if kind == "columns":
        points = case["mats"] * case["L"] * case["cols"]
        return {"bytes": 16 * points, "flops": _transform_flops(points, case["L"])}
    N = case["N"]
    points = case["rows"] * N
    flops = _transform_flops(points, N)
    if kind == "half":
        return {"bytes": 8 * points, "flops": flops}
    if kind == "train":  # x and g_y in, y and grad_x out, H in and grad_H out; four transforms
        return {"bytes": 32 * points + 16 * N, "flops": 4 * flops}
    if kind == "step":  # x and the mask in, y and grad_x out
        return {"bytes": 28 * points + 16 * N, "flops": 4 * flops}
    return {"bytes": 16 * points, "flops": flops}


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "ragged":
        d, x = s["d"], s["x"]
        y = torch.empty(x.shape, dtype=torch.complex128, device="cuda")
        for N in np.unique(d["N"]):
            for sign, f in ((-1, torch.fft.fft), (1, torch.fft.ifft)):
                at = d["offset"][(d["N"] == N) & (d["direction"] == sign)]
                index = (torch.from_numpy(at)[:, None] + torch.arange(int(N))[None, :]).cuda()
                y[index] = f(x[index].to(torch.complex128))
        return y
    if kind == "half":
        x = torch.view_as_complex(torch.view_as_real(s["x"]).to(torch.float64))
    else:
        x = s["x"].to(torch.complex128)
    if kind in ("train", "step"):
        N = case["N"]
        H = s["H"].to(torch.complex128)
        X = torch.fft.fft(x)
        y = torch.fft.ifft(X * H)
        gy = s["gy"].to(torch.complex128) if kind == "train" else 2 * s["mask"].to(torch.float64) * y
        gz = torch.fft.fft(gy) / N
        gH = (X.conj() * gz).sum(0)
        gx = torch.fft.ifft(H.conj() * gz) * N
        if kind == "train":
            return [y, gx, gH]
        return [y, (s["mask"].to(torch.float64) * (y.real**2 + y.imag**2)).sum(), gx, gH]
    f = torch.fft.ifft if case["inverse"] else torch.fft.fft
    return f(x, dim=-2 if kind == "columns" else -1)
