"""Workloads of the library as its users call it, for timing and comparison.

A case is a dict of plain values:

  call       "fft2" / "fft1" (the functions, output allocated by the call),
             "plan" (a kept Plan, output buffer given), "fft2_grad" (forward
             and backward through autograd), "loss" (weighted_power_loss,
             forward and backward), "ragged" (a kept RaggedPlan)
  nx, ny, batch, inverse, precision
             as the entry points take them (ny = 1: signals of nx points)
  data       "uniform" U[-1, 1), "normal" N(0, 1) or "tones" (noise plus 8
             unit exponentials per slice)
  count, shapes_seed
             ragged only: instances, and the seed of their shapes (each axis
             a power of two, log-uniform on 32..1024)

Sizes are those of the repository's tests, benchmark and design notes, or
generic ones (image and frame sizes, signal lengths).
"""
import math

import torch

import paper_2506_15437_gb300 as g


def _case(name, call, nx=0, ny=1, batch=1, inverse=False, precision="fp32", data="uniform", count=0, shapes_seed=0):
    c = {"call": call, "nx": nx, "ny": ny, "batch": batch, "inverse": inverse, "precision": precision, "data": data,
         "count": count, "shapes_seed": shapes_seed}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small image, a call at a time: latency of the call and its launches
        _case("image_256", "fft2", 256, 256),
        # the paper's own 2D workload: one megapixel image
        _case("image_1024", "fft2", 1024, 1024, data="normal"),
        # a spectral layer inside a training step on a batch of images
        _case("train_16x1024", "fft2_grad", 1024, 1024, 16, data="normal"),
        # one large field through a kept plan (simulation, imaging)
        _case("field_8192", "plan", 8192, 8192, data="normal"),
        # the same size in the split-FP16 tensor-core precision
        _case("field_8192_split", "plan", 8192, 8192, precision="split_tc", data="tones"),
        # many short signals: channelisers, spectrograms
        _case("signals_4096", "plan", 4096, 1, 16384, data="tones"),
        # a few very long signals, back to the time domain
        _case("long_2p24_inverse", "fft1", 1 << 24, 1, 4, inverse=True),
        # a spectral loss and its gradient (phase retrieval, regularisers)
        _case("loss_8x2048", "loss", 2048, 2048, 8),
        # a batch of patches of mixed sizes in one call
        _case("ragged_512", "ragged", count=512, shapes_seed=2506),
        # signals of a round decimal length
        _case("signals_3000", "plan", 3000, 1, 16384),
        # video frames
        _case("frames_8x1080p", "fft2", 1920, 1080, 8),
        # signals whose length has no small factors
        _case("signals_prime_4093", "fft1", 4093, 1, 16384),
    ]


def _log_int(rng, lo, hi):
    """An integer log-uniform on lo..hi."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _batch(rng, points, lo, hi):
    """A batch that brings slices of `points` to between lo and hi points in all."""
    return max(1, _log_int(rng, max(lo, points), max(hi, points)) // points)


def draw(rng):
    kind = rng.choice(["pow2_2d", "pow2_2d", "pow2_1d", "long", "loss", "ragged", "signals", "signals", "images",
                       "images", "long_any"])
    inv = rng.random() < 0.5
    data = rng.choice(["uniform", "normal", "tones"])
    if kind == "pow2_2d":
        # powers of two on both axes, any aspect ratio
        while True:
            nx, ny = 1 << rng.randint(5, 13), 1 << rng.randint(5, 13)
            if nx * ny <= 1 << 26:
                break
        call = rng.choice(["fft2", "plan", "fft2_grad"])
        split = call == "plan" and min(nx, ny) >= 1024
        return _case("", call, nx, ny, _batch(rng, nx * ny, 1 << 16, 1 << 25), inv, "split_tc" if split else "fp32",
                     data)
    if kind == "pow2_1d":
        n = 1 << rng.randint(6, 13)
        return _case("", rng.choice(["fft1", "plan"]), n, 1, _batch(rng, n, 1 << 16, 1 << 26), inv,
                     data="normal" if data == "tones" else data)
    if kind == "long":
        n = 1 << rng.randint(14, 26)
        return _case("", "fft1", n, 1, _batch(rng, n, 1 << 18, 1 << 26), inv, data="uniform")
    if kind == "loss":
        nx, ny = 1 << rng.randint(6, 12), 1 << rng.randint(6, 12)
        return _case("", "loss", nx, ny, _batch(rng, nx * ny, 1 << 18, 1 << 25), data="uniform")
    if kind == "ragged":
        return _case("", "ragged", count=_log_int(rng, 16, 512), shapes_seed=rng.randint(1, 10 ** 6), inverse=inv)
    if kind == "signals":
        # any length: half of them round numbers, half whatever comes
        n = _log_int(rng, 50, 14000)
        n = max(10, n // 10 * 10) if rng.random() < 0.5 else n
        return _case("", rng.choice(["fft1", "plan"]), n, 1, _batch(rng, n, 1 << 17, 1 << 24), inv, data="uniform")
    if kind == "images":
        # any image size: half of them multiples of 16, as cameras and codecs have them
        nx, ny = _log_int(rng, 60, 4000), _log_int(rng, 60, 4000)
        if rng.random() < 0.5:
            nx, ny = max(64, nx // 16 * 16), max(64, ny // 16 * 16)
        return _case("", rng.choice(["fft2", "fft2_grad"]), nx, ny, _batch(rng, nx * ny, 1 << 16, 1 << 23), inv,
                     data="uniform")
    # long signals of any round length
    n = _log_int(rng, 15, 4000) * 1000
    return _case("", "fft1", n, 1, _batch(rng, n, 1 << 18, 1 << 23), inv, data="uniform")


def _shapes(case):
    gen = torch.Generator().manual_seed(case["shapes_seed"])
    e = torch.randint(5, 11, (case["count"], 2), generator=gen)
    return [1 << int(v) for v in e[:, 0]], [1 << int(v) for v in e[:, 1]]


def _tones(x, gen):
    """Adds 8 unit exponentials at random integer frequencies to each slice of
    x ([batch, ny, nx]; one frequency set for the slices of a 2D batch, one per
    signal otherwise)."""
    b, ny, nx = x.shape
    dev = x.device
    t = torch.arange(nx, device=dev)
    if ny == 1:
        for _ in range(8):
            f = torch.randint(0, nx, (b, 1), generator=gen, device=dev)
            ph = (f * t % nx).to(torch.float32).mul_(2 * math.pi / nx)
            x[:, 0] += torch.polar(torch.ones_like(ph), ph)
        return
    u = torch.arange(ny, device=dev)
    for _ in range(8):
        fx = torch.randint(0, nx, (1,), generator=gen, device=dev)
        fy = torch.randint(0, ny, (1,), generator=gen, device=dev)
        px = (fx * t % nx).to(torch.float32).mul_(2 * math.pi / nx)
        py = (fy * u % ny).to(torch.float32).mul_(2 * math.pi / ny)
        x += torch.polar(torch.ones_like(py), py)[:, None] * torch.polar(torch.ones_like(px), px)[None, :]


def _inputs(case, seed):
    """The call's input arrays, from the seed alone: x, then the upstream
    gradient ("fft2_grad") or the mask ("loss")."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))

    def cplx(shape, data):
        if data == "normal":
            return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device=dev))
        return torch.view_as_complex(torch.rand(*shape, 2, generator=gen, device=dev).mul_(2).sub_(1))

    if case["call"] == "ragged":
        nx, ny = _shapes(case)
        return [cplx((sum(a * b for a, b in zip(nx, ny)),), case["data"])]
    shape = (case["batch"], case["ny"], case["nx"])
    x = cplx(shape, case["data"])
    if case["data"] == "tones":
        _tones(x, gen)
    if case["ny"] == 1:
        x = x.reshape(case["batch"], case["nx"])
    if case["call"] == "fft2_grad":
        return [x, cplx(shape, "normal")]
    if case["call"] == "loss":
        return [x, torch.rand(*shape, generator=gen, device=dev)]
    return [x]


def prepare(case, seed):
    arrays = _inputs(case, seed)
    s = {"case": case, "x": arrays[0]}
    call = case["call"]
    if call == "plan":
        s["plan"] = g.Plan(case["nx"], case["ny"], case["batch"], inverse=case["inverse"],
                           precision=case["precision"])
        s["out"] = torch.empty_like(s["x"])
    elif call == "ragged":
        s["plan"] = g.RaggedPlan(*_shapes(case), inverse=case["inverse"])
        s["out"] = torch.empty_like(s["x"])
    elif call in ("fft2_grad", "loss"):
        s["x"].requires_grad_(True)
        s["other"] = arrays[1]
    return s


def run(state):
    case = state["case"]
    call, x = case["call"], state["x"]
    if call in ("plan", "ragged"):
        return state["plan"].execute(x, out=state["out"])
    if call == "fft2":
        return g.fft2(x, inverse=case["inverse"])
    if call == "fft1":
        return g.fft1(x, inverse=case["inverse"])
    if call == "fft2_grad":
        y = g.fft2(x, inverse=case["inverse"])
        (gx,) = torch.autograd.grad(y, x, state["other"])
        return {"y": y, "grad": gx}
    loss = g.weighted_power_loss(x, state["other"])
    (gx,) = torch.autograd.grad(loss, x)
    return {"loss": loss, "grad": gx}


def work(case):
    """Inputs read once and outputs written once (8 bytes a point each, 4 for
    a mask); 5 N log2 N operations per transform."""
    call = case["call"]
    if call == "ragged":
        sizes = [a * b for a, b in zip(*_shapes(case))]
        return {"bytes": 16 * sum(sizes), "flops": sum(5 * n * math.log2(n) for n in sizes)}
    n = case["nx"] * case["ny"]
    points = n * case["batch"]
    transforms, per_point = {"fft2_grad": (2, 32), "loss": (2, 20)}.get(call, (1, 16))
    return {"bytes": per_point * points, "flops": transforms * 5 * points * math.log2(n)}


def _dft2(x, inverse):
    """Unnormalised transform of [batch, ny, nx] over its last two axes."""
    return torch.fft.ifft2(x, norm="forward") if inverse else torch.fft.fft2(x)


def exact(case, seed):
    arrays = _inputs(case, seed)
    x = arrays[0].to(torch.complex128)
    call, inv = case["call"], case["inverse"]
    if call == "ragged":
        out, at = torch.empty_like(x), 0
        for nx, ny in zip(*_shapes(case)):
            out[at:at + nx * ny] = _dft2(x[at:at + nx * ny].view(ny, nx), inv).reshape(-1)
            at += nx * ny
        return out
    if case["ny"] == 1:
        y = torch.fft.ifft(x, norm="forward") if inv else torch.fft.fft(x)
        return y
    y = _dft2(x, inv)
    if call == "fft2_grad":
        return {"y": y, "grad": _dft2(arrays[1].to(torch.complex128), not inv)}
    if call == "loss":
        w = arrays[1].to(torch.float64)
        return {"loss": (w * (y.real ** 2 + y.imag ** 2)).sum(), "grad": 2 * _dft2(w * y, True)}
    return y
