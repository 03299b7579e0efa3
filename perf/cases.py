"""The measured workloads: what a program that uses this library has it do.

Each case is one call pattern of the public interface (`fft3.Plan`, the
batched plans, the cost model's training calls), at sizes of this repository's
benchmark, tests and plan-selection data: single complex64 cubes from 64^3 to
1024^3, mixed-radix and odd boxes, the volumetric decomposition, split-BF16
tensor-core transforms, complex128, batches of uneven boxes, and the training
steps of the plan cost model.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_1904_10119_gb300 import fft3, synth

_DTYPES = {"c64": fft3.FFT3_C64_FP32, "split_bf16": fft3.FFT3_C64_SPLITBF16_TC, "c128": fft3.FFT3_C128_FP64}
# box sides: every 2*3*5-smooth length up to 160, odd ones among them, then the multiples of 16 that large grids use
_SIDES = [n for n in synth.smooth_sizes(4, 1024) if n <= 160 or n % 16 == 0]
_MLP_FEATURES, _MLP_HIDDEN = 32, 64  # the shape of the shipped cost model


def _fft(name, n0, n1, n2, batch=1, dtype="c64", decomposition="auto", direction="forward", values="uniform"):
    case = dict(kind="fft", n0=n0, n1=n1, n2=n2, batch=batch, dtype=dtype, decomposition=decomposition,
                direction=direction, values=values)
    return dict(name=name, **case) if name else case


def _many(name, count, dims_seed, direction="forward"):
    case = dict(kind="many", count=count, dims_seed=dims_seed, direction=direction)
    return dict(name=name, **case) if name else case


def _train(name, batch, steps):
    case = dict(kind="train", batch=batch, steps=steps)
    return dict(name=name, **case) if name else case


def listed():
    return [
        # the paper's smallest cube under its pencil-pencil-pencil decomposition: latency and launches
        _fft("cube64_ppp_forward", 64, 64, 64, decomposition="ppp"),
        # a few equal boxes with odd sides in one plan, back to real space
        _fft("odd_60x45x50_batch8_inverse", 60, 45, 50, batch=8, direction="inverse"),
        # the paper's middle cube, default plan
        _fft("cube256_forward", 256, 256, 256),
        # an ordinary simulation cube on its way back from the spectrum
        _fft("cube512_inverse", 512, 512, 512, direction="inverse"),
        # the benchmark's transform and the largest one
        _fft("cube1024_forward", 1024, 1024, 1024),
        # sides 3*2^k and 5*2^k, the ordinary non-power-of-two box
        _fft("mixed_384x320x240_forward", 384, 320, 240),
        # lines split over cooperating blocks: the paper's volumetric decomposition
        _fft("volumetric_512x512x256_inverse", 512, 512, 256, decomposition="volumetric", direction="inverse"),
        # tensor-core transform of the precision study, on its high-dynamic-range inputs
        _fft("split_bf16_512_hdr_forward", 512, 512, 512, dtype="split_bf16", values="hdr"),
        # the paper's own precision at its middle cube
        _fft("c128_256_forward", 256, 256, 256, dtype="c128"),
        # thousands of uneven boxes in one plan: the batching workload
        _many("many_4096_forward", 4096, 7),
        # a handful of uneven boxes in one plan
        _many("many_24_inverse", 24, 11, direction="inverse"),
        # training the plan cost model: minibatch gradients and Adam updates
        _train("cost_model_16_steps_of_128", 128, 16),
    ]


def _log_pick(rng, values, lo, hi):
    """One of the sorted values in [lo, hi], spread over the logarithm."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ok = [v for v in values if lo <= v <= hi]
    return min(ok, key=lambda v: abs(math.log(v / x)))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "volumetric", "split_bf16", "c128", "many", "train"])
    direction = rng.choice(["forward", "inverse"])
    if kind == "box":
        while True:
            n = [_log_pick(rng, _SIDES, 16, 1024) for _ in range(3)]
            if n[0] * n[1] * n[2] <= 1 << 27:
                break
        room = max(1, (1 << 22) // (n[0] * n[1] * n[2]))
        return _fft(None, *n, batch=rng.randint(1, min(16, room)), direction=direction,
                    decomposition=rng.choice(["auto", "auto", "ppp", "slab_pencil"]))
    if kind == "volumetric":
        n = [rng.choice([64, 128, 256, 512, 1024]), rng.choice([64, 128, 256, 512, 1024]), rng.choice([64, 128, 256, 512])]
        return _fft(None, *n, decomposition="volumetric", direction=direction)
    if kind == "split_bf16":
        n = [rng.choice([128, 256, 512, 1024]), rng.choice([128, 256, 512, 1024]), rng.choice([128, 256, 512])]
        return _fft(None, *n, dtype="split_bf16", direction=direction, values=rng.choice(["uniform", "hdr"]))
    if kind == "c128":
        while True:
            n = [_log_pick(rng, _SIDES, 24, 512) for _ in range(3)]
            if n[0] * n[1] * n[2] <= 1 << 24:
                break
        return _fft(None, *n, dtype="c128", direction=direction)
    if kind == "many":
        return _many(None, int(round(math.exp(rng.uniform(math.log(8), math.log(4096))))), rng.randint(0, 1 << 30),
                     direction=direction)
    return _train(None, rng.randint(32, 1000), rng.randint(4, 32))


# ----------------------------------------------------------------- inputs -- #
def _values(shape, dtype, values, seed):
    """Uniform [-1, 1) parts, or magnitudes log-uniform in [1e-3, 1e3] with uniform phases."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    ctype, rtype = (torch.complex128, torch.float64) if dtype == "c128" else (torch.complex64, torch.float32)
    x = torch.empty(shape, dtype=ctype, device="cuda")
    if values == "hdr":
        mag = torch.pow(10.0, torch.empty(shape, dtype=rtype, device="cuda").uniform_(-3, 3, generator=g))
        ph = torch.empty(shape, dtype=rtype, device="cuda").uniform_(0, 2 * math.pi, generator=g)
        return torch.polar(mag, ph, out=x)
    torch.view_as_real(x).uniform_(-1, 1, generator=g)
    return x


def _dims(case):
    """(dims, offsets, total): the boxes of a batch and where each starts."""
    dims = synth.batched_dims(case["count"], case["dims_seed"])
    vols = dims.prod(axis=1)
    offs = np.concatenate([[0], np.cumsum(vols[:-1])]).astype(np.int64)
    return dims, offs, int(vols.sum())


def _train_data(case, seed):
    """(parameters, X, y): He-style weights, plan features and centred log run times."""
    F, H = _MLP_FEATURES, _MLP_HIDDEN
    rng = np.random.default_rng(seed)
    p = np.concatenate([rng.normal(0, math.sqrt(2 / F), H * F), np.zeros(H), rng.normal(0, math.sqrt(2 / H), H * H),
                        np.zeros(H), rng.normal(0, math.sqrt(2 / H), H), np.zeros(1)]).astype(np.float32)
    n = case["batch"] * case["steps"]
    X = rng.normal(size=(n, F)).astype(np.float32)
    y = (np.tanh(X[:, 0]) + 0.5 * X[:, 1] * X[:, 2] + 0.1 * rng.normal(size=n)).astype(np.float32)
    return p, X, y


class _Many:
    """Owns a batched plan's handle."""

    def __init__(self, case):
        dims, offs, self.total = _dims(case)
        self.handle = fft3.fft3_plan_create_many(dims, offs, direction=_sign(case))

    def __del__(self):
        if getattr(self, "handle", 0):
            fft3.fft3_plan_destroy(self.handle)


def _sign(case):
    return fft3.FFT3_FORWARD if case["direction"] == "forward" else fft3.FFT3_INVERSE


def prepare(case, seed):
    if case["kind"] == "fft":
        x = _values((case["batch"], case["n2"], case["n1"], case["n0"]), case["dtype"], case["values"], seed)
        plan = fft3.Plan(case["n0"], case["n1"], case["n2"], case["batch"],
                         decomposition=fft3.DECOMP[case["decomposition"]], direction=_sign(case),
                         dtype=_DTYPES[case["dtype"]])
        return dict(kind="fft", plan=plan, x=x, out=torch.empty_like(x))
    if case["kind"] == "many":
        plan = _Many(case)
        x = _values((plan.total,), "c64", "uniform", seed)
        return dict(kind="many", plan=plan, x=x, out=torch.empty_like(x))
    p, X, y = _train_data(case, seed)
    B, F = case["batch"], _MLP_FEATURES
    return dict(kind="train", model=fft3.Mlp(F, _MLP_HIDDEN, seed=1), p0=p, batch=B, steps=case["steps"],
                X=torch.from_numpy(X).cuda(), y=torch.from_numpy(y).cuda(), loss=torch.zeros(case["steps"], device="cuda"))


def run(state):
    if state["kind"] == "fft":
        state["plan"].execute(state["x"], state["out"])
        return state["out"]
    if state["kind"] == "many":
        fft3.fft3_plan_execute(state["plan"].handle, state["x"].data_ptr(), state["out"].data_ptr(),
                               torch.cuda.current_stream().cuda_stream)
        return state["out"]
    # one epoch of the user's own loop over the C ABI: gradient and Adam update per minibatch
    L, m, B = fft3.load(), state["model"], state["batch"]
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    m.set_params(state["p0"])
    x, y, loss = state["X"].data_ptr(), state["y"].data_ptr(), state["loss"].data_ptr()
    for k in range(state["steps"]):
        if L.fft3_mlp_grad(m.handle, x + 4 * k * B * _MLP_FEATURES, y + 4 * k * B, B, None, loss + 4 * k, st) or \
                L.fft3_mlp_adam_step(m.handle, None, 1e-3, st):
            raise RuntimeError(fft3.last_error())
    torch.cuda.current_stream().synchronize()  # get_params copies on the default stream
    return {"params": m.get_params(), "loss": state["loss"]}


# --------------------------------------------------------- work, accuracy -- #
def work(case):
    if case["kind"] == "train":
        F, H, B = _MLP_FEATURES, _MLP_HIDDEN, case["batch"]
        p = H * F + H + H * H + H + H + 1
        # inputs and targets in, the parameters in and out; forward, weight and input gradients
        return {"bytes": case["steps"] * (4 * B * (F + 1) + 4) + 8 * p,
                "flops": case["steps"] * B * (2 * (H * F + H * H + H) * 2 + 2 * (H * H + H))}
    if case["kind"] == "many":
        dims, _, total = _dims(case)
        vols = dims.prod(axis=1).astype(np.float64)
        return {"bytes": 16 * total, "flops": float((5 * vols * np.log2(vols)).sum())}
    n = case["n0"] * case["n1"] * case["n2"]
    esize = 16 if case["dtype"] == "c128" else 8
    return {"bytes": 2 * esize * n * case["batch"], "flops": 5 * n * math.log2(n) * case["batch"]}


def tolerance(case):
    # about four times the measured distance from exact(): 2.0e-7 (FP32), 4.5e-6 (split BF16), 5.0e-16 (FP64),
    # 3.5e-7 (a training epoch's losses)
    if case["kind"] == "train":
        return {"rel": 2e-6}
    if case["kind"] == "many" or case["dtype"] == "c64":
        return {"rel": 1e-6}
    return {"rel": 2e-15} if case["dtype"] == "c128" else {"rel": 2e-5}


def _exact_fft(x, forward):
    x = x.to(torch.complex128)
    f = torch.fft.fftn if forward else torch.fft.ifftn
    return f(x, dim=(-3, -2, -1), norm="backward" if forward else "forward")


def _exact_train(case, seed):
    F, H, B = _MLP_FEATURES, _MLP_HIDDEN, case["batch"]
    p, X, y = _train_data(case, seed)
    p, X, y = (torch.from_numpy(v).double().cuda() for v in (p, X, y))
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for t in range(case["steps"]):
        p.requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = torch.split(p, [H * F, H, H * H, H, H, 1])
        xb, yb = X[t * B:(t + 1) * B], y[t * B:(t + 1) * B]
        h = torch.nn.functional.gelu(xb @ w1.view(H, F).T + b1)
        h = torch.nn.functional.gelu(h @ w2.view(H, H).T + b2)
        loss = ((h @ w3 + b3 - yb) ** 2).mean()
        (g,) = torch.autograd.grad(loss, p)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p.detach() - 1e-3 * (m / (1 - 0.9 ** (t + 1))) / ((v / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
        losses.append(loss.detach())
    return {"params": p.cpu().numpy(), "loss": torch.stack(losses)}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    forward = case["direction"] == "forward"
    if case["kind"] == "fft":
        shape = (case["batch"], case["n2"], case["n1"], case["n0"])
        return _exact_fft(_values(shape, case["dtype"], case["values"], seed), forward)
    dims, offs, total = _dims(case)
    x = _values((total,), "c64", "uniform", seed)
    out = torch.empty(total, dtype=torch.complex128, device="cuda")
    for (n0, n1, n2), o in zip(dims.tolist(), offs.tolist()):
        n = n0 * n1 * n2
        out[o:o + n] = _exact_fft(x[o:o + n].view(n2, n1, n0), forward).reshape(-1)
    return out
