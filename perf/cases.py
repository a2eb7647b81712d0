"""Performance cases of the sampler and of the recurrent-network workload.

A case is one call (for the recurrent network: one gradient computation) as a user's program makes it, through
the package's public entry points.  A program that samples holds ONE model and draws many batches from it, so
the model of a case is built once from fixed seeds and kept, and the seed of a state makes what changes from call
to call: the random numbers of the batch (or the sequences of the recurrent network).

Families (``case["family"]``):

* ``binary``  bf16 masked MLP with binary positions and logistic noise;
* ``cat``     bf16 masked MLP with 256-way positions, Gumbel noise or one uniform number per position;
* ``f32``     fp32 masked MLP with binary positions and uniform noise;
* ``real``    fp32 masked MLP with continuous states and a stopping tolerance;
* ``conv``    bf16 masked-convolution stack with 256-way sub-pixels and Gumbel noise;
* ``rnn``     loss, exact or Jacobi_n state gradients and parameter gradients of a recurrent network.
"""
import math

import numpy as np
import torch

import paper_2002_03629_b200 as js
from paper_2002_03629_b200 import rnn

MODES = {"jacobi": js.JS_JACOBI, "gs_jacobi": js.JS_GS_JACOBI, "jacobi_gs": js.JS_JACOBI_GS}
REAL_EPS = 0.01


def _mlp(name, family, T, H, batch, mode="jacobi", block=0, noise="logistic", w_var=1.0, b_var=0.0, host=False):
    return {"name": name, "family": family, "T": T, "H": ",".join(str(h) for h in H), "batch": batch, "mode": mode,
            "block": block, "noise": noise, "w_var": w_var, "b_var": b_var, "host": host}


def listed():
    return [
        # the smallest call: a toy model, where launches and latency are everything
        _mlp("tiny_f32", "f32", 16, (64,), 8, noise="uniform"),
        # a binary 28 x 28 image sampler at an ordinary batch
        _mlp("made_784", "binary", 784, (1024, 1024), 256, b_var=0.1),
        # the same kind of sampler on 27 x 27 images with round decimal widths: rows of odd length; 100 images a call
        _mlp("made_729_odd", "binary", 729, (1000, 1000), 100, b_var=0.1),
        # the strict feedforward order on the 28 x 28 model, what a user runs to check or to compare
        _mlp("made_784_sequential", "binary", 784, (1024, 1024), 256, mode="sequential", b_var=0.1),
        # logistic conditionals on 784 real-valued pixels, fp32, stopped at a tolerance
        _mlp("made_784_real", "real", 784, (1024, 1024), 256, w_var=2.0, b_var=0.05),
        # 256 grey levels at 1024 positions: the output layer's weights outweigh everything else
        _mlp("made_cat", "cat", 1024, (2048, 2048), 64, noise="gumbel"),
        # the same model served from host memory: one uniform number per position in, samples out
        _mlp("made_cat_host", "cat", 1024, (2048, 2048), 64, noise="uniform_cat", host=True),
        # the largest masked MLP: 4096 positions, four hidden layers, 512 samples
        _mlp("made_4096", "binary", 4096, (4096, 4096, 4096, 4096), 512, w_var=0.5),
        # the same by Jacobi-GS with blocks of 128 positions, the hybrid its configuration asks for
        _mlp("made_4096_jacobi_gs", "binary", 4096, (4096, 4096, 4096, 4096), 512, mode="jacobi_gs", block=128, w_var=0.5),
        # colour images of 32 x 32 through eight masked convolutions
        {"name": "conv_32", "family": "conv", "height": 32, "width": 32, "in_ch": 3, "ch": 128, "layers": 8, "batch": 16,
         "mode": "jacobi", "block": 0},
        # one sequence at a time, exact gradients: the recurrent network's original training setting
        {"name": "rnn_single", "family": "rnn", "T": 100, "H": 128, "d_in": 1, "d_out": 1, "batch": 1, "n_iters": 0},
        # a large batch of sequences with the truncated Jacobi backward pass
        {"name": "rnn_batch", "family": "rnn", "T": 100, "H": 128, "d_in": 1, "d_out": 1, "batch": 592, "n_iters": 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A hidden width: as often a round number (multiple of 64) as a multiple of 100 or any number at all."""
    w = _log_int(rng, lo, hi)
    step = rng.choice((64, 64, 100, 1))
    return min(hi, max(lo, w // step * step))


def _round_to_8(w):
    return (w + 7) // 8 * 8


def draw(rng):
    family = rng.choice(("binary",) * 8 + ("cat",) * 3 + ("f32",) * 2 + ("real",) * 2 + ("conv",) * 2 + ("rnn",) * 3)
    if family == "binary":
        mode = rng.choice(("jacobi",) * 5 + ("sequential", "gs_jacobi", "jacobi_gs"))
        if mode == "jacobi":         # square images of 8 x 8 to 44 x 44
            side = _log_int(rng, 8, 44)
            H = [_width(rng, 128, 2048) for _ in range(rng.randint(1, 3))]
            block = 0
        else:                        # the solvers that go through positions or blocks in order: up to 28 x 28, even rows
            side = 4 * rng.randint(2, 7)
            H = [_round_to_8(_width(rng, 128, 1024)) for _ in range(rng.randint(1, 3))]
            block = 0 if mode == "sequential" else side * rng.randint(max(1, side // 7), side // 4)
        c = _mlp("", family, side * side, H, _log_int(rng, 1, 512), mode=mode, block=block, w_var=rng.choice((0.5, 1.0)),
                 b_var=rng.choice((0.0, 0.1)))
    elif family == "cat":
        noise = rng.choice(("gumbel", "uniform_cat"))
        c = _mlp("", family, _log_int(rng, 48, 640), [_width(rng, 256, 1536) for _ in range(rng.randint(1, 2))],
                 _log_int(rng, 1, 64), noise=noise, host=noise == "uniform_cat" and rng.random() < 0.5)
    elif family == "f32":
        c = _mlp("", family, _log_int(rng, 12, 256), [_width(rng, 48, 512) for _ in range(rng.randint(1, 2))],
                 _log_int(rng, 1, 64), noise="uniform")
    elif family == "real":
        c = _mlp("", family, _log_int(rng, 48, 784), [_width(rng, 96, 1024) for _ in range(rng.randint(1, 2))],
                 _log_int(rng, 1, 256), w_var=2.0, b_var=0.05)
    elif family == "conv":
        width = rng.choice((16, 32, 32))
        c = {"name": "", "family": family, "height": rng.randint(10, 32), "width": width, "in_ch": rng.choice((1, 3, 3)),
             "ch": rng.choice((64, 128)), "layers": rng.randint(2, 8), "batch": _log_int(rng, 1, 16), "mode": "jacobi",
             "block": 0}
    else:
        c = {"name": "", "family": family, "T": rng.randint(12, 128), "H": 4 * rng.randint(8, 32),
             "d_in": rng.randint(1, 3), "d_out": rng.randint(1, 3), "batch": _log_int(rng, 1, 592),
             "n_iters": rng.choice((0, 0, 5, 10, 20))}
    if family in ("binary", "cat") and any(n % 8 for n in [c["T"], *_widths(c)]):
        # models with rows of any length: no more work than the listed one of their kind
        most = work(next(k for k in listed() if k["name"] == "made_729_odd"))["flops"]
        while c["batch"] > 1 and work(c)["flops"] > most:
            c["batch"] = (c["batch"] + 1) // 2
        if work(c)["flops"] > most:
            c["H"] = ",".join(str(_round_to_8(h)) for h in _widths(c))
            c["T"] = _round_to_8(c["T"])
    del c["name"]
    return c


# ---------------------------------------------------------------- models, from fixed seeds
_model = {}          # the model in use (one at a time): a program keeps the model it samples from


def _randn(g, shape, var):
    return (torch.randn(shape, generator=g, device="cuda") * math.sqrt(var)).cpu().numpy()


def _widths(c):
    return [int(h) for h in c["H"].split(",")]


def _build(c):
    g = torch.Generator("cuda").manual_seed(20020362)
    if c["family"] == "conv":
        W, cin = [], c["in_ch"]
        for _ in range(c["layers"]):
            W.append(_randn(g, (c["ch"], 3, 3, cin), 2.0 / (4.5 * cin)))
            cin = c["ch"]
        W.append(_randn(g, (c["in_ch"] * 256, cin), 1.5 / cin))
        b = [np.zeros(w.shape[0], np.float32) for w in W]
        lut = (np.arange(256) / 127.5 - 1.0).astype(np.float32)
        return js.Model.conv(c["height"], c["width"], c["in_ch"], c["ch"], c["layers"], 256, js.JS_BF16, W, b, lut, c["batch"])
    C = {"cat": 256, "real": 2}.get(c["family"], 1)
    n = [c["T"], *_widths(c), c["T"] * C]
    W = [_randn(g, (n[l + 1], n[l]), c["w_var"] / n[l]) for l in range(len(n) - 1)]
    b = [_randn(g, (n[l + 1],), c["b_var"]) for l in range(len(n) - 1)]
    lut = np.array([0.0, 1.0], np.float32)
    if C == 256:
        lut = (np.arange(256) / 127.5 - 1.0).astype(np.float32)
    if C == 2:                                     # narrow conditionals: damped log-scales around -1
        W[-1][1::2] *= np.float32(0.25)
        b[-1][1::2] -= np.float32(1.0)
    return js.Model.made(c["T"], C, _widths(c), js.JS_ACT_GELU_TANH if C == 256 else js.JS_ACT_RELU,
                         js.JS_F32 if c["family"] in ("f32", "real") else js.JS_BF16, W, b, lut, c["batch"])


def _get_model(c):
    key = tuple(sorted((k, v) for k, v in c.items() if k not in ("name", "mode", "block", "noise", "host")))
    if key not in _model:
        _model.clear()
        _model[key] = _build(c)
    return _model[key]


def _uniform(g, shape):
    """Uniform numbers strictly between 0 and 1 (23 random bits)."""
    return (torch.randint(0, 1 << 23, shape, generator=g, device="cuda").to(torch.float32) + 0.5) * 2.0 ** -23


def _sequences(g, c):
    """Images of three soft strokes read pixel by pixel, and the next pixel as the target."""
    B, T, side = c["batch"], c["T"], math.ceil(math.sqrt(c["T"]))
    at = torch.arange(side, device="cuda", dtype=torch.float32)
    p = torch.rand((B, c["d_in"], 3, 4, 1, 1), generator=g, device="cuda")
    cy, cx = 1 + p[:, :, :, 0] * (side - 3), 1 + p[:, :, :, 1] * (side - 3)
    sy, sx = 0.6 + 1.4 * p[:, :, :, 2], 0.6 + 1.4 * p[:, :, :, 3]
    img = torch.exp(-0.5 * (((at[:, None] - cy) / sy) ** 2 + ((at[None, :] - cx) / sx) ** 2)).sum(2).clamp(0, 1)
    x = img.reshape(B, c["d_in"], side * side)[:, :, :T].permute(0, 2, 1).contiguous()
    r = torch.zeros((B, T, c["d_out"]), device="cuda")
    k = min(c["d_in"], c["d_out"])
    r[:, :-1, :k] = x[:, 1:, :k]
    return x, r


def prepare(case, seed):
    c = case
    g = torch.Generator("cuda").manual_seed(seed)
    if c["family"] == "rnn":
        w = torch.Generator("cuda").manual_seed(20020362)
        H, d_in, d_out = c["H"], c["d_in"], c["d_out"]

        def normal(*shape):
            return torch.randn(shape, generator=w, device="cuda") * 0.1
        x, r = _sequences(g, c)
        return {"case": c, "Wh": normal(H, H), "Wx": normal(H, d_in), "b": torch.zeros(H, device="cuda"),
                "Wo": normal(d_out, H), "bo": torch.zeros(d_out, device="cuda"), "x": x, "r": r}
    model = _get_model(c)
    B = c["batch"]
    T = c["height"] * c["width"] * c["in_ch"] if c["family"] == "conv" else c["T"]
    kind = "gumbel" if c["family"] == "conv" else c["noise"]
    u = _uniform(g, (B, T, 256) if kind == "gumbel" else (B, T))
    if kind == "gumbel":
        noise, nk = -torch.log(-torch.log(u)), js.JS_NOISE_GUMBEL
    elif kind == "logistic":
        noise, nk = torch.log(u) - torch.log1p(-u), js.JS_NOISE_LOGISTIC
    else:
        noise, nk = u, js.JS_NOISE_UNIFORM_CAT if kind == "uniform_cat" else js.JS_NOISE_UNIFORM_ICDF
    out = torch.empty((B, T), dtype=torch.float32 if c["family"] == "real" else torch.uint8, device="cuda")
    if c.get("host"):
        noise, out = noise.cpu().pin_memory(), torch.empty((B, T), dtype=torch.uint8).pin_memory()
    return {"case": c, "model": model, "noise": noise, "nk": nk, "out": out}


def run(state):
    c = state["case"]
    if c["family"] == "rnn":
        Wh, x = state["Wh"], state["x"]
        h, d, l, loss = rnn.rnn_forward(Wh, state["Wx"], state["b"], state["Wo"], state["bo"], x, state["r"])
        if c["n_iters"] > 0:
            s = rnn.rnn_bptt_jacobi(Wh, l, d, c["n_iters"])
        else:
            s = rnn.rnn_bptt_sequential(Wh, l, d)
        dWh, dWx, db = rnn.rnn_param_grads(s, d, h, x)
        return {"loss": loss, "h": h, "s": s, "dWh": dWh, "dWx": dWx, "db": db}
    model, noise, nk, out = state["model"], state["noise"], state["nk"], state["out"]
    if c["family"] == "real":
        js.jacobi_sample_real(model, noise, None, js.JS_JACOBI, 0, 0, REAL_EPS, out)
    elif c["mode"] == "sequential":
        js.sequential_sample(model, noise, nk, out)
    elif c.get("host"):
        js.jacobi_sample_host(model, noise, nk, None, MODES[c["mode"]], c["block"], 0, out)
    else:
        js.jacobi_sample(model, noise, nk, None, MODES[c["mode"]], c["block"], 0, out)
    return out


# ---------------------------------------------------------------- what a pass cannot do without
def _mlp_macs(c, C):
    """Unmasked multiply-accumulates of the network for one sample, every unit evaluated once."""
    T = c["T"]
    deg = [np.arange(1, T + 1)] + [1 + np.arange(h) * (T - 1) // h for h in _widths(c)]
    deg.append(np.repeat(np.arange(1, T + 1), C))
    macs = 0
    for l in range(len(deg) - 1):
        macs += int(np.searchsorted(deg[l], deg[l + 1], side="left" if l == len(deg) - 2 else "right").sum())
    return macs


def work(case):
    """One evaluation of every unit (of every state gradient, for the recurrent network one Jacobi iteration per
    requested iteration), every input and every unmasked weight read once, every output written once."""
    c = case
    B = c["batch"]
    if c["family"] == "rnn":
        T, H, di, do = c["T"], c["H"], c["d_in"], c["d_out"]
        params = 4 * (H * H + H * di + H + do * H + do)
        # read x and r, write h, s and the gradients; h, d, l and s once more on their way through the three calls
        io = 4 * B * (T * (di + do) + 2 * T * H + H * H + H * di + H + 1)
        back = max(1, c["n_iters"]) * H * H
        return {"bytes": params + io, "flops": 2.0 * B * T * (H * (H + di + do) + back + H * do + H * (H + di))}
    if c["family"] == "conv":
        ch, ic = c["ch"], c["in_ch"]
        grp = ic * np.arange(ch) // ch
        macs = 0
        for l in range(c["layers"]):
            gi = np.arange(ic) if l == 0 else grp
            centre = (gi[None, :] < grp[:, None]) if l == 0 else (gi[None, :] <= grp[:, None])
            macs += 4 * len(gi) * ch + int(centre.sum())
        macs += int((grp[None, :] <= (np.arange(ic * 256) // 256)[:, None]).sum())
        pixels = c["height"] * c["width"]
        return {"bytes": 2.0 * macs + B * pixels * ic * (1024 + 1), "flops": 2.0 * macs * pixels * B}
    C = {"cat": 256, "real": 2}.get(c["family"], 1)
    macs = _mlp_macs(c, C)
    size = 4 if c["family"] in ("f32", "real") else 2
    noise = 4 * c["T"] * (C if c["noise"] == "gumbel" else 1)
    return {"bytes": float(macs * size + B * (noise + c["T"] * (4 if C == 2 else 1))), "flops": 2.0 * macs * B}


def tolerance(case):
    """Samples are whole numbers, decided by a comparison of a logit with noise: two correct implementations differ
    where the two scores of a decision are closer than the rounding of the sums (fp32; bf16 hidden units that round
    the other way), and in the few later positions that such a decision moves.  Deep bf16 convolution stacks
    compound those roundings over layers.  Continuous states and gradients are sums in fp32; a sample that stops
    one iteration earlier or later moves by at most the stopping tolerance."""
    if case["family"] == "rnn":
        return {"rel": 1e-5}
    if case["family"] == "real":
        return {"rel": 1e-4, "max": 2 * REAL_EPS}
    return {"rel": 0.0, "differ": 1e-2 if case["family"] == "conv" else 1e-3}
