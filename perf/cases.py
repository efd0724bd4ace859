"""The work that programs built on this library have it do, as measurable cases.

Every case goes through the public entry points of the Python binding.  Kinds:

* ``step``      one FPO training step: error signal, then the grouped down-projection
                update of every target layer (bf16 or fp32)
* ``error``     the error signal alone (loss, lse and g~ of one batch of tokens)
* ``optimize``  the optimizer form of the update (AdamW or momentum, relative clip)
* ``gate_up``   the W1 / W2 half of a SwiGLU layer: signals through the cached W3_init,
                then the update of both matrices
* ``signals``   the per-layer signals through the post-FFN and / or pre-MLP norms
* ``diagnostic``  pseudogradients of many layers with their cosines to given gradients
* ``ratio``     the update-magnitude ratio ||G_l|| / ||W_l|| of every layer
* ``cosine``    the grouped cosine of given gradients (drawn cases only)

Sizes are those of the repository's workloads and tests, or generic ones of the same
ranges.  Inputs follow the distributions the workloads use: h ~ N(0, 1),
w = 1 + 0.1 N(0, 1), W_U and W ~ N(0, 0.02^2), A = SiLU(N) N, targets Zipf(1.1) or uniform.
"""
import math

import torch

import paper_2608_14563_gb300 as fpo

EPS, MIN_RMS = 1e-6, 0.5


# ------------------------------------------------------------------------ the cases
def listed():
    return [
        # the fp32 workload of the test-suite: a step where launches are all there is
        dict(name="step-f32-tiny", kind="step", dtype="f32", T=128, d=64, d_ff=256, V=512,
             layers=2, targets="uniform", lr=1e-3, grads=False),
        # a short bf16 step with a ragged token count, as a smoke run or a unit test makes it
        dict(name="step-bf16-short", kind="step", dtype="bf16", T=200, d=256, d_ff=384, V=1024,
             layers=2, targets="zipf", lr=1e-2, grads=True),
        # an fp32 reference run at a small model's size, odd token count and vocabulary
        dict(name="step-f32-small-model", kind="step", dtype="f32", T=777, d=768, d_ff=3072,
             V=32001, layers=2, targets="zipf", lr=1e-3, grads=False),
        # one packed 2048-token sequence through a 1B-sized model, G kept for logging
        dict(name="step-bf16-one-sequence", kind="step", dtype="bf16", T=2048, d=2048, d_ff=8192,
             V=50304, layers=4, targets="zipf", lr=1e-4, grads=True),
        # the training batch of the 7B-shaped workload: 8 packed sequences, 8 layers
        dict(name="step-bf16-training-batch", kind="step", dtype="bf16", T=16384, d=4096,
             d_ff=11008, V=100352, layers=8, targets="zipf", lr=1e-4, grads=False),
        # one unpacked document of a few hundred tokens at the 7B shape (adaptation on the fly)
        dict(name="error-bf16-document", kind="error", dtype="bf16", T=333, d=4096, V=100352,
             targets="zipf"),
        # the paper's optimizer setting on two sequences: AdamW, relative clip on the step
        dict(name="adamw-step-clip", kind="optimize", dtype="bf16", T=4096, d=4096, d_ff=11008,
             layers=8, opt="adamw", clip="step"),
        # momentum with the clip on the pseudogradient (the App. A pseudocode), wide d_ff
        dict(name="momentum-gradient-clip", kind="optimize", dtype="bf16", T=2048, d=3072,
             d_ff=23040, layers=3, opt="momentum", clip="gradient"),
        # W1 and W2 of one SwiGLU layer
        dict(name="gate-up-layer", kind="gate_up", dtype="bf16", T=4096, d=4096, d_ff=11008),
        # both per-layer norms for the training batch's 8 layers
        dict(name="signals-both-norms", kind="signals", dtype="bf16", T=16384, d=4096, layers=8,
             post=True, pre=True),
        # the layer-viability diagnostic on a quarter of the 36 layers
        dict(name="diagnostic-cosine", kind="diagnostic", dtype="bf16", T=4096, d=4096,
             d_ff=12288, layers=9),
        # update-magnitude ratios of the training batch's layers: bf16 G, fp32 master
        dict(name="norm-ratio", kind="ratio", d=4096, d_ff=11008, layers=8, g="bf16", w="f32"),
    ]


def _log(rng, lo, hi, mult=1):
    """A size spread over the logarithm of [lo, hi], a multiple of mult."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(max(int(round(v / mult)) * mult, -(-lo // mult) * mult), hi // mult * mult)


def draw(rng):
    kind = rng.choice(["step", "step", "step32", "error", "error", "optimize", "optimize",
                       "gate_up", "signals", "diagnostic", "ratio", "cosine"])
    while True:
        if kind == "step32":
            c = dict(kind="step", dtype="f32", T=_log(rng, 32, 2048), d=_log(rng, 64, 1024),
                     d_ff=_log(rng, 128, 4096), V=_log(rng, 512, 32768), layers=rng.randint(1, 3),
                     targets=rng.choice(["zipf", "uniform"]), lr=1e-3,
                     grads=rng.random() < 0.5)
            if work(c)["flops"] <= 1.2e11:
                return c
            continue
        d = _log(rng, 256, 4096, 8)
        if kind == "step":
            c = dict(kind="step", dtype="bf16", T=_log(rng, 64, 16384), d=d,
                     d_ff=_log(rng, 2 * d, 5 * d, 8), V=_log(rng, 1024, 131072, 8),
                     layers=rng.randint(1, 8), targets=rng.choice(["zipf", "uniform"]), lr=1e-4,
                     grads=rng.random() < 0.5)
        elif kind == "error":
            c = dict(kind="error", dtype="bf16", T=_log(rng, 64, 16384), d=d,
                     V=_log(rng, 1024, 151936, 8), targets=rng.choice(["zipf", "uniform"]))
        elif kind == "optimize":
            c = dict(kind="optimize", dtype="bf16", T=_log(rng, 256, 16384), d=d,
                     d_ff=_log(rng, 2 * d, 5 * d, 8), layers=rng.randint(1, 8),
                     opt=rng.choice(["adamw", "momentum", "sgd"]),
                     clip=rng.choice(["step", "gradient", "none"]))
        elif kind == "gate_up":
            c = dict(kind="gate_up", dtype="bf16", T=_log(rng, 128, 16384), d=d,
                     d_ff=_log(rng, 2 * d, 5 * d, 8))
        elif kind == "signals":
            norms = rng.choice([(True, False), (False, True), (True, True)])
            c = dict(kind="signals", dtype=rng.choice(["bf16", "bf16", "f32"]),
                     T=_log(rng, 64, 16384), d=_log(rng, 256, 8192, 8), layers=rng.randint(1, 9),
                     post=norms[0], pre=norms[1])
        elif kind == "diagnostic":
            c = dict(kind="diagnostic", dtype="bf16", T=_log(rng, 256, 4096), d=d,
                     d_ff=_log(rng, 2 * d, 5 * d, 8), layers=rng.randint(1, 9))
        elif kind == "ratio":
            c = dict(kind="ratio", d=d, d_ff=_log(rng, 2 * d, 5 * d), layers=rng.randint(1, 9),
                     g=rng.choice(["bf16", "f32"]), w=rng.choice(["bf16", "f32"]))
        else:
            c = dict(kind="cosine", d=d, d_ff=_log(rng, 2 * d, 5 * d), layers=rng.randint(1, 9),
                     dtype=rng.choice(["bf16", "f32"]))
        w = work(c)
        if w["flops"] <= 3.8e13 and w["bytes"] <= 2.0e10:
            return c


# ------------------------------------------------------------------------ inputs
def _dt(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


class _Source:
    """Seeded tensors on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def normal(self, *shape, std=1.0, mean=0.0, dtype=torch.float32):
        x = torch.randn(shape, generator=self.gen, device="cuda")
        if std != 1.0:
            x.mul_(std)
        if mean != 0.0:
            x.add_(mean)
        return x.to(dtype)

    def swiglu(self, T, d_ff, dtype):
        a, b = self.normal(T, d_ff), self.normal(T, d_ff)
        return torch.nn.functional.silu(a).mul_(b).to(dtype)

    def targets(self, T, V, how):
        if how == "uniform":
            return torch.randint(0, V, (T,), generator=self.gen, device="cuda", dtype=torch.int32)
        ranks = torch.arange(1, V + 1, device="cuda", dtype=torch.float64)
        cdf = torch.cumsum(ranks.pow(-1.1), 0)
        u = torch.rand((T,), generator=self.gen, device="cuda", dtype=torch.float64)
        idx = torch.searchsorted(cdf / cdf[-1], u, right=True).clamp_(max=V - 1)
        return idx.to(torch.int32)

    def rows(self, T, d, spread, every, at, low, dtype):
        """Rows of log-normal scale, every so many a row of small RMS (the clamp acts there)."""
        scale = torch.exp(spread * self.normal(T, 1))
        scale[at::every] = low
        return (self.normal(T, d) * scale).to(dtype)


# The error signal of a random batch has entries of about this size: 1 / T (the mean's
# factor) times the 0.02 of the unembedding rows.
def _signal_std(T):
    return 0.02 / T


A_RMS = 0.6  # root mean square of SiLU(N) N


def _inputs(c, seed):
    s, kind = _Source(seed), c["kind"]
    dt = _dt(c.get("dtype", "bf16"))
    i = {}
    if kind in ("step", "error"):
        T, d, V = c["T"], c["d"], c["V"]
        i.update(h=s.normal(T, d, dtype=dt), w=s.normal(d, std=0.1, mean=1.0, dtype=dt),
                 W_U=s.normal(V, d, std=0.02, dtype=dt), y=s.targets(T, V, c["targets"]))
    if kind == "step":
        i["A"] = [s.swiglu(c["T"], c["d_ff"], dt) for _ in range(c["layers"])]
        i["W"] = [s.normal(c["d"], c["d_ff"], std=0.02) for _ in range(c["layers"])]
    elif kind == "optimize":
        T, d, d_ff, n = c["T"], c["d"], c["d_ff"], c["layers"]
        i["g"] = s.normal(T, d, std=_signal_std(T), dtype=dt)
        i["A"] = [s.swiglu(T, d_ff, dt) for _ in range(n)]
        i["W"] = [s.normal(d, d_ff, std=0.02) for _ in range(n)]
        # moments as a run in progress has them, at the size of the gradients
        G = _signal_std(T) * A_RMS * math.sqrt(T)
        i["s1"] = [s.normal(d, d_ff, std=0.3 * G) for _ in range(n)] if c["opt"] != "sgd" else None
        i["s2"] = ([s.normal(d, d_ff).square_().add_(0.5).mul_(G * G) for _ in range(n)]
                   if c["opt"] == "adamw" else None)
    elif kind == "gate_up":
        T, d, d_ff = c["T"], c["d"], c["d_ff"]
        i.update(g=s.normal(T, d, std=_signal_std(T), dtype=dt),
                 W3=s.normal(d, d_ff, std=0.02, dtype=dt), a=s.normal(T, d_ff, dtype=dt),
                 b=s.normal(T, d_ff, dtype=dt), x=s.normal(T, d, dtype=dt),
                 W=[s.normal(d_ff, d, std=0.02) for _ in range(2)])
    elif kind == "signals":
        T, d, n = c["T"], c["d"], c["layers"]
        i["g"] = s.normal(T, d, std=_signal_std(T), dtype=dt)
        if c["post"]:
            i["m"] = [s.rows(T, d, 0.5, 64, 0, 0.1, dt) for _ in range(n)]
            i["gp"] = [s.normal(d, std=0.05, mean=0.3, dtype=dt) for _ in range(n)]
        if c["pre"]:
            i["x"] = [s.rows(T, d, 0.3, 64, 32, 0.2, dt) for _ in range(n)]
            i["gq"] = [s.normal(d, std=0.1, mean=1.0, dtype=dt) for _ in range(n)]
    elif kind == "diagnostic":
        T, d, d_ff, n = c["T"], c["d"], c["d_ff"], c["layers"]
        i["g"] = s.normal(T, d, std=_signal_std(T), dtype=dt)
        i["A"] = [s.swiglu(T, d_ff, dt) for _ in range(n)]
        # the 'true' gradients: the pseudogradient plus noise of 4.0 to 1.5 times its size
        i["Y"] = []
        for l, A in enumerate(i["A"]):
            G = torch.matmul(i["g"].t(), A)
            sigma = 4.0 - 2.5 * l / max(n - 1, 1)
            noise = s.normal(d, d_ff, std=sigma * _signal_std(T) * A_RMS * math.sqrt(T))
            i["Y"].append(noise.add_(G).to(dt))
    elif kind == "ratio":
        i["G"] = [s.normal(c["d"], c["d_ff"], std=1e-4, dtype=_dt(c["g"]))
                  for _ in range(c["layers"])]
        i["W"] = [s.normal(c["d"], c["d_ff"], std=0.02, dtype=_dt(c["w"]))
                  for _ in range(c["layers"])]
    elif kind == "cosine":
        i["X"] = [s.normal(c["d"], c["d_ff"], std=1e-4, dtype=dt) for _ in range(c["layers"])]
        i["Y"] = [s.normal(c["d"], c["d_ff"], std=2e-4).add_(X).to(dt) for X in i["X"]]
    return i


def _empty(*shape, dtype):
    return torch.empty(shape, dtype=dtype, device="cuda")


def _bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


OPTS = {"sgd": fpo.OPT_SGD, "momentum": fpo.OPT_SGD_MOMENTUM, "adamw": fpo.OPT_ADAMW}
CLIPS = {"none": fpo.CLIP_NONE, "step": fpo.CLIP_STEP, "gradient": fpo.CLIP_GRADIENT}
OPT_LR, OPT_STEP = 1e-3, 100


def prepare(c, seed):
    """The inputs, and the output buffers and workspaces a training program keeps."""
    i, kind = _inputs(c, seed), c["kind"]
    st = {"case": c, "in": i}
    dt = _dt(c.get("dtype", "bf16"))
    if kind in ("step", "error"):
        T, d, V = c["T"], c["d"], c["V"]
        code = fpo.BF16 if c["dtype"] == "bf16" else fpo.F32
        st["g"] = _empty(T, d, dtype=dt)
        st["lse"], st["loss"] = _empty(T, dtype=torch.float32), _empty(1, dtype=torch.float32)
        st["ws"] = _bytes(fpo.error_signal_workspace(
            fpo.error_signal_desc(T, d, V, code, eps=EPS, min_rms=MIN_RMS)))
    if kind == "step":
        st["Wo"] = [torch.empty_like(W, dtype=dt) for W in i["W"]]
        st["G"] = [torch.empty_like(W, dtype=dt) for W in i["W"]] if c["grads"] else None
        st["ws2"] = _bytes(fpo.layer_update_workspace())
    elif kind == "optimize":
        st["opt"] = fpo.optimizer_desc(OPTS[c["opt"]], lr=OPT_LR, clip=CLIPS[c["clip"]],
                                       step=OPT_STEP)
        st["Wo"] = [torch.empty_like(W, dtype=dt) for W in i["W"]]
        st["ws"] = _bytes(fpo.layer_optimize_workspace(c["layers"], c["d"], c["d_ff"]))
    elif kind == "gate_up":
        st["dA"], st["dB"] = torch.empty_like(i["a"]), torch.empty_like(i["b"])
        st["Wo"] = [torch.empty_like(W, dtype=dt) for W in i["W"]]
        st["ws"] = _bytes(fpo.layer_update_workspace())
    elif kind == "signals":
        st["out"] = [torch.empty_like(i["g"]) for _ in range(c["layers"])]
    elif kind == "diagnostic":
        st["G"] = [_empty(c["d"], c["d_ff"], dtype=dt) for _ in range(c["layers"])]
        st["cos"] = _empty(c["layers"], 4, dtype=torch.float64)
        st["ws"] = _bytes(fpo.layer_grad_cosine_workspace(c["layers"], c["d"], c["d_ff"]))
    elif kind == "ratio":
        st["out"] = _empty(c["layers"], 4, dtype=torch.float64)
        st["ws"] = _bytes(fpo.norm_ratio_workspace(c["layers"], c["d"] * c["d_ff"]))
    elif kind == "cosine":
        st["out"] = _empty(c["layers"], 4, dtype=torch.float64)
        st["ws"] = _bytes(fpo.cosine_grouped_workspace(c["layers"], c["d"] * c["d_ff"]))
    return st


# ------------------------------------------------------------------------ one pass
def run(st):
    c, i = st["case"], st["in"]
    kind = c["kind"]
    if kind in ("step", "error"):
        fpo.error_signal(i["h"], i["w"], i["W_U"], i["y"], st["g"], eps=EPS, min_rms=MIN_RMS,
                         lse_out=st["lse"], loss_out=st["loss"], workspace=st["ws"])
        out = {"g": st["g"], "lse": st["lse"], "loss": st["loss"]}
        if kind == "step":
            fpo.layer_update_grouped(st["g"], i["A"], c["lr"], W_masters=i["W"], W_outs=st["Wo"],
                                     G_outs=st["G"], workspace=st["ws2"])
            out["W"], out["Wo"] = list(i["W"]), list(st["Wo"])
            if st["G"] is not None:
                out["G"] = list(st["G"])
        return out
    if kind == "optimize":
        n = c["layers"]
        fpo.layer_optimize_grouped([i["g"]] * n, i["A"], st["opt"], i["W"], W_outs=st["Wo"],
                                   states1=i["s1"], states2=i["s2"], workspace=st["ws"])
        out = {"W": list(i["W"]), "Wo": list(st["Wo"])}
        if i["s1"] is not None:
            out["s1"] = list(i["s1"])
        if i["s2"] is not None:
            out["s2"] = list(i["s2"])
        return out
    if kind == "gate_up":
        fpo.gate_up_signals(i["g"], i["W3"], i["a"], i["b"], st["dA"], st["dB"],
                            workspace=st["ws"])
        fpo.layer_update_grouped_signals([st["dA"], st["dB"]], [i["x"], i["x"]], 1e-4,
                                         W_masters=i["W"], W_outs=st["Wo"], workspace=st["ws"])
        return {"dA": st["dA"], "dB": st["dB"], "W": list(i["W"]), "Wo": list(st["Wo"])}
    if kind == "signals":
        fpo.layer_signals(i["g"], st["out"], m=i.get("m"), gamma_post=i.get("gp"), x=i.get("x"),
                          gamma_pre=i.get("gq"), eps=EPS, min_rms=MIN_RMS)
        return list(st["out"])
    if kind == "diagnostic":
        fpo.layer_grad_cosine_grouped(i["g"], i["A"], i["Y"], st["G"], st["cos"],
                                      workspace=st["ws"])
        return {"G": list(st["G"]), "cos": st["cos"]}
    if kind == "ratio":
        return fpo.norm_ratio(i["G"], i["W"], 0.01, st["out"], workspace=st["ws"])
    return fpo.cosine_grouped(i["X"], i["Y"], st["out"], workspace=st["ws"])


# ------------------------------------------------------------------------ the work
def work(c):
    """Bytes (each input read once, each output written once) and floating-point operations."""
    kind, e = c["kind"], 2 if c.get("dtype", "bf16") == "bf16" else 4
    b = f = 0.0
    if kind in ("step", "error"):
        T, d, V = c["T"], c["d"], c["V"]
        b += e * (2.0 * T * d + d + V * d) + 8.0 * T + 4  # h, g~, w, W_U; y, lse; loss
        f += 4.0 * T * V * d
    if kind == "step":
        T, n, p = c["T"], c["layers"], c["d"] * c["d_ff"]
        b += n * (e * T * c["d_ff"] + p * (8.0 + e + (e if c["grads"] else 0)))
        f += 2.0 * n * T * p
    elif kind == "optimize":
        T, n, p = c["T"], c["layers"], c["d"] * c["d_ff"]
        states = {"sgd": 0, "momentum": 1, "adamw": 2}[c["opt"]]
        b += e * T * c["d"] + n * (e * T * c["d_ff"] + p * (8.0 + e + 8.0 * states))
        f += 2.0 * n * T * p
    elif kind == "gate_up":
        T, d, d_ff = c["T"], c["d"], c["d_ff"]
        b += e * (2.0 * T * d + d * d_ff + 4.0 * T * d_ff) + 2.0 * d * d_ff * (8 + e)
        f += 6.0 * T * d * d_ff
    elif kind == "signals":
        T, d, n, k = c["T"], c["d"], c["layers"], int(c["post"]) + int(c["pre"])
        b += e * (T * d * (1.0 + n * (k + 1.0)) + n * k * d)
        f += n * T * d * 8.0 * k
    elif kind == "diagnostic":
        T, n, p = c["T"], c["layers"], c["d"] * c["d_ff"]
        b += e * (T * c["d"] + n * (T * c["d_ff"] + 2.0 * p)) + 32.0 * n
        f += n * (2.0 * T * p + 6.0 * p)
    elif kind == "ratio":
        p = c["layers"] * c["d"] * c["d_ff"]
        b += p * ((2.0 if c["g"] == "bf16" else 4) + (2.0 if c["w"] == "bf16" else 4))
        f += 4.0 * p
    elif kind == "cosine":
        p = c["layers"] * c["d"] * c["d_ff"]
        b += 2.0 * e * p
        f += 6.0 * p
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------ tolerances
def tolerance(c):
    kind = c["kind"]
    if kind in ("ratio", "cosine"):
        # 32-bit sums of a few hundred terms, then 64-bit
        return {"rel": 1e-6}
    if c["dtype"] == "f32":
        # sums of up to 32768 32-bit terms in one order or another: 4e-6 from 64 bits
        return {"rel": 1e-5}
    # bf16 results of 32-bit sums, 1.7e-3 from 64 bits by their own rounding; G, which also
    # carries the rounding of g~, 2.4e-3
    return {"rel": 1e-2}


# ------------------------------------------------------------------------ 64 bits
EXACT_FLOPS = 5e12  # a few seconds of fp64 matrix products


def _vjp(g, x, w):
    """RMSNorm's Jacobian at x applied to g; the clamp acts on the 1 / rho prefactor."""
    rho = (x.square().mean(1, keepdim=True) + EPS).sqrt()
    xh, wg = x / rho, w * g
    return (wg - xh * (xh * wg).mean(1, keepdim=True)) / rho.clamp(min=MIN_RMS)


def _exact_error(i, scale):
    W_U, w = i["W_U"].double(), i["w"].double()
    T, rows = i["h"].shape[0], 512
    g, lse = torch.empty_like(i["h"], dtype=torch.float64), []
    ce = torch.zeros((), dtype=torch.float64, device="cuda")
    for t in range(0, T, rows):
        h, y = i["h"][t:t + rows].double(), i["y"][t:t + rows].long()
        z = (h / (h.square().mean(1, keepdim=True) + EPS).sqrt() * w) @ W_U.t()
        l = torch.logsumexp(z, 1)
        ce += (l - z.gather(1, y[:, None])[:, 0]).sum()
        lse.append(l)
        p = z.sub_(l[:, None]).exp_()
        p.scatter_(1, y[:, None], 0.0)
        p.scatter_(1, y[:, None], -p.sum(1, keepdim=True))
        g[t:t + rows] = _vjp(p.mul_(scale) @ W_U, h, w)
    return {"g": g, "lse": torch.cat(lse), "loss": (ce / T)[None]}


def _exact_optimizer(c, W, G, s1, s2):
    lr, frac = OPT_LR, 0.01
    limit = frac * W.norm()
    if c["clip"] == "gradient":
        G = G * torch.clamp(limit / G.norm(), max=1.0)
    if c["opt"] == "sgd":
        step = -lr * G
    elif c["opt"] == "momentum":
        s1 = 0.9 * s1.double() + G
        step = -lr * s1
    else:
        s1 = 0.9 * s1.double() + 0.1 * G
        s2 = 0.999 * s2.double() + 0.001 * G * G
        m, v = s1 / (1 - 0.9 ** OPT_STEP), s2 / (1 - 0.999 ** OPT_STEP)
        step = -lr * (m / (v.sqrt() + 1e-8) + 0.01 * W)
    if c["clip"] == "step":
        step = step * torch.clamp(limit / step.norm(), max=1.0)
    return W + step, s1, s2


def exact(c, seed):
    if work(c)["flops"] > EXACT_FLOPS:
        return None
    i, kind = _inputs(c, seed), c["kind"]
    if kind in ("step", "error"):
        out = _exact_error(i, 1.0 / c["T"])
        if kind == "step":
            G = [out["g"].t() @ A.double() for A in i["A"]]
            out["W"] = [W.double() - c["lr"] * x for W, x in zip(i["W"], G)]
            out["Wo"] = list(out["W"])
            if c["grads"]:
                out["G"] = G
        return out
    if kind == "optimize":
        g, n = i["g"].double(), c["layers"]
        got = [_exact_optimizer(c, i["W"][l].double(), g.t() @ i["A"][l].double(),
                                i["s1"][l] if i["s1"] is not None else None,
                                i["s2"][l] if i["s2"] is not None else None) for l in range(n)]
        out = {"W": [x[0] for x in got], "Wo": [x[0] for x in got]}
        if i["s1"] is not None:
            out["s1"] = [x[1] for x in got]
        if i["s2"] is not None:
            out["s2"] = [x[2] for x in got]
        return out
    if kind == "gate_up":
        a, b, x = i["a"].double(), i["b"].double(), i["x"].double()
        e = i["g"].double() @ i["W3"].double()
        sg = torch.sigmoid(a)
        dA, dB = e * b * sg * (1 + a * (1 - sg)), e * a * sg
        W = [i["W"][k].double() - 1e-4 * (D.t() @ x) for k, D in enumerate((dA, dB))]
        return {"dA": dA, "dB": dB, "W": W, "Wo": list(W)}
    if kind == "signals":
        out, g = [], i["g"].double()
        for l in range(c["layers"]):
            u = g
            if c["post"]:
                u = _vjp(u, i["m"][l].double(), i["gp"][l].double())
            if c["pre"]:
                u = _vjp(u, i["x"][l].double(), i["gq"][l].double())
            out.append(u)
        return out
    if kind == "diagnostic":
        # the sums are those of the stored (bf16) pseudogradient
        g, Gs, rows = i["g"].double(), [], []
        for A, Y in zip(i["A"], i["Y"]):
            G, Y = g.t() @ A.double(), Y.double()
            Gs.append(G)
            rows.append(_cosine(G, Y))
        return {"G": Gs, "cos": torch.stack(rows)}
    if kind == "ratio":
        rows = []
        for G, W in zip(i["G"], i["W"]):
            g2, w2 = G.double().square().sum(), W.double().square().sum()
            r = (g2 / w2).sqrt()
            rows.append(torch.stack([g2, w2, r, 0.01 / r]))
        return torch.stack(rows)
    return torch.stack([_cosine(X.double(), Y.double()) for X, Y in zip(i["X"], i["Y"])])


def _cosine(X, Y):
    xy, xx, yy = (X * Y).sum(), X.square().sum(), Y.square().sum()
    return torch.stack([xy, xx, yy, xy / (xx.sqrt() * yy.sqrt())])
