"""The calls whose speed this library is judged by, with their inputs, costs and tolerances.

Every case is one call that a training program makes once per optimizer step, through the
public binding (paper_2608_05088_gb300.malt): a MALT, MALTER or Muon step over a list of
2-D weight matrices, the whole-optimizer step of a model, AdamW on the tensors that are
not matrices, a step with gradients and weights in host memory, and the statistics stage
alone.  The state is that of a run under way (step 100): gradients are
z * a_i * b_j with z ~ N(0, 1) and log-normal row and column scales a, b, the momentum is
the stationary average of such gradients, the row and column statistics are their
expected squares, and the weights are N(0, 0.02^2).
"""
import math

import numpy as np
import torch

from paper_2608_05088_gb300 import inputs, malt

MU1, MU2, EPS, NS_EPS = 0.95, 0.99, 1e-8, 1e-7
BETA1, BETA2 = 0.9, 0.95
NS_COEFFS = (3.4445, -4.7750, 2.0315)
T0 = 100                      # steps already taken
DECAY = 0.1                   # weight decay of the whole-optimizer step's matrices and embeddings
ALIGN = 64                    # elements between the starts of two tensors of a flat buffer
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
DEV = "cuda"


def _case(name, path, **kw):
    d = {"name": name, "path": path, "shapes": "", "copies": 1, "variant": "malt",
         "weights": "bf16", "grads": "f32", "sigma": 1.5, "ns_steps": 5, "lr": 0.02, "layers": 0, "width": 0}
    d.update(kw)
    return d


def _layer(d):
    return "%dx%d %dx%d %dx%d %dx%d" % (d, 3 * d, d, d, d, 4 * d, 4 * d, d)


def listed():
    return [
        # The smallest model a user steps: one fp32 matrix.  Launches and latency count.
        _case("single_256x512", "step", shapes="256x512", weights="f32", sigma=1.0),
        # A small network of odd layer sizes (every matrix padded inside the library), fp32
        # weights, bf16 gradients, MALTER.
        _case("odd_sizes", "step", shapes="509x251 77x300 129x515 3x250 251x509 300x77", weights="f32",
              grads="bf16", variant="malter"),
        # The GPT-2 parameter sets at their learning rates: the optimizer step of a training run.
        _case("gpt2_small", "step", shapes=_layer(768), copies=12, lr=0.0013),
        _case("gpt2_medium_malter", "step", shapes=_layer(1024), copies=24, variant="malter", lr=0.009),
        _case("gpt2_large", "step", shapes=_layer(1280), copies=36, lr=0.0007),
        # One transformer layer, stepped alone (as when the optimizer is interleaved with the
        # backward pass), Muon through the same engine, bf16 gradients.
        _case("layer_1280_muon", "step", shapes=_layer(1280), variant="muon", grads="bf16"),
        # One large matrix: square, and tall at the longer Newton-Schulz run and widest scales.
        _case("square_4096", "step", shapes="4096x4096", sigma=1.0),
        _case("tall_16384x4096", "step", shapes="16384x4096", sigma=3.0, ns_steps=8),
        # The whole optimizer of GPT-2 Small: fp32 master weights with bf16 copies, weight decay,
        # AdamW on the embeddings, LayerNorms and biases.
        _case("gpt2_small_whole", "whole", shapes=_layer(768), copies=12, weights="f32", lr=0.0013,
              layers=12, width=768),
        # The same set with gradients arriving from pinned host memory and weights going back.
        _case("gpt2_small_host", "host", shapes=_layer(768), copies=12, lr=0.0013),
        # AdamW alone on GPT-2 Medium's other tensors.
        _case("adamw_gpt2_medium", "adamw", layers=24, width=1024, weights="f32", lr=0.0009),
        # The statistics stage alone, with caller-provided outputs and no allocation.
        _case("stats_1280x5120", "stats", shapes="1280x5120"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A layer size: usually a multiple of 64 or 8, now and then odd."""
    n = _log_int(rng, lo, hi)
    step = rng.choice([64, 64, 8, 8, 1])
    return max(1, n // step * step) if n >= step else n


def draw(rng):
    path = rng.choice(["step"] * 7 + ["whole", "host", "adamw", "stats"])
    sigma = rng.choice([0.0, 1.0, 1.5, 3.0])
    grads = rng.choice(["f32", "f32", "bf16"])
    if path in ("whole", "adamw"):
        width = 64 * rng.randint(4, 20)
        layers = _log_int(rng, 1, 24)
        if path == "adamw":
            return _draw(path, layers=layers, width=width, weights="f32", lr=0.0009)
        return _draw(path, shapes=_layer(width), copies=layers, weights="f32", sigma=sigma,
                     lr=rng.choice([0.0007, 0.0013, 0.02]), layers=layers, width=width,
                     variant=rng.choice(["malt", "malter"]))
    if path == "stats":
        return _draw(path, shapes="%dx%d" % (_size(rng, 8, 4096) // 8 * 8 or 8, _size(rng, 8, 4096) // 8 * 8 or 8),
                     sigma=sigma, grads=grads)
    kinds = rng.randint(1, 4)
    shapes = []
    for _ in range(kinds):
        m, n = _size(rng, 16, 4096), _size(rng, 16, 8192)
        if rng.random() < 0.3:            # a multiple of the other side, as in transformer layers
            n = min(4 * m, 8192)
        shapes.append((m, n) if rng.random() < 0.7 else (n, m))
    if path == "host":
        shapes = [(m, n) for m, n in shapes if m * n <= 1 << 22] or [(768, 2304)]
    ns_steps = rng.choice([5, 5, 5, 8, 3])
    flops = sum(_ns_flops(m, n, ns_steps) for m, n in shapes)
    elems = sum(m * n for m, n in shapes)
    most = max(1, min(24, int(6e12 / flops), int((64e6 if path == "host" else 256e6) / elems)))
    return _draw(path, shapes=" ".join("%dx%d" % s for s in shapes), copies=_log_int(rng, 1, most),
                 variant="malt" if path == "host" else rng.choice(["malt", "malt", "malter", "muon"]),
                 weights=rng.choice(["bf16", "bf16", "f32"]), grads=grads, sigma=sigma, ns_steps=ns_steps,
                 lr=rng.choice([0.0007, 0.02]))


def _draw(path, **kw):
    d = _case("", path, **kw)
    del d["name"]
    return d


# ------------------------------------------------------------------ inputs
def _shapes(case):
    one = [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split()]
    return one * case["copies"]


def _ns_flops(m, n, steps):
    """Newton-Schulz with symmetric products counted once: p^2 q + p^3 + 2 p^2 q per iteration."""
    p, q = min(m, n), max(m, n)
    return (3.0 * p * p * q + float(p) ** 3) * steps


def _adam_tensors(case):
    """(shape, weight decay) of the tensors of a GPT-2 model that are not matrices of a layer: token and
    position embeddings, per layer the LayerNorm gains and biases and the Linear biases, the last LayerNorm."""
    d = case["width"]
    layer = [(d,), (d,), (3 * d,), (d,), (d,), (d,), (4 * d,), (d,)]
    return ([((inputs.GPT2_VOCAB, d), DECAY), ((inputs.GPT2_BLOCK, d), DECAY)]
            + [(s, 0.0) for s in layer * case["layers"]] + [((d,), 0.0), ((d,), 0.0)])


def _flat(counts, dtype, device=DEV):
    """One zeroed buffer holding tensors of the given element counts at aligned offsets, and their views."""
    offs, at = [], 0
    for c in counts:
        offs.append(at)
        at += -(-c // ALIGN) * ALIGN
    buf = torch.zeros(max(at, 1), dtype=dtype, device=device)
    return buf, [buf[o:o + c] for o, c in zip(offs, counts)]


class _Matrices:
    """The matrices of a case and their state at step T0, in flat buffers."""

    def __init__(self, case, seed):
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        self.shapes = shapes = _shapes(case)
        n = [a * b for a, b in shapes]
        self.w, W = _flat(n, DTYPES[case["weights"]])
        self.g, G = _flat(n, DTYPES[case["grads"]])
        self.m, M = _flat(n, torch.float32)
        self.l, L = _flat([a for a, _ in shapes], torch.float32)
        self.r, R = _flat([b for _, b in shapes], torch.float32)
        self.views = [(W[i].view(s), G[i].view(s), M[i].view(s), L[i], R[i]) for i, s in enumerate(shapes)]
        sig = case["sigma"]
        self.scales = []
        for (a, b), (w, gr, _, _, _) in zip(shapes, self.views):
            ra = torch.exp(sig * torch.randn(a, generator=g, device=DEV))
            rb = torch.exp(sig * torch.randn(b, generator=g, device=DEV))
            self.scales.append((ra, rb))
            w.copy_(0.02 * torch.randn(a, b, generator=g, device=DEV))
            gr.copy_(torch.randn(a, b, generator=g, device=DEV).mul_(ra[:, None]).mul_(rb[None, :]))
        self.gen = g

    def under_way(self):
        """Fill M, l, r with their values at step T0 and return MALTER's nu per matrix."""
        nu = []
        spread = math.sqrt((1 - MU1) / (1 + MU1))        # an EMA of independent draws
        for (ra, rb), (_, _, m, l, r) in zip(self.scales, self.views):
            m.copy_(torch.randn(m.shape, generator=self.gen, device=DEV).mul_(ra[:, None]).mul_(rb[None, :]).mul_(spread))
            a2, b2 = ra.double() ** 2, rb.double() ** 2
            full = 1.0 - MU2 ** T0
            le, re_ = full * a2 * b2.sum(), full * b2 * a2.sum()
            l.copy_(le)
            r.copy_(re_)
            nu.append(full * ((le + EPS) ** -0.25 * a2).sum() * ((re_ + EPS) ** -0.25 * b2).sum())
        return torch.stack(nu).cpu().numpy().astype(np.float32) if nu else np.zeros(0, np.float32)


class _Others:
    """The AdamW tensors of a case and their moments at step T0, in flat buffers."""

    def __init__(self, case, seed):
        g = torch.Generator(device=DEV)
        g.manual_seed(seed + 1_000_003)
        self.spec = spec = _adam_tensors(case)
        n = [int(np.prod(s)) for s, _ in spec]
        self.w, W = _flat(n, torch.float32)
        self.c, C = _flat(n, torch.bfloat16)
        self.g, G = _flat(n, torch.float32)
        self.m, M = _flat(n, torch.float32)
        self.v, V = _flat(n, torch.float32)
        self.views = [(W[i], C[i], G[i], M[i], V[i], spec[i][1]) for i in range(len(n))]
        self.scale = torch.exp(case["sigma"] * torch.randn(self.w.numel(), generator=g, device=DEV))
        self.w.copy_(0.02 * torch.randn(self.w.numel(), generator=g, device=DEV))
        self.g.copy_(torch.randn(self.w.numel(), generator=g, device=DEV) * self.scale)
        self.gen = g

    def under_way(self):
        self.m.copy_(torch.randn(self.w.numel(), generator=self.gen, device=DEV) * self.scale
                     * math.sqrt((1 - BETA1) / (1 + BETA1)))
        self.v.copy_(self.scale * self.scale * (1 - BETA2 ** T0))


def prepare(case, seed):
    path = case["path"]
    st = {"path": path, "variant": case["variant"]}
    hp = dict(lr=case["lr"], mu1=MU1, mu2=MU2, eps=EPS, ns_steps=case["ns_steps"])
    if path == "adamw":
        o = st["others"] = _Others(case, seed)
        st["opt"] = malt.AdamW(o.views)
        o.under_way()
        st["opt"].set_step(T0)
        st["hp"] = malt.adamw_hparams(lr=case["lr"], betas=(BETA1, BETA2), eps=EPS)
        return st
    x = st["mats"] = _Matrices(case, seed)
    if path == "stats":
        x.under_way()
        _, _, _, l, r = x.views[0]
        st["out"] = (torch.empty_like(l), torch.empty_like(r))
        return st
    if path == "whole":
        o = st["others"] = _Others(case, seed)
        st["copies"], cv = _flat([a * b for a, b in x.shapes], torch.bfloat16)
        st["opt"] = malt.WholeOptimizer(x.views, o.views, copies=[c.view(s) for c, s in zip(cv, x.shapes)])
        nu = x.under_way()
        o.under_way()
        st["opt"].malt.set_scalars(nu, T0)
        st["opt"].adamw.set_step(T0)
        st["hp"] = malt.hparams(weight_decay=DECAY, **hp)
        st["adam_hp"] = malt.adamw_hparams(lr=case["lr"], betas=(BETA1, BETA2), eps=EPS)
        return st
    st["opt"] = malt.MaltOptimizer(x.views)
    st["opt"].set_scalars(x.under_way(), T0)
    st["hp"] = malt.hparams(**hp)
    if path == "host":
        gh, wh = torch.empty(x.g.shape, dtype=x.g.dtype, pin_memory=True), torch.empty(x.w.shape, dtype=x.w.dtype, pin_memory=True)
        gh.copy_(x.g)
        wh.zero_()
        x.g.zero_()
        st["w_host"], st["buffers"] = wh, (gh, wh)
        n, off = [a * b for a, b in x.shapes], 0
        st["gh"], st["wh"] = [], []
        for c, s in zip(n, x.shapes):
            st["gh"].append(gh[off:off + c].view(s))
            st["wh"].append(wh[off:off + c].view(s))
            off += -(-c // ALIGN) * ALIGN
    return st


def run(st):
    path = st["path"]
    if path == "adamw":
        st["opt"].step(st["hp"])
        o = st["others"]
        return {"w": o.w, "copy": o.c, "m": o.m, "v": o.v}
    x = st["mats"]
    if path == "stats":
        _, g, m, l, r = x.views[0]
        L, R = st["out"]
        if malt.malt_stats_noalloc(g, m, l, r, L, R, mu1=MU1, mu2=MU2, eps=EPS) != malt.MALT_OK:
            raise RuntimeError("malt_stats_noalloc failed")
        return {"m": x.m, "l": x.l, "r": x.r, "L": L, "R": R}
    if path == "whole":
        st["opt"].step(st["hp"], st["adam_hp"], malter=st["variant"] == "malter")
        o = st["others"]
        return {"w": x.w, "copies": st["copies"], "m": x.m, "l": x.l, "r": x.r,
                "other_w": o.w, "other_copy": o.c, "other_m": o.m, "other_v": o.v}
    if path == "host":
        st["opt"].step_host(st["hp"], st["gh"], st["wh"], malter=st["variant"] == "malter")
        return {"w_host": st["w_host"], "w": x.w, "m": x.m, "l": x.l, "r": x.r}
    st["opt"].step(st["hp"], malter=st["variant"] == "malter", muon=st["variant"] == "muon")
    return {"w": x.w, "m": x.m, "l": x.l, "r": x.r}


# ------------------------------------------------------------------- costs
def work(case):
    size = {"f32": 4.0, "bf16": 2.0}
    total, flops = 0.0, 0.0
    path = case["path"]
    if path in ("whole", "adamw"):
        total += 30.0 * sum(int(np.prod(s)) for s, _ in _adam_tensors(case))   # g; w, m, v in and out; copy
    if path != "adamw":
        for m, n in _shapes(case):
            total += m * n * (size[case["grads"]] + 8.0)                     # G; M in and out
            if case["variant"] != "muon":
                total += 8.0 * (m + n)                                       # l, r in and out
            if path == "stats":
                total += 4.0 * (m + n)                                       # L, R
                flops += 7.0 * m * n
                continue
            total += m * n * 2.0 * size[case["weights"]]                     # W in and out
            if path == "whole":
                total += 2.0 * m * n                                         # bf16 copy
            flops += _ns_flops(m, n, case["ns_steps"])
    else:
        flops += 15.0 * total / 30.0
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """fp32 streams (AdamW, the statistics) agree to a few ulps of fp32, or of bf16 where a
    bf16 copy of the weights is written.  A step moves W by lr * ||O|| (about lr sqrt(p)) out of
    0.02 sqrt(p q), and 16-bit Newton-Schulz operands leave about 1 % on the direction O (2.5 %
    at eight iterations and on thin matrices), which is what W may differ by; bf16 weights that
    round the other way differ by 2^-8 each."""
    path = case["path"]
    if path == "stats":
        return {"rel": 1e-6}
    if path == "adamw":
        return {"rel": 1e-4, "max": 1e-2}
    q = min(max(s) for s in _shapes(case))
    lr = case["lr"] * (0.25 if case["variant"] == "malter" else 1.0)     # alpha is about 0.16 here
    rel = 0.04 * lr * 50.0 / math.sqrt(q) + (2e-3 if case["weights"] == "bf16" or path == "whole" else 1e-5)
    return {"rel": min(0.03, rel), "max": min(0.9, 40.0 * rel)}


# ------------------------------------------------------------------- exact
def _newton_schulz(x, steps):
    a, b, c = (float(np.float32(v)) for v in NS_COEFFS)
    tall = x.shape[-2] > x.shape[-1]
    if tall:
        x = x.transpose(-1, -2)
    x = x / (torch.linalg.matrix_norm(x, keepdim=True) + float(np.float32(NS_EPS)))
    for _ in range(steps):
        A = x @ x.transpose(-1, -2)
        B = b * A + c * (A @ A)
        x = a * x + B @ x
    return x.transpose(-1, -2) if tall else x


def _exact_matrix(case, lr, decay, w, g, m, l, r, nu, direction):
    """One step of one matrix in fp64; W is None where the direction is not asked for."""
    f = lambda v: float(np.float32(v))  # noqa: E731  (the hyperparameters are passed as fp32)
    mu1, mu2, eps = f(MU1), f(MU2), f(EPS)
    variant = case["variant"]
    w, g, m, l, r = (v.double() for v in (w, g, m, l, r))
    m = mu1 * m + (1 - mu1) * g
    if variant != "muon":
        l = mu2 * l + (1 - mu2) * (g * g).sum(1)
        r = mu2 * r + (1 - mu2) * (g * g).sum(0)
        L, R = (l + eps) ** -0.125, (r + eps) ** -0.125
    else:
        L, R = torch.ones_like(l), torch.ones_like(r)
    if not direction:
        return None, m, l, r, L, R
    mt = L[:, None] * m * R[None, :]
    o = _newton_schulz(mt, case["ns_steps"])
    d = L[:, None] * o * R[None, :]
    s = lr * torch.linalg.matrix_norm(o) / (torch.linalg.matrix_norm(d) + eps)
    if variant == "malter":
        t = T0 + 1
        nu = mu2 * nu + (1 - mu2) * ((L[:, None] * g * R[None, :]) ** 2).sum()
        s = s * math.sqrt(1 - mu2 ** t) / (1 - mu1 ** t + eps) * torch.linalg.matrix_norm(mt) / (torch.sqrt(nu) + eps)
    return decay * w - s * d, m, l, r, L, R


def exact(case, seed):
    f = lambda v: float(np.float32(v))  # noqa: E731
    path, lr = case["path"], f(case["lr"])
    out = {}
    if path in ("adamw", "whole"):
        o = _Others(case, seed)
        o.under_way()
        t, b1, b2 = T0 + 1, f(BETA1), f(BETA2)
        m = b1 * o.m.double() + (1 - b1) * o.g.double()
        v = b2 * o.v.double() + (1 - b2) * o.g.double() ** 2
        decay, dv = _flat([int(np.prod(s)) for s, _ in o.spec], torch.float64)
        for d, (_, wd) in zip(dv, o.spec):
            d.fill_(1.0 - lr * f(wd))
        w = decay * o.w.double() - lr * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + f(EPS))
        if path == "adamw":
            # gaps between the tensors are not part of any of them
            mask = _gaps(o)
            return {"w": torch.where(mask, w, o.w.double()), "copy": torch.where(mask, w, 0.0),
                    "m": torch.where(mask, m, o.m.double()), "v": torch.where(mask, v, o.v.double())}
        mask = _gaps(o)
        out = {"other_w": torch.where(mask, w, o.w.double()), "other_copy": torch.where(mask, w, 0.0),
               "other_m": torch.where(mask, m, o.m.double()), "other_v": torch.where(mask, v, o.v.double())}
    x = _Matrices(case, seed)
    nu = x.under_way()
    # fp64 runs at about 1 TFLOP/s here: the direction (and with it W) where it takes seconds
    direction = path != "stats" and 4.0 / 3.0 * sum(_ns_flops(m, n, case["ns_steps"]) for m, n in x.shapes) < 1.2e13
    W, _ = _flat([a * b for a, b in x.shapes], torch.float64)
    M, L, R = torch.zeros_like(x.m, dtype=torch.float64), torch.zeros_like(x.l, dtype=torch.float64), torch.zeros_like(x.r, dtype=torch.float64)
    PL, PR = torch.zeros_like(L), torch.zeros_like(R)
    decay = 1.0 - lr * f(DECAY) if path == "whole" else 1.0
    am = al = ar = 0
    up = lambda c: -(-c // ALIGN) * ALIGN  # noqa: E731
    for i, ((a, b), v) in enumerate(zip(x.shapes, x.views)):
        w, m, l, r, pl, pr = _exact_matrix(case, lr, decay, *v, float(nu[i]), direction)
        if w is not None:
            W[am:am + a * b] = w.reshape(-1)
        M[am:am + a * b] = m.reshape(-1)
        L[al:al + a], R[ar:ar + b] = l, r
        PL[al:al + a], PR[ar:ar + b] = pl, pr
        am, al, ar = am + up(a * b), al + up(a), ar + up(b)
    if path == "stats":
        return {"m": M, "l": L, "r": R, "L": PL[:x.shapes[0][0]], "R": PR[:x.shapes[0][1]]}
    out.update({"w": W if direction else None, "m": M, "l": L, "r": R})
    if path == "whole":
        out["copies"] = W
    if path == "host":
        out["w_host"] = W
    return out


def _gaps(o):
    """True where a flat buffer of the AdamW tensors holds an element of one."""
    mask, views = _flat([int(np.prod(s)) for s, _ in o.spec], torch.bool)
    for v in views:
        v.fill_(True)
    return mask
