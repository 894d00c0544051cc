"""The work that programs have this library do, as measurable cases.

Every case goes through a public entry point of the Python binding: a step of
the optimizer (``LionMuon.step``, or a replay of ``capture_steps``) over a
parameter set, or one msign call.  The sets and sizes are those of the
repository's benchmark and tests, or generic ones of the same kind.

``listed()`` and ``draw(rng)`` give cases, ``prepare`` makes what a program has
in hand before the call (parameters, gradients, the optimizer in mid-training),
``run`` is one pass, ``exact`` the same in plain 64-bit torch, ``work`` the bytes
and operations no implementation can do without.
"""

from __future__ import annotations

import math

import torch

ETA_MUON, ETA_LION, DECAY = 3e-3, 2e-5, 0.1
BETA1, BETA2 = 0.9, 0.99
SHAPE_SCALE, NS_STEPS, NS_EPS = 0.2, 5, 1e-7
QUINTIC = (3.4445, -4.7750, 2.0315)
# The degree-5 minimax table for singular values from 1e-3 (ns_coeffs.polar_express), to four decimals.
TABLE = ((8.4703, -25.1081, 18.6293), (4.1828, -3.1087, 0.5806), (3.9619, -2.9541, 0.5630),
         (3.2866, -2.4647, 0.5074), (2.2737, -1.6447, 0.4162))
ADAM_LR, ADAM_B1, ADAM_B2, ADAM_EPS = 1e-3, 0.8, 0.999, 1e-8
T0 = 1000            # the step index the optimizer is at: mid-training, a multiple of every period used
EXACT_FLOPS = 9e12   # 64-bit reference runs above this many operations are left out (about 20 s)


# ------------------------------- the cases ---------------------------------
def listed():
    return [
        # The smallest training set of the benchmark plan, all fp32 (parameters,
        # Newton-Schulz on fp32): a step is a few launches over 0.8 M elements.
        _step("tiny_f32_muon", set="tiny", dtype="f32", precision="f32", phase="muon", grads="normal"),
        # A small bf16 language model, as the tests train it for 8 steps: launch-bound.
        _step("small_muon", set="gpt", layers=2, d=128, vocab=1000, phase="muon"),
        # One transformer layer replayed from a CUDA graph, as a latency-critical
        # training loop runs its optimizer: Muon step, no host work.
        _step("layer_graph_muon", set="layers", layers=1, d=768, phase="muon", graph=True),
        # Ragged model: widths and vocabulary that are no multiple of 8, AdamW on
        # the vectors, a per-iteration coefficient table.
        _step("ragged_adamw_table", set="gpt", layers=3, d=300, vocab=5003, phase="muon", vectors="adamw", table=True),
        # GPT-2-124M-shaped set, the ordinary size: each kind of step by itself.
        _step("gpt2_124m_muon", set="gpt", layers=12, d=768, vocab=50304, phase="muon"),
        _step("gpt2_124m_lion", set="gpt", layers=12, d=768, vocab=50304, phase="lion"),
        # 355M-shaped set under the adaptive schedule: power iteration on every
        # momentum buffer, Muon where its stable rank is low, Lion elsewhere.
        _step("gpt_355m_srank", set="gpt", layers=24, d=1024, vocab=50304, phase="srank"),
        # The benchmark's set: one period (a Muon and a Lion step) of 772 M parameters.
        _step("gpt_720m_period", set="gpt", layers=36, d=1280, vocab=50304, phase="period"),
        # fp32 parameters with the fast fp32 Newton-Schulz on the tensor cores.
        _step("layers_f32tc_muon", set="layers", layers=4, d=1280, dtype="f32", precision="f32tc", phase="muon"),
        # msign by itself: a hidden matrix in bf16, the call that allocates nothing
        # on an ordinary MLP matrix, and full fp32 on a square one.
        _msign("msign_bf16", rows=1280, cols=5120),
        _msign("msign_noalloc_bf16", rows=3072, cols=768, noalloc=True),
        _msign("msign_f32", rows=1024, cols=1024, dtype="f32", precision="f32"),
    ]


def _step(name=None, *, set, layers=0, d=0, vocab=0, dtype="bf16", precision="bf16", phase="muon", vectors="lion",
          table=False, graph=False, grads="student_t"):
    case = {"kind": "step", "set": set, "layers": layers, "d": d, "vocab": vocab, "dtype": dtype,
            "precision": precision, "phase": phase, "vectors": vectors, "table": table, "graph": graph, "grads": grads}
    return dict(case, name=name) if name else case


def _msign(name=None, *, rows, cols, dtype="bf16", precision="bf16", noalloc=False, table=False):
    case = {"kind": "msign", "rows": rows, "cols": cols, "dtype": dtype, "precision": precision,
            "noalloc": noalloc, "table": table}
    return dict(case, name=name) if name else case


def draw(rng):
    """One more case: steps over sets from a few thousand to about 150 M
    parameters in every precision and phase, and msign of matrices from a few
    rows to the embedding's shape."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def size(lo, hi):                      # widths: mostly multiples of 64 or 8, some odd
        x = log(lo, hi)
        q = rng.choice((64, 64, 8, 1))
        return max(lo, x // q * q)

    if rng.random() < 0.35:                # msign
        precision = rng.choice(("bf16", "bf16", "f32", "f32tc"))
        noalloc = precision != "f32tc" and rng.random() < 0.4
        a, b = size(8, 2048), size(8, 2048)
        if rng.random() < 0.5:             # long matrices, up to the embedding's shape
            b = size(a, 5120 if noalloc or precision == "f32" else 50304)
        if noalloc:                        # what fits its fixed 64 MiB workspace
            a, b = min(a, 1024), min(b, 4096)
        if rng.random() < 0.5:
            a, b = b, a
        dtype = rng.choice(("bf16", "f32")) if precision == "bf16" else "f32"
        return _msign(rows=a, cols=b, dtype=dtype, precision=precision, noalloc=noalloc,
                      table=not noalloc and rng.random() < 0.25)
    precision = rng.choice(("bf16", "bf16", "bf16", "f32", "f32tc"))
    phase = rng.choice(("muon", "muon", "muon", "lion", "period", "srank"))
    embed = rng.random() < 0.5
    d = size(32, 1024 if precision == "bf16" else 768)
    if phase == "srank":
        d = max(64, d)
    if embed:                              # flat parameter and momentum buffers: widths of whole 64s
        d = max(64, d // 64 * 64)
    most = 150e6 if precision == "bf16" else 50e6
    vocab = log(256, 50304) // 64 * 64 if embed else 0
    layers = min(log(1, 16), max(1, int((most - vocab * d) / (12 * d * d)))) if embed else log(1, 4)
    vectors = "adamw" if embed and rng.random() < 0.3 else "lion"
    graph = vectors == "lion" and phase == "muon" and rng.random() < 0.25
    return _step(set="gpt" if embed else "layers", layers=layers, d=d, vocab=vocab,
                 dtype=rng.choice(("bf16", "bf16", "f32")) if precision == "bf16" else "f32", precision=precision,
                 phase=phase, vectors=vectors, table=phase != "srank" and rng.random() < 0.25, graph=graph,
                 grads=rng.choice(("student_t", "normal")))


# ------------------------------- the inputs --------------------------------
def _shapes(case):
    if case["kind"] == "msign":
        return [(case["rows"], case["cols"])]
    if case["set"] == "tiny":
        return [(256, 256), (256, 1024), (1024, 256), (256, 256), (256,)]
    d, out = case["d"], []
    full = case["set"] == "gpt"
    if full:
        out.append((case["vocab"], d))
    for _ in range(case["layers"]):
        out += ([(d,), (d,)] if full else []) + [(d, 3 * d), (d, d)] + ([(d,), (d,)] if full else [])
        out += [(d, 4 * d), (4 * d, d)]
    return out + ([(d,), (d,)] if full else [])


def _numel(shape):
    return math.prod(shape)


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _views(flat, shapes):
    """The tensors of ``shapes`` in one flat buffer, each on a 64-element boundary."""
    out, at = [], 0
    for s in shapes:
        out.append(flat[at:at + _numel(s)].view(s))
        at += (_numel(s) + 63) // 64 * 64
    return out


def _flat_size(shapes):
    return sum((_numel(s) + 63) // 64 * 64 for s in shapes)


def _alpha(case):
    """Threshold of the adaptive schedule: its default 0.01, more for matrices so small that it would select none."""
    return max(0.01, 6.0 / case["d"])


def _noise(gen, n, kind):
    """n gradient entries: N(0, 1), or Student-t with nu = 3 scaled to a standard deviation of 1e-3."""
    z = torch.randn(n, generator=gen, device="cuda")
    if kind == "normal":
        return z
    chi = torch.zeros(n, device="cuda")
    for _ in range(3):
        e = torch.randn(n, generator=gen, device="cuda")
        chi.addcmul_(e, e)
    return z.mul_(torch.rsqrt(chi.div_(3.0))).mul_(1e-3 / 3.0 ** 0.5)


def _inputs(case, seed):
    """(W, G, M): flat buffers of the parameters, gradients and momentum (fp32)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    shapes = _shapes(case)
    n = _flat_size(shapes)
    W = (torch.randn(n, generator=gen, device="cuda") * 0.02).to(_dtype(case))
    G = _noise(gen, n, case["grads"])
    # momentum: an average of many gradients, a tenth of one in size, sharing
    # a part of the present one
    M = torch.randn(n, generator=gen, device="cuda").mul_(0.1 * (1.0 if case["grads"] == "normal" else 1e-3))
    M.add_(G, alpha=0.02)
    if case["phase"] == "srank":
        # Every third matrix has a dominant direction in its gradients and its
        # momentum (stable rank about 4), so both branches run; the others are
        # noise, far from the threshold on the other side.
        for k, (g, m) in enumerate(zip(_views(G, shapes), _views(M, shapes))):
            if g.dim() != 2:
                continue
            u = torch.nn.functional.normalize(torch.randn(g.shape[0], generator=gen, device="cuda"), dim=0)
            v = torch.nn.functional.normalize(torch.randn(g.shape[1], generator=gen, device="cuda"), dim=0)
            if k % 3 == 0:
                m.addr_(u, v, alpha=0.57 * float(m.norm()))
                g.addr_(u, v, alpha=0.57 * float(g.norm()))
    # the gaps between tensors hold nothing
    for flat in (W, G, M):
        at = 0
        for s in shapes:
            end = at + _numel(s)
            at += (_numel(s) + 63) // 64 * 64
            flat[end:at] = 0
    return W, G.to(_dtype(case)), M


def _msign_input(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.randn(case["rows"], case["cols"], generator=gen, device="cuda") * 1e-3
    return x.to(_dtype(case))


class _Buffer:
    """A stretch of the optimizer's memory as an array that torch can view;
    the view keeps the optimizer, and so the memory, alive."""

    def __init__(self, opt, ptr, n):
        self.owner = opt
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<f4", "data": (ptr, False), "version": 3,
                                         "strides": None}


def _momentum_views(opt, shapes):
    """Views of the optimizer's momentum buffers, as few as cover them:
    buffers that follow one another without a gap are one view."""
    runs = []
    for i, s in enumerate(shapes):
        ptr, n = opt.momentum(i).data_ptr(), _numel(s)
        if runs and runs[-1][0] + 4 * runs[-1][1] == ptr:
            runs[-1][1] += n
        else:
            runs.append([ptr, n])
    return [torch.as_tensor(_Buffer(opt, p, n), device="cuda") for p, n in runs]


def prepare(case, seed):
    from paper_2605_19811_gb300 import lionmuon as L
    precision = {"bf16": L.LM_BF16, "f32": L.LM_F32, "f32tc": L.LM_NS_F32_TC}[case["precision"]]
    if case["kind"] == "msign":
        x = _msign_input(case, seed)
        return {"case": case, "x": x, "out": torch.empty_like(x), "precision": precision}
    shapes = _shapes(case)
    W, G, M = _inputs(case, seed)
    params, grads, momentum = _views(W, shapes), _views(G, shapes), _views(M, shapes)
    cfg = dict(eta_muon=ETA_MUON, eta_lion=ETA_LION, weight_decay=DECAY, beta1=BETA1, beta2=BETA2, period=2,
               ns_precision=precision)
    if case["table"]:
        cfg["ns_coeffs"] = TABLE
    if case["vectors"] == "adamw":
        cfg.update(vector_rule=L.LM_VECTOR_ADAMW, adamw_lr=ADAM_LR, adamw_beta1=ADAM_B1, adamw_beta2=ADAM_B2,
                   adamw_eps=ADAM_EPS, adamw_weight_decay=DECAY)
    if case["phase"] == "srank":
        cfg.update(schedule=L.LM_SCHEDULE_STABLE_RANK, srank_alpha=_alpha(case))
    opt = L.LionMuon(params, **cfg)
    for i, m in enumerate(momentum):
        opt.set_momentum(i, m)
        if case["vectors"] == "adamw" and m.dim() == 1:
            opt.set_second_moment(i, (m * m).mul_(0.5).add_(1e-8))
    state = {"case": case, "opt": opt, "grads": grads, "t": T0, "W": W,
             "out": [W] + _momentum_views(opt, shapes)}
    if case["vectors"] == "adamw":
        vectors = [i for i, s in enumerate(shapes) if len(s) == 1]
        if len(vectors) <= 30:
            state["out"] += [torch.as_tensor(_Buffer(opt, opt.second_moment(i).data_ptr(), _numel(shapes[i])),
                                             device="cuda") for i in vectors]
    if case["graph"]:
        state["graphs"] = opt.capture_steps(grads)
    torch.cuda.synchronize()
    return state


# --------------------------------- one pass --------------------------------
def run(state):
    case = state["case"]
    if case["kind"] == "msign":
        from paper_2605_19811_gb300 import lionmuon as L
        if case["table"]:
            return L.msign_ns_coeffs(state["x"], state["out"], TABLE, precision=state["precision"])
        call = L.msign_ns_noalloc if case["noalloc"] else L.msign_ns
        return call(state["x"], state["out"], steps=NS_STEPS, precision=state["precision"])
    t, phase = state["t"], case["phase"]
    state["t"] = t + 2
    if case["graph"]:
        state["graphs"][0].replay()
    elif phase == "lion":
        state["opt"].step(state["grads"], t + 1)
    else:
        state["opt"].step(state["grads"], t)
        if phase == "period":
            state["opt"].step(state["grads"], t + 1)
    return state["out"]


# ------------------------------- the reference -----------------------------
def _ns64(x, coeffs):
    """The odd-polynomial msign iteration on the wide orientation, fp64."""
    tall = x.shape[0] > x.shape[1]
    x = x.t().contiguous() if tall else x
    x = x / (x.norm() + NS_EPS)
    for a, b, c in coeffs:
        A = x @ x.t()
        x = a * x + (b * A + c * (A @ A)) @ x
    return x.t() if tall else x


def _coeffs(case):
    return TABLE if case["table"] else (QUINTIC,) * NS_STEPS


def exact(case, seed):
    if work(case)["flops"] > EXACT_FLOPS:
        return None
    if case["kind"] == "msign":
        return _ns64(_msign_input(case, seed).double(), _coeffs(case))
    shapes = _shapes(case)
    W, G, M = (x.double() for x in _inputs(case, seed))
    phases = {"muon": ("muon",), "lion": ("lion",), "srank": ("srank",), "period": ("muon", "lion")}[case["phase"]]
    V = {}
    for k, phase in enumerate(phases):
        t = T0 + (1 if case["phase"] == "lion" else k)
        for i, (w, g, m) in enumerate(zip(_views(W, shapes), _views(G, shapes), _views(M, shapes))):
            if w.dim() == 1 and case["vectors"] == "adamw":
                v = V.setdefault(i, (m.float() * m.float()).mul_(0.5).add_(1e-8).double())
                m.mul_(ADAM_B1).add_(g, alpha=1 - ADAM_B1)
                v.mul_(ADAM_B2).addcmul_(g, g, value=1 - ADAM_B2)
                w.mul_(1 - ADAM_LR * DECAY)
                den = (v.sqrt() / math.sqrt(1 - ADAM_B2 ** (t + 1))).add_(ADAM_EPS)
                w.addcdiv_(m, den, value=-ADAM_LR / (1 - ADAM_B1 ** (t + 1)))
                continue
            gh = BETA1 * m + (1 - BETA1) * g
            muon = phase == "muon" and w.dim() == 2
            if phase == "srank" and w.dim() == 2:
                small = m @ m.t() if m.shape[0] <= m.shape[1] else m.t() @ m
                muon = _low_rank(small, _alpha(case) * min(m.shape))
            if muon:
                o = _ns64(gh, _coeffs(case)) * (SHAPE_SCALE * math.sqrt(max(w.shape)))
                w.sub_(ETA_MUON * (o + DECAY * w))
            else:
                w.sub_(ETA_LION * (gh.sign() + DECAY * w))
            m.mul_(BETA2).add_(g, alpha=1 - BETA2)
    # laid out as run() returns it: W, the momentum buffers, the second moments
    runs = []
    for m in _views(M, shapes):
        if runs and runs[-1][1]:
            runs[-1][0].append(m.reshape(-1))
        else:
            runs.append([[m.reshape(-1)], True])
        runs[-1][1] = m.numel() % 64 == 0
    out = [W] + [torch.cat(parts) for parts, _ in runs]
    vectors = [i for i, s in enumerate(shapes) if len(s) == 1]
    if case["vectors"] == "adamw" and len(vectors) <= 30:
        out += [V[i] for i in vectors]
    return out


def _low_rank(gram, most):
    """Whether the stable rank of the buffer with this Gram matrix is at most
    ``most`` (every buffer made here is far from it on one side)."""
    v = torch.ones(gram.shape[0], device=gram.device, dtype=gram.dtype)
    for _ in range(20):
        v = gram @ v
        v = v / v.norm()
    return float(gram.trace()) <= most * float(v @ (gram @ v))


# ---------------------------- work and tolerance ---------------------------
def work(case):
    """Bytes: parameters and momentum read and written, gradients read (msign:
    input read, output written).  Operations: Newton-Schulz with its symmetric
    products counted once, 3 s^2 l + s^3 per iteration."""
    e = 4 if case["dtype"] == "f32" else 2
    shapes = _shapes(case)
    ns = 0.0
    for shape in shapes:
        if len(shape) == 2:
            s, l = min(shape), max(shape)
            ns += NS_STEPS * (3.0 * s * s * l + float(s) ** 3)
    n = float(sum(_numel(s) for s in shapes))
    if case["kind"] == "msign":
        return {"bytes": 2.0 * e * n, "flops": ns}
    step = n * (3 * e + 8)
    if case["phase"] == "lion":
        return {"bytes": step, "flops": 8.0 * n}
    if case["phase"] == "period":
        return {"bytes": 2 * step, "flops": ns + 16.0 * n}
    if case["phase"] == "srank":     # 5 products with M and 4 with its transpose; a third of the matrices take Muon
        matrices = [x for x in enumerate(shapes) if len(x[1]) == 2]
        share = sum(_numel(x) for k, x in matrices if k % 3 == 0) / max(1.0, sum(_numel(x) for _, x in matrices))
        return {"bytes": step, "flops": 18.0 * n + share * ns}
    return {"bytes": step, "flops": ns + 8.0 * n}


def tolerance(case):
    """Relative error another implementation at the same precision would show,
    about four times what the path shows against exact()."""
    if case["kind"] == "msign":
        if case["precision"] == "bf16":
            return {"rel": 0.03, "max": 0.5}
        if case["dtype"] == "bf16":
            return {"rel": 8e-3, "max": 0.1}
        return {"rel": 4e-5 if case["precision"] == "f32" else 8e-5, "max": 2e-3}
    if case["dtype"] == "bf16":         # the parameter's own rounding is 1.7e-3
        return {"rel": 2e-4, "max": 0.02} if case["phase"] == "lion" else {"rel": 7e-3, "max": 0.1}
    if case["phase"] == "lion":
        return {"rel": 1e-6, "max": 1e-4}
    if case["precision"] == "bf16":     # fp32 parameters, bf16 Newton-Schulz: 1 % of an update that is 3 % of W
        return {"rel": 2e-3, "max": 0.1}
    return {"rel": 1e-6, "max": 1e-4}
