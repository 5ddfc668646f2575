"""The calls whose speed and results a change to the kernels is judged by.

A case is one thing that a training program asks of the library for M worker
replicas of a flattened tensor list:

  step   one local step of every worker, from gradients on the device
         (``clip``: with the per-worker global-norm clip of Algorithms 1 and 3)
  fused  the same step where averages fall due at its end (``mask``: which
         states, bit 0 = x, then u_1.., then v)
  run    a communication round of ``count`` steps in one call, every state
         averaged by the last one
  sync   the averages alone
  diag   the end of a round with the paper's section 4.1 diagnostics: the
         change of x since the last average, then the average of the masked
         states with its cross-worker variance, norms and cosines

Sizes: the tensor lists of the synthetic workloads (a GPT-2-small-shaped list,
a ~350M decoder list, the flat 2^20 vector), the 256-worker toy problem, the
sizes of the tests' ragged lists, and flat vectors in between.  States are
those of a run under way: workers apart by a small part of x, momenta and
second moments of the gradients' scale, t = 1024.
"""
import math
import random

import torch

import paper_2510_05361_gb300 as mt

BETAS = (0.9, 0.999, 0.5, 0.99)
T0 = 1024                # steps already taken
LR = 1e-3
SIGMA = 1e-3             # gradient scale (the decoder workloads' N(0, 1e-3))
PRECISE = torch.float64


def listed():
    small_gpt = {"vocab": 50257, "d": 768, "ffn": 3072, "blocks": 12}
    decoder = {"vocab": 50257, "d": 1024, "ffn": 4096, "blocks": 24}
    return [
        # a model of a few thousand parameters (an MLP head, a unit test): launch and call latency
        {"name": "step-5k-m4", "kind": "step", "base": "adam", "n_mom": 2, "M": 4, "grad": "f32",
         "numel": 5436, "tensors": 4, "clip": False},
        # noisy Rosenbrock with 256 workers and 256 independent problems, at the end of a period
        {"name": "fused-toy-m256", "kind": "fused", "base": "adam", "n_mom": 1, "M": 256, "grad": "f32",
         "numel": 512, "tensors": 1, "mask": 0b111},
        # the flat 2^20 workload: one round of 16 steps
        {"name": "run-1m-m4", "kind": "run", "base": "adam", "n_mom": 2, "M": 4, "grad": "f32",
         "numel": 1 << 20, "tensors": 1, "count": 16},
        # an ordinary model: the step taken 31 times out of 32 ...
        {"name": "step-gpt2-m4", "kind": "step", "base": "adam", "n_mom": 3, "M": 4, "grad": "f32",
         "clip": False, **small_gpt},
        # ... and the 32nd
        {"name": "fused-gpt2-m4", "kind": "fused", "base": "adam", "n_mom": 3, "M": 4, "grad": "f32",
         "mask": 0b11111, **small_gpt},
        # the same list trained with clipping at rho = 1 and bf16 gradients
        {"name": "clip-gpt2-m4-bf16", "kind": "step", "base": "adam", "n_mom": 2, "M": 4, "grad": "bf16",
         "clip": True, **small_gpt},
        # the largest: ~350M parameters, 8 workers, ADOPT, bf16 gradients, momenta and v due (K = 16)
        {"name": "fused-350m-m8-adopt", "kind": "fused", "base": "adopt", "n_mom": 2, "M": 8, "grad": "bf16",
         "mask": 0b1110, **decoder},
        # more workers than a thread can hold: 16 on 2^23 parameters, 64 on an odd size
        {"name": "fused-8m-m16", "kind": "fused", "base": "adam", "n_mom": 3, "M": 16, "grad": "f32",
         "numel": 1 << 23, "tensors": 1, "mask": 0b11111},
        {"name": "fused-1.9m-m64-sgdm", "kind": "fused", "base": "sgdm", "n_mom": 1, "M": 64, "grad": "bf16",
         "numel": 1900543, "tensors": 7, "mask": 0b11},
        # an average on demand: 32 workers of a ragged 5M-parameter list
        {"name": "sync-5m-m32", "kind": "sync", "base": "adopt", "n_mom": 1, "M": 32, "grad": "f32",
         "numel": 5000011, "tensors": 9, "mask": 0b111},
        # a round's end with diagnostics: the ordinary model, and many workers on a small one
        {"name": "diag-gpt2-m4", "kind": "diag", "base": "adam", "n_mom": 2, "M": 4, "grad": "f32",
         "mask": 0b1111, **small_gpt},
        {"name": "diag-75k-m100", "kind": "diag", "base": "sgdm", "n_mom": 1, "M": 100, "grad": "f32",
         "numel": 75096, "tensors": 3, "mask": 0b11},
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "fused", "fused", "fused", "run", "sync", "diag"])
    base = rng.choice(["adam", "adopt", "sgdm"])
    n_mom = rng.choice([1, 2, 2, 3, 4])
    most_m = {"step": 32, "run": 16}.get(kind, 256)
    M = int(round(2 ** rng.uniform(0.0 if kind == "step" else 1.0, math.log2(most_m))))
    per_elem = 8 * _n_states(base, n_mom) + 4
    count = rng.randrange(8, 33) if kind == "run" else 1
    # 10^3.5 to 10^9.5 bytes of state over all workers, run's gradients within 4 GB
    total = 10 ** rng.uniform(3.5, 9.5) / per_elem * 8
    total = min(total, 1e9 / count)
    numel = max(2, int(total / M))
    if rng.random() < 0.5:
        numel |= 1
    case = {"kind": kind, "base": base, "n_mom": n_mom, "M": M, "grad": rng.choice(["f32", "bf16"]),
            "numel": numel, "tensors": rng.randrange(1, 13) if numel > 64 else 1}
    if kind == "step":
        case["clip"] = base != "adopt" and rng.random() < 0.5
    elif kind == "run":
        case["count"] = count
    else:
        states = _n_states(base, n_mom)
        every = (1 << states) - 1
        case["mask"] = rng.choice([1, every, every, rng.randrange(1, every + 1)])
    return case


# ------------------------------------------------------------------ inputs

def _n_states(base, n_mom):
    return 1 + n_mom + (0 if base == "sgdm" else 1)


def _numels(case):
    """The case's tensor list: a decoder's (embedding, then per block qkv, proj,
    fc1, fc2 and four norm vectors, then the final norm), or ``numel`` elements
    cut into ``tensors`` uneven pieces."""
    if "blocks" in case:
        d, ffn = case["d"], case["ffn"]
        block = [3 * d * d, d * d, d * ffn, ffn * d, d, d, d, d]
        return [case["vocab"] * d] + block * case["blocks"] + [d, d]
    rng = random.Random(case["numel"])
    cuts = sorted(rng.sample(range(1, case["numel"]), case["tensors"] - 1)) if case["tensors"] > 1 else []
    edges = [0] + cuts + [case["numel"]]
    return [b - a for a, b in zip(edges, edges[1:])]


def _opt(case):
    n = case["n_mom"]
    adam = case["base"] == "adam"
    period = case.get("count", 32)
    return {"base": case["base"], "n_mom": n, "beta1": list(BETAS[:n]), "omega": [0.95 / n] * n,
            "beta2": 0.9999 if case["base"] == "adopt" else 0.999, "eps": 1e-8, "bias_correction": adam,
            "clip_mode": "global_norm" if case.get("clip") else "none", "clip_rho": 1.0,
            "period_x": period, "period_u": [period] * n,
            "period_v": 0 if case["base"] == "sgdm" else period, "sync_phase": "alg1"}


def _layout(case):
    """(offset and numel of each tensor, padded length) of the flattened list."""
    numels = _numels(case)
    offsets, n_padded = mt.mtdao_plan_layout(numels)
    return list(zip(offsets, numels)), n_padded


def _zero_padding(t, tensors):
    end = 0
    for off, k in tensors:
        if off > end:
            t[..., end:off].zero_()
        end = off + k
    if t.shape[-1] > end:
        t[..., end:].zero_()


def _gradients(case, tensors, n, gen):
    """[count][M][n]: N(0, SIGMA), one position in a hundred 100 times larger."""
    shape = (case.get("count", 1), case["M"], n)
    g = torch.empty(shape, device="cuda", dtype=torch.bfloat16 if case["grad"] == "bf16" else torch.float32)
    far = torch.rand((n,), device="cuda", generator=gen) < 0.01
    outlier = torch.where(far, 100.0, 1.0).to(g.dtype)
    for row in g.view(-1, n):
        row.normal_(0.0, SIGMA, generator=gen).mul_(outlier)
    _zero_padding(g, tensors)
    return g


def _states(case, states, x0, tensors, gen):
    """Fills the state vectors [M][n] of a run under way; x0: the last average."""
    n_mom = case["n_mom"]
    states[0].normal_(0.0, 1e-3, generator=gen).add_(x0)
    for u in states[1:1 + n_mom]:
        # ADOPT's momenta follow the normalised gradient, the others' the gradient
        u.normal_(0.0, 0.3 if case["base"] == "adopt" else 0.3 * SIGMA, generator=gen)
    for v in states[1 + n_mom:]:
        v.uniform_(0.25 * SIGMA ** 2, 2.0 * SIGMA ** 2, generator=gen)
    for s in states:
        _zero_padding(s, tensors)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _start(tensors, n, gen):
    x0 = torch.empty((n,), device="cuda").normal_(0.0, 0.02, generator=gen)
    _zero_padding(x0, tensors)
    return x0


def prepare(case, seed):
    gen = _generator(seed)
    tensors, n = _layout(case)
    eng = mt.MTDAO(_opt(case), case["M"], _numels(case))
    x0 = _start(tensors, n, gen)
    eng.set_params(x0)
    if case["kind"] == "diag":
        eng.track_anchor(1)
    states = [eng.state_view(s) for s in range(eng.n_states)]
    for view in states:
        view.engine = eng            # the views are the engine's memory: who holds one holds the engine
    _states(case, states, x0, tensors, gen)
    eng.t = T0 // case["count"] * case["count"] if case["kind"] == "run" else T0
    state = {"kind": case["kind"], "engine": eng, "states": states, "mask": case.get("mask", 0)}
    if case["kind"] in ("step", "fused", "run"):
        g = _gradients(case, tensors, n, gen)
        state["grads"] = g if case["kind"] == "run" else g[0]
        state["lrs"] = [LR] * case.get("count", 1)
    return state


def run(state):
    eng, kind = state["engine"], state["kind"]
    if kind == "run":
        eng.run(state["grads"], state["lrs"])
    elif kind == "sync":
        eng.sync(state["mask"])
    elif kind == "diag":
        change = eng.pseudo_grad_stats(0)
        stats = eng.sync_stats(state["mask"])
        return {"change": change, "stats": stats, "states": state["states"]}
    else:
        eng.step(state["grads"], LR, state["mask"])
    return {"states": state["states"]}


# ------------------------------------------------------------------ what is asked of a pass

def work(case):
    """Every state read and written once, every gradient read once (a step that
    clips needs the norm first, but not a second copy of the gradient)."""
    elems = case["M"] * sum(_numels(case))
    grad = 2 if case["grad"] == "bf16" else 4
    kind = case["kind"]
    if kind in ("step", "fused", "run"):
        count = case.get("count", 1)
        per_step = 6 * case["n_mom"] + (10 if case["base"] != "sgdm" else 3)
        return {"bytes": elems * (8 * _n_states(case["base"], case["n_mom"]) + grad * count),
                "flops": elems * per_step * count}
    k = bin(case["mask"]).count("1")
    if kind == "sync":
        return {"bytes": elems * 8 * k, "flops": elems * 4 * k}
    anchor = 8 * sum(_numels(case)) if case["mask"] & 1 else 4 * sum(_numels(case))
    read_x = 0 if case["mask"] & 1 else 4 * elems
    return {"bytes": elems * 8 * k + read_x + anchor, "flops": elems * (12 * k + 8)}


def tolerance(case):
    """States are fp32.  A step's few roundings leave about 5e-8 of a state's
    size, a round of steps their random walk (2e-7 seen); an average of
    replicas that cancel loses more of the (smaller) mean, 4e-7 seen for 100
    workers' independent momenta."""
    return {"rel": 2e-6, "max": 5e-5}


# ------------------------------------------------------------------ the same in 64 bits

def _update(case, opt, t, g, scale, s):
    """One local step (Algorithms 1-3) of the states s (64 bits), in place."""
    n, base = case["n_mom"], case["base"]
    x, v = s[0], s[-1]
    if base != "sgdm":
        v.mul_(opt["beta2"]).add_((1.0 - opt["beta2"]) * g * g)
    target = g * scale if scale is not None else g
    if base == "adopt":
        target = g / (v.sqrt() + opt["eps"])
    delta = (1.0 - sum(opt["omega"])) * target
    for j in range(n):
        beta = opt["beta1"][j]
        s[1 + j].mul_(beta).add_((1.0 - beta) * target)
        b = 1.0 - beta ** (t + 1) if opt["bias_correction"] else 1.0
        delta = delta + opt["omega"][j] / b * s[1 + j]
    if base == "adam":
        b = 1.0 - opt["beta2"] ** (t + 1) if opt["bias_correction"] else 1.0
        delta = delta / ((v / b).sqrt() + opt["eps"])
    x.sub_(LR * delta)


def exact(case, seed):
    gen = _generator(seed)
    tensors, n = _layout(case)
    opt, M, kind = _opt(case), case["M"], case["kind"]
    x0 = _start(tensors, n, gen)
    start = [torch.empty((M, n), device="cuda") for _ in range(_n_states(case["base"], case["n_mom"]))]
    _states(case, start, x0, tensors, gen)
    every = (1 << len(start)) - 1
    mask = case.get("mask", 0)
    out = [torch.empty((M, n), dtype=PRECISE, device="cuda") for _ in start]
    cols = max(1, (1 << 25) // M)
    pieces = [slice(i, min(n, i + cols)) for i in range(0, n, cols)]
    if kind in ("step", "fused", "run"):
        grads = _gradients(case, tensors, n, gen)
        scale = None
        if case.get("clip"):
            sq = sum(grads[0][:, p].to(PRECISE).square().sum(1, keepdim=True) for p in pieces)
            scale = torch.clamp(1.0 / (sq.sqrt() + 1e-6), max=1.0)
        t0 = T0 // case["count"] * case["count"] if kind == "run" else T0
        for p in pieces:
            s = [a[:, p].to(PRECISE) for a in start]
            for k in range(grads.shape[0]):
                _update(case, opt, t0 + k, grads[k][:, p].to(PRECISE), scale, s)
            due = every if kind == "run" else mask
            for i, a in enumerate(s):
                out[i][:, p] = a.mean(0, keepdim=True) if (due >> i) & 1 else a
        return {"states": out}

    change = torch.zeros((2 * M + 2,), dtype=PRECISE, device="cuda")
    rows = {i: torch.zeros((2 + 2 * M,), dtype=PRECISE, device="cuda")
            for i in range(len(start)) if (mask >> i) & 1}
    for p in pieces:
        for i, a in enumerate(start):
            s = a[:, p].to(PRECISE)
            mean = s.mean(0, keepdim=True)
            if i == 0 and kind == "diag":
                anchor = x0[p].to(PRECISE)
                local, overall = s - anchor, mean - anchor
                change[:M] += local.square().sum(1)
                change[M:2 * M] += (local * overall).sum(1)
                change[2 * M] += overall.square().sum()
                change[2 * M + 1] += anchor.square().sum()
            if i in rows:
                row = rows[i]
                row[0] += (s - mean).square().sum() / M
                row[1] += mean.square().sum()
                row[2:2 + M] += s.square().sum(1)
                row[2 + M:] += (s * mean).sum(1)
            out[i][:, p] = mean if i in rows else s
    if kind == "sync":
        return {"states": out}
    return {"change": change, "stats": torch.stack([rows[i] for i in sorted(rows)]), "states": out}
