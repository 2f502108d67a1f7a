"""The work this library is used for, as cases that can be timed and checked.

A case is one call (or one short chain of calls) through the package's Python
entry points on seeded inputs:

  round   aloco.sync            one outer round on device-resident state
  shard   aloco.sync_shard      one contiguous shard (views into the vector)
  host    aloco.sync_host       the round on page-locked host state
  int8    aloco.sync_int8       the INT8-communicated round
  codec   aloco.int8_encode, aloco.int8_decode     a worker's payload
  adamw   aloco.adamw_step      one inner optimizer step on every replica

Rounds and optimizer steps update their state in place, as a training loop
has them do, and return it whole.
"""
import math

import numpy as np
import torch

from paper_2609_36662_gb300 import aloco as A
from paper_2609_36662_gb300 import workloads as W

H_BASE, H_SEL, STEP = 100, 150, 4000
OUTER_LR, OUTER_BETA = 0.7, 0.9
ADAM_STEP, ADAM_LR = 500, 3e-4

# Largest pass of any case, listed or drawn (bytes read and written).
MOST_BYTES = 36e9


def listed():
    return [
        # The smallest round of the repository's own configurations: one
        # small parameter set, four workers; latency and launch bound.
        {"name": "round_toy", "kind": "round", "n": 1 << 20, "m": 4, "x": "f32"},
        # An ordinary small model of odd size, 8 workers.
        {"name": "round_25m", "kind": "round", "n": 25_000_003, "m": 8, "x": "f32"},
        # The Llama-style 150M set with 8 fp32 workers.
        {"name": "round_150m", "kind": "round", "n": W.LLAMA_150M.numel(), "m": 8, "x": "f32"},
        # The Llama-style 1.1B set with 4 bf16 workers: the largest round.
        {"name": "round_1b", "kind": "round", "n": W.LLAMA_1B.numel(), "m": 4, "x": "bf16"},
        # The most workers a round takes.
        {"name": "round_m32", "kind": "round", "n": 6_000_000, "m": 32, "x": "bf16"},
        # One of three shards of a vector whose size three does not divide
        # into aligned pieces: the shard's views start off a 16-byte boundary.
        {"name": "shard_odd", "kind": "shard", "n": 50_000_021, "m": 6, "x": "bf16",
         "shards": 3, "index": 1},
        # State kept in host memory (a GPU shared with the inner loops).
        {"name": "host_150m", "kind": "host", "n": W.LLAMA_150M.numel(), "m": 4, "x": "bf16"},
        # INT8 communication on the 150M set with its tensor parts.
        {"name": "int8_150m", "kind": "int8", "n": W.LLAMA_150M.numel(), "m": 8, "x": "f32",
         "parts": "llama150m"},
        # INT8 communication with 16 bf16 workers and tensor parts of odd sizes.
        {"name": "int8_m16", "kind": "int8", "n": 20_000_000, "m": 16, "x": "bf16",
         "parts": "odd"},
        # One worker's payload: encode its pseudo-gradient, decode what came.
        {"name": "codec_150m", "kind": "codec", "n": W.LLAMA_150M.numel(),
         "parts": "llama150m"},
        # The inner step of the 150M set, called some hundred times a round.
        {"name": "adamw_150m", "kind": "adamw", "n": W.LLAMA_150M.numel(), "m": 8, "x": "f32",
         "g": "f32"},
        # The inner step of a small set held in bf16: launches and host work
        # count.
        {"name": "adamw_small", "kind": "adamw", "n": 1_500_007, "m": 4, "x": "bf16",
         "g": "bf16"},
    ]


def draw(rng):
    kind = rng.choice(["round", "round", "shard", "host", "int8", "int8", "codec", "adamw"])
    x = rng.choice(["f32", "bf16"])
    if kind == "codec":
        c = {"kind": kind, "n": _size(rng, 200_000, 300e6),
             "parts": rng.choice(["flat", "odd"])}
    elif kind == "int8":
        m = rng.randint(1, 16)
        c = {"kind": kind, "n": _size(rng, 200_000, 150e6), "m": m, "x": x,
             "parts": rng.choice(["flat", "odd"])}
    elif kind == "adamw":
        c = {"kind": kind, "n": _size(rng, 200_000, 150e6), "m": rng.randint(1, 12),
             "x": x, "g": rng.choice(["f32", "bf16"])}
    elif kind == "shard":
        k = rng.randint(2, 8)
        c = {"kind": kind, "n": _size(rng, 500_000, 300e6), "m": rng.randint(1, 16), "x": x,
             "shards": k, "index": rng.randrange(k)}
    elif kind == "host":
        c = {"kind": kind, "n": _size(rng, 200_000, 100e6), "m": rng.randint(1, 8), "x": x}
    else:
        m = rng.choice([1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 16, 24, 32])
        c = {"kind": kind, "n": _size(rng, 200_000, 500e6), "m": m, "x": x}
    while work(c)["bytes"] > (3e9 if kind == "host" else MOST_BYTES):
        c["n"] = c["n"] * 2 // 3
    return c


def _size(rng, lo, hi):
    """Log-uniform; one in three sizes is a multiple of 4096, the rest fall
    where they fall."""
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    return max(4096, n // 4096 * 4096) if rng.random() < 1 / 3 else n


def parts_of(case):
    """Tensor part sizes of an INT8 vector (None: one part)."""
    n, how = case["n"], case["parts"]
    if how == "llama150m":
        return [k for _, k, _ in W.LLAMA_150M.tensors()]
    if how == "flat":
        return None
    # Matrices, vectors and single scalars of odd sizes in turn.
    unit = max(1, n // 1_600_000)
    cycle = [150_000 * unit, 769, 50_257 * unit, 1, 12_289 * unit, 4096]
    out, left = [], n
    while left:
        out.append(min(left, cycle[len(out) % len(cycle)]))
        left -= out[-1]
    return out


# ------------------------------------------------------------------ inputs

def _dtype(case, key="x"):
    return torch.float32 if case[key] == "f32" else torch.bfloat16


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(n, std, gen):
    return torch.empty(n, dtype=torch.float32, device="cuda").normal_(0.0, std, generator=gen)


def _round_inputs(case, seed):
    """theta ~ N(0, 0.02), a running momentum, and endpoints that drifted from
    theta by noise the workers share and noise of their own."""
    gen, n = _gen(seed), case["n"]
    theta = _normal(n, 0.02, gen)
    v = _normal(n, 1e-3, gen)
    shared = _normal(n, 0.6e-3, gen).add_(theta)
    xs = [_normal(n, 0.8e-3, gen).add_(shared).to(_dtype(case)) for _ in range(case["m"])]
    return theta, v, xs


def _adam_inputs(case, seed):
    """Mid-training state: moments of the gradients' size, and gradients whose
    norms lie around the clipping threshold."""
    gen, n = _gen(seed), case["n"]
    sigma = 1.0 / math.sqrt(n)
    out = {"params": [], "grads": [], "m": [], "v": []}
    for k in range(case["m"]):
        out["params"].append(_normal(n, 0.02, gen).to(_dtype(case)))
        out["grads"].append(_normal(n, sigma * (0.5 + 0.5 * (k % 4)), gen).to(_dtype(case, "g")))
        out["m"].append(_normal(n, 0.3 * sigma, gen))
        out["v"].append(_normal(n, sigma, gen).square_().add_(0.1 * sigma * sigma))
    return out


def _bounds(case):
    n, k, i = case["n"], case["shards"], case["index"]
    return n * i // k, n * (i + 1) // k


def _schedule():
    s = W.SCHED_20K
    return A.Schedule.make(s.kind, s.peak_lr, s.final_lr, s.warmup_steps, s.total_steps)


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "codec":
        st["x"] = _normal(case["n"], 1e-3, _gen(seed))
        st["parts"] = parts_of(case)
        return st
    if kind == "adamw":
        st.update(_adam_inputs(case, seed))
        st["cfg"] = A.adamw_cfg(lr=ADAM_LR, step=ADAM_STEP)
        return st
    theta, v, xs = _round_inputs(case, seed)
    if kind == "shard":
        lo, hi = _bounds(case)
        theta, v, xs = theta[lo:hi], v[lo:hi], [x[lo:hi] for x in xs]
    elif kind == "host":
        theta, v, xs = _pinned(theta), _pinned(v), [_pinned(x) for x in xs]
    elif kind == "int8":
        st["parts"] = parts_of(case)
    st.update(theta=theta, v=v, xs=xs,
              args=dict(H_sel=H_SEL, H_base=H_BASE, step=STEP, schedule=_schedule(),
                        outer_lr=OUTER_LR, outer_beta=OUTER_BETA))
    return st


# --------------------------------------------------------------------- run

def run(state):
    kind = state["kind"]
    if kind == "codec":
        codes, scales, _ = A.int8_encode(state["x"], state["parts"], want_decoded=False)
        return {"codes": codes, "scales": scales,
                "decoded": A.int8_decode(codes, scales, state["parts"])}
    if kind == "adamw":
        A.adamw_step(state["params"], state["grads"], state["m"], state["v"], state["cfg"],
                     want_stats=False)
        return {"params": state["params"], "m": state["m"], "v": state["v"]}
    theta, v, xs, args = state["theta"], state["v"], state["xs"], state["args"]
    out = {"theta": theta, "v": v, "xs": xs}
    if kind == "shard":
        _, p = A.sync_shard(theta, v, xs, **args)
        out["sum_sq"] = p.sum_sq
        out["drift"] = np.array(p.drift[:len(xs)])
        return out
    if kind == "host":
        stats = A.sync_host(theta, v, xs, **args)
        del out["xs"]  # host endpoints are read only
    elif kind == "int8":
        stats = A.sync_int8(theta, v, xs, parts=state["parts"], **args)
    else:
        stats = A.sync(theta, v, xs, **args)
    out["D"], out["C"] = stats["D"], stats["C"]
    out["drift"] = np.array(stats["drift"])
    return out


# -------------------------------------------------------------------- work

def work(case):
    n, kind = case["n"], case["kind"]
    if kind == "codec":
        # x in, codes out and in again, the decoded vector out; scales
        blocks = _blocks(case)
        return {"bytes": 10 * n + 8 * blocks, "flops": 6 * n}
    m = case["m"]
    size = 4 if case["x"] == "f32" else 2
    if kind == "adamw":
        g = 4 if case["g"] == "f32" else 2
        return {"bytes": n * m * (2 * size + g + 16), "flops": 16 * n * m}
    if kind == "shard":
        lo, hi = _bounds(case)
        n = hi - lo
    if kind == "host":
        return {"bytes": n * (16 + m * size), "flops": n * (4 * m + 12)}
    per = 10 if kind == "int8" else 4
    return {"bytes": 2 * n * (8 + m * size), "flops": n * (per * m + 12)}


def _blocks(case):
    return sum((k + 4095) // 4096 for k in (parts_of(case) or [case["n"]]))


# --------------------------------------------------------------- tolerance

def tolerance(case):
    """Each state's elements come from a few fp32 operations on inputs of their
    own size, and the statistics from fp32 partials summed in fp64."""
    kind = case["kind"]
    if kind == "codec":
        return "exact"
    if kind == "int8":
        # a last-bit change in the workers' mean moves a few of its codes by one
        return {"rel": 5e-5, "max": 0.05}
    if kind != "host" and case["x"] == "bf16":
        # a result within fp32 rounding of a bf16 tie may land one step away
        return {"rel": 2e-5, "max": 8e-3}
    return {"rel": 1e-6, "max": 2e-5}


# ------------------------------------------------------------------- exact

def _coefficients():
    """The correction's scalars for this horizon, from their definitions: the
    summed inner learning rates, rho, the clipped momentum mu^rho and the
    matching outer rate (without normalisation)."""
    s = W.SCHED_20K

    def lr(k):
        f = (k - s.warmup_steps) / (s.total_steps - s.warmup_steps)
        return s.final_lr + 0.5 * (s.peak_lr - s.final_lr) * (1.0 + math.cos(math.pi * f))
    sel = math.fsum(lr(STEP + h) for h in range(H_SEL))
    base = math.fsum(lr(STEP + h) for h in range(H_BASE))
    rho = max(sel / (base + 1e-8), 1.0)
    mu = min(max(OUTER_BETA ** rho, 0.45), 0.90)
    eta = OUTER_LR * min(rho, 1.6) * (1.0 - mu) / (1.0 - OUTER_BETA)
    return mu, eta


def _div(y, by):
    """fp32 division (torch multiplies by the reciprocal of a plain number)."""
    return y / torch.full((1,), by, dtype=y.dtype, device=y.device)


def _codec(y, parts):
    """Codes, scales and decoded values of an fp32 vector, as the codec defines
    them in fp32: scale max|y| / 127 per block of at most 4096 elements of a
    part, code rint(y / scale)."""
    codes, scales, dec = torch.empty_like(y), [], torch.empty_like(y)
    off = 0
    for size in parts or [y.numel()]:
        whole = size // 4096 * 4096
        for lo, hi, width in ((off, off + whole, 4096), (off + whole, off + size, size - whole)):
            if lo == hi:
                continue
            t = y[lo:hi].view(-1, width)
            s = _div(t.abs().amax(dim=1, keepdim=True), 127.0)
            s = torch.where(s == 0, torch.ones_like(s), s)
            q = torch.round(t / s)
            codes[lo:hi] = q.view(-1)
            dec[lo:hi] = (q * s).view(-1)
            scales.append(s.view(-1))
        off += size
    return codes, torch.cat(scales), dec


def exact(case, seed):
    kind = case["kind"]
    if kind == "codec":
        codes, scales, dec = _codec(_normal(case["n"], 1e-3, _gen(seed)), parts_of(case))
        return {"codes": None, "scales": scales.double(), "decoded": dec.double()}
    if kind == "adamw":
        return _exact_adamw(case, seed)
    theta, v, xs = _round_inputs(case, seed)
    if kind == "shard":
        lo, hi = _bounds(case)
        theta, v, xs = theta[lo:hi], v[lo:hi], [x[lo:hi] for x in xs]
    mu, eta = _coefficients()
    m, n = len(xs), theta.numel()
    drift, sq = np.zeros(m), 0.0
    mean8 = None
    if kind == "int8":
        # the codec and the workers' sum are defined in fp32
        total, parts = torch.zeros_like(theta), parts_of(case)
        for x in xs:
            total += _codec(theta - x.float(), parts)[2]
        mean8 = _codec(_div(total, float(m)), parts)[2]
    t64 = torch.empty(n, dtype=torch.float64, device=theta.device)
    v64 = torch.empty_like(t64)
    for lo in range(0, n, 1 << 26):
        at = slice(lo, min(n, lo + (1 << 26)))
        t = theta[at].double()
        s = torch.zeros_like(t)
        for k, x in enumerate(xs):
            d = t - x[at].double()
            s += d
            drift[k] += float(d.square().sum())
        mean = s / m if mean8 is None else mean8[at].double()
        sq += float(mean.square().sum())
        nv = mu * v[at].double() + mean
        v64[at] = nv
        t64[at] = t - eta * (mean + mu * nv)
    out = {"theta": t64, "v": v64, "xs": [t64] * m, "drift": drift}
    if kind == "shard":
        out["sum_sq"] = sq * m * m
        return out
    if kind == "host":
        del out["xs"]
        out["theta"], out["v"] = t64.cpu(), v64.cpu()
    D = float(drift.sum()) / m
    out["D"], out["C"] = D, m * sq / (D + 1e-8)
    return out


def _exact_adamw(case, seed):
    st = _adam_inputs(case, seed)
    b1, b2, eps, decay = 0.9, 0.95, 1e-8, 0.1
    c1, c2 = 1.0 - b1 ** ADAM_STEP, 1.0 - b2 ** ADAM_STEP
    out = {"params": [], "m": [], "v": []}
    for x, g, m, v in zip(st["params"], st["grads"], st["m"], st["v"]):
        norm = math.sqrt(sum(float(p.double().square().sum()) for p in g.split(1 << 26)))
        c = min(1.0, 1.0 / (norm + 1e-6))
        g64 = g.double() * c
        m64 = b1 * m.double() + (1.0 - b1) * g64
        v64 = b2 * v.double() + (1.0 - b2) * g64.square_()
        step = (m64 / c1) / ((v64 / c2).sqrt_() + eps)
        out["params"].append(x.double() * (1.0 - ADAM_LR * decay) - ADAM_LR * step)
        out["m"].append(m64)
        out["v"].append(v64)
    return out
