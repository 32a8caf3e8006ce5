"""Performance cases of the determinant library: what a user has it do, from
one small matrix handed over as a host array to the 256-matrix batch and a
streamed four-variable Sylvester matrix, through the public entry points
(``pipeline.determinant``, ``runner.PlainRunner`` / ``BatchedRunner``, the
stage calls of ``binding.Plan``, the predictor's training step).

A case is a dict of plain values; ``kind`` says which entry point it goes
through:

* ``call``    ``determinant(coeffs, degs)`` on host arrays, options included;
* ``plain``   ``PlainRunner``: upload, every stage, download of one prepared
              matrix (all primes in one launch per stage where they fit);
* ``batch``   ``BatchedRunner`` over ``count`` matrices of the batched
              distribution (n 4-24, 1-3 variables, degrees 1-4, int16), with
              or without CUDA graphs;
* ``eval``, ``condense``, ``interp_crt``  single stages of a ``Plan`` on
              device buffers, as a program with its own memory plan (per-prime
              chunks, several streams) calls them;
* ``full``    the power-of-two grid of the paper: evaluation, condensation,
              inverse transform;
* ``stream``  slab-streamed evaluation + condensation of a four-variable
              Sylvester matrix with the entry map, then interpolation;
* ``mlp``     one training step of the run-time predictor.

Inputs depend on the seed alone; shapes on the case alone.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_2010_12117_gb300 import binding, synth
from paper_2010_12117_gb300.pipeline import determinant, entry_l1
from paper_2010_12117_gb300.predictor import init_params
from paper_2010_12117_gb300.runner import BatchedRunner, PlainRunner

LR, BETA1, BETA2, EPS, DECAY = 3e-3, 0.9, 0.999, 1e-8, 1e-4  # the predictor's training settings


def listed():
    return [
        # the smallest use: one dense 4x4 over Z[x, y] as a host array, exact integers back
        {"name": "call_4x4", "kind": "call", "make": "dense", "n": 4, "degs": "2,2", "density": 1.0, "mag": 10,
         "tight": False, "unique": False, "early": False},
        # resultant of two univariate-coefficient polynomials: a few hundred nodes per prime, latency counts
        {"name": "plain_16x16_sylvester", "kind": "plain", "make": "sylvester", "n": 16, "degs": "6",
         "density": 1.0, "mag": 32767},
        # one sparse trivariate matrix: 50,653 nodes per prime, a few primes
        {"name": "plain_12x12_xyz", "kind": "plain", "make": "dense", "n": 12, "degs": "3,3,3", "density": 0.3,
         "mag": 127},
        # the large request of the served stream: order 32, the largest the library takes
        {"name": "plain_32x32_xy", "kind": "plain", "make": "dense", "n": 32, "degs": "6,6", "density": 1.0,
         "mag": 32767},
        # one wave of the continuous-batching server: a handful of mixed jobs, no graphs
        {"name": "wave_16", "kind": "batch", "count": 16, "shapes": 11, "graphs": False},
        # the throughput batch: 256 mixed matrices, captured graphs, autotuned
        {"name": "batch_256", "kind": "batch", "count": 256, "shapes": 0, "graphs": True},
        # evaluation of a trivariate matrix on the node grid, more output than L2 holds
        {"name": "eval_12x12_xyz", "kind": "eval", "n": 12, "degs": "3,3,3", "P": 20},
        # the paper's own grid (powers of two): forward and inverse transforms in full
        {"name": "full_12x12_xyz", "kind": "full", "n": 12, "degs": "3,3,3", "P": 5},
        # condensation of the batch's largest order, the stage most of its time goes to
        {"name": "condense_24", "kind": "condense", "n": 24, "degs": "6,6", "P": 10},
        # from determinant values back to integers: 73^3 nodes and coefficients
        {"name": "interp_crt_73x3", "kind": "interp_crt", "n": 24, "degs": "3,3,3", "P": 18},
        # the largest: 2.8e8 nodes per prime, two primes of a longer run
        {"name": "stream_15x15_4vars", "kind": "stream", "degs_f": "22,13,9,3", "degs_g": "18,10,7,3", "m": 8,
         "l": 7, "density": 0.01, "P": 2, "ws_gb": 24.0},
        # predictor training (calibration sets are a few dozen jobs): forward, backward, Adam in fp32
        {"name": "mlp_step_64", "kind": "mlp", "rows": 64},
    ]


# ---------------------------------------------------------------------------
# Drawn cases
# ---------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _degs(rng, n, k, cap, most=7):
    """At most k degrees in [1, most] whose node grid prod (n d + 1) stays within cap."""
    while k > 1 and (n + 1) ** k > cap:
        k -= 1
    while True:
        d = [rng.randint(1, most) for _ in range(k)]
        if math.prod(n * x + 1 for x in d) <= cap:
            return ",".join(map(str, d))


def draw(rng):
    kind = rng.choice(["call", "plain", "plain", "batch", "batch", "eval", "full", "condense", "condense",
                       "interp_crt", "interp_crt", "stream", "mlp"])
    if kind == "call":
        n, k = rng.randint(2, 12), rng.randint(1, 3)
        return {"kind": "call", "make": "dense", "n": n, "degs": _degs(rng, n, k, 20_000, 4),
                "density": round(rng.uniform(0.3, 1.0), 3), "mag": _log_int(rng, 3, 32767),
                "tight": rng.random() < 0.5, "unique": rng.random() < 0.3, "early": rng.random() < 0.3}
    if kind == "plain":
        n, k = rng.randint(4, 32), rng.randint(1, 3)
        return {"kind": "plain", "make": "dense", "n": n, "degs": _degs(rng, n, k, 200_000 if n <= 24 else 60_000),
                "density": round(rng.uniform(0.3, 1.0), 3), "mag": _log_int(rng, 10, 32767)}
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 2, 160), "shapes": rng.randrange(1, 1 << 20),
                "graphs": rng.random() < 0.5}
    if kind == "eval":
        n, k = rng.randint(3, 32), rng.randint(1, 4)
        degs = _degs(rng, n, k, 400_000)
        words = n * n * math.prod(n * int(d) + 1 for d in degs.split(","))
        return {"kind": "eval", "n": n, "degs": degs, "P": _log_int(rng, 1, max(1, min(30, 500_000_000 // words)))}
    if kind == "full":
        n, k = rng.randint(3, 16), rng.randint(1, 3)
        degs = _degs(rng, n, k, 60_000, 4)
        return {"kind": "full", "n": n, "degs": degs, "P": rng.randint(2, 8)}
    if kind == "condense":
        n, k = rng.randint(2, 32), rng.randint(1, 3)
        degs = _degs(rng, n, k, 300_000)
        g = math.prod(n * int(d) + 1 for d in degs.split(","))
        most = max(1, min(40, 400_000_000 // (n * n * g), 20_000_000_000 // (g * n ** 3)))
        return {"kind": "condense", "n": n, "degs": degs, "P": _log_int(rng, 1, most)}
    if kind == "interp_crt":
        n, k = rng.randint(2, 32), rng.randint(1, 4)
        degs = _degs(rng, n, k, 500_000)
        return {"kind": "interp_crt", "n": n, "degs": degs, "P": _log_int(rng, 2, 40)}
    if kind == "stream":
        m, l = rng.randint(2, 8), rng.randint(2, 7)
        while True:
            f = [rng.randint(1, 12) for _ in range(rng.randint(2, 4))]
            g = [max(1, x - rng.randint(0, 3)) for x in f]
            if 50_000 <= math.prod(l * a + m * b + 1 for a, b in zip(f, g)) <= 20_000_000:
                break
        return {"kind": "stream", "degs_f": ",".join(map(str, f)), "degs_g": ",".join(map(str, g)), "m": m, "l": l,
                "density": 0.2, "P": 2, "ws_gb": round(rng.uniform(2.0, 6.0), 2)}
    return {"kind": "mlp", "rows": _log_int(rng, 8, 600)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _ints(text):
    return tuple(int(x) for x in str(text).split(","))


def _matrix(case, seed):
    """The polynomial matrix of a call / plain case."""
    rng = np.random.default_rng(seed)
    degs, mag = _ints(case["degs"]), case["mag"]
    if case["make"] == "sylvester":
        half = case["n"] // 2
        f, g = (rng.integers(-mag, mag + 1, (half + 1, degs[0] + 1)).astype(np.int64) for _ in range(2))
        return synth.sylvester_layout(f, g)
    return synth.random_matrix(rng, case["n"], degs, case["density"], -mag, mag + 1)


def _members(case, seed):
    """The matrices of a batch: shapes from the case, coefficients from the seed."""
    shapes, values = np.random.default_rng(case["shapes"]), np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        n, k = int(shapes.integers(4, 25)), int(shapes.integers(1, 4))
        degs = tuple(int(d) for d in shapes.integers(1, 5, k))
        density = float(shapes.uniform(0.3, 1.0))
        out.append(synth.random_matrix(values, n, degs, density, synth.INT16_LO, synth.INT16_HI))
    return out


_COUNTS = {}


def _prime_counts(case):
    """Primes per matrix, a property of the case: the coefficient bound of one drawing of its matrices with 15 % larger
    entries, so that inputs of every seed have outputs of one size."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _COUNTS:
        mats = _members(case, 0) if case["kind"] == "batch" else [_matrix(case, 0)]
        _COUNTS[key] = [binding.hadamard_primes(np.ceil(1.15 * entry_l1(m.coeffs)).astype(np.int64))[0] for m in mats]
    return _COUNTS[key]


def _sylvester(case, seed):
    return synth.sylvester(np.random.default_rng(seed), case["m"], case["l"], _ints(case["degs_f"]),
                           _ints(case["degs_g"]), case["density"], -128, 128)


def _residues(plan, words, seed):
    """[P][words] uniform residues, row q in [0, p_q)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty(plan.P, words, dtype=torch.int32, device="cuda")
    for q, p in enumerate(plan.primes):
        torch.randint(0, p, (words,), generator=gen, dtype=torch.int32, device="cuda", out=out[q])
    return out.reshape(-1)


def _coefficients(n, degs, seed):
    rng = np.random.default_rng(seed)
    return synth.random_matrix(rng, n, degs, 0.7, synth.INT16_LO, synth.INT16_HI).coeffs.astype(np.int32)


def _empty(words, dtype=torch.int32):
    return torch.empty(max(1, int(words)), dtype=dtype, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "call":
        pm = _matrix(case, seed)
        s.update(coeffs=pm.coeffs, degs=pm.degs, P=_prime_counts(case)[0])
    elif kind == "plain":
        s["runner"] = PlainRunner([_matrix(case, seed)], nprimes=_prime_counts(case))
    elif kind == "batch":
        st = s["stream"] = torch.cuda.Stream()
        s["runner"] = BatchedRunner(_members(case, seed), nprimes=_prime_counts(case),
                                    tune=True if case["graphs"] else "cache", stream=st)
        if case["graphs"]:
            s["runner"].upload(st)
            s["runner"].capture(st)
    elif kind == "stream":
        pm = _sylvester(case, seed)
        D = tuple(case["l"] * f + case["m"] * g for f, g in zip(_ints(case["degs_f"]), _ints(case["degs_g"])))
        order = sorted(range(len(D)), key=lambda v: (pm.degs[v], v))  # lowest degree first, as determinant() takes them
        shape = tuple(d + 1 for d in pm.degs)
        c = pm.coeffs.reshape((pm.n, pm.n) + shape).transpose((0, 1) + tuple(2 + v for v in order))
        emap, U, uniq = binding.unique_entries(c.reshape(pm.n, pm.n, -1))
        plan = s["plan"] = binding.Plan(pm.n, [pm.degs[v] for v in order], case["P"], det_degs=[D[v] for v in order])
        plan.set_entry_map(emap, U)
        s["coeffs"] = torch.from_numpy(uniq.reshape(-1)).cuda()
        words = max(plan.stream_ws_words(1), plan.interp_ws_words,
                    min(plan.stream_ws_words(plan.M[0]), int(case["ws_gb"] * 2 ** 28)))
        s.update(ws=_empty(words), detv=_empty(plan.G), residues=_empty(plan.P * plan.C))
    elif kind == "mlp":
        B, gen = case["rows"], torch.Generator(device="cuda").manual_seed(seed)
        f32 = dict(dtype=torch.float32, device="cuda")
        p = torch.from_numpy(init_params(seed)).cuda()
        s.update(params=p, m=torch.zeros_like(p), v=torch.zeros_like(p), grads=torch.empty_like(p), step=0,
                 x=torch.rand(B, 8, generator=gen, **f32), t=torch.randn(B, 2, generator=gen, **f32),
                 y=torch.empty(B, 2, **f32), act=torch.empty(B, 128, **f32), delta=torch.empty(B, 130, **f32),
                 loss=torch.empty(1, **f32))
    else:
        n, degs, P = case["n"], _ints(case["degs"]), case["P"]
        plan = s["plan"] = binding.Plan(n, degs, P, full_grid=kind == "full")
        if kind in ("eval", "full"):
            s["coeffs"] = torch.from_numpy(_coefficients(n, degs, seed).reshape(-1)).cuda()
            s["evals"] = _empty(P * plan.entries * plan.G)
            s["ws"] = plan.workspace(P)
        elif kind == "condense":
            s["evals"] = _residues(plan, plan.entries * plan.G, seed)
        else:
            s["detv"] = _residues(plan, plan.G, seed)
            s.update(ws=_empty(P * plan.interp_ws_words), limbs=_empty(plan.C * plan.W))
        if kind in ("full", "condense"):
            s["detv"] = _empty(P * plan.G)
        if kind in ("full", "interp_crt"):
            s["residues"] = _empty(P * plan.C)
    return s


def run(s):
    kind, plan, st = s["kind"], s.get("plan"), s.get("stream") or torch.cuda.current_stream()
    if kind == "call":
        c = s["case"]
        r = determinant(s["coeffs"], s["degs"], nprimes=s["P"], tight_degrees=c["tight"],
                        unique_entries=c["unique"], early_stop=c["early"])
        return {"limbs": r.limbs.view(np.int32), "D": list(r.D), "P": r.P}
    if kind in ("plain", "batch"):
        r = s["runner"]
        r.upload(st)
        r.compute(st)
        r.download(st)
        return r.limbs
    if kind == "eval":
        plan.eval(s["coeffs"], 0, plan.P, s["evals"], s["ws"], st)
        return s["evals"]
    if kind == "condense":
        plan.condense(s["evals"], 0, plan.P, s["detv"], st)
        return s["detv"]
    if kind == "interp_crt":
        plan.interp(s["detv"], 0, plan.P, s["residues"], s["ws"], st)
        plan.crt(s["residues"], s["limbs"], st)
        return {"residues": s["residues"], "limbs": s["limbs"]}
    if kind == "full":
        plan.eval(s["coeffs"], 0, plan.P, s["evals"], s["ws"], st)
        plan.condense(s["evals"], 0, plan.P, s["detv"], st)
        plan.interp(s["detv"], 0, plan.P, s["residues"], s["ws"], st)
        return {"evals": s["evals"], "dets": s["detv"], "residues": s["residues"]}
    if kind == "stream":
        for q in range(plan.P):
            plan.eval_condense(s["coeffs"], q, q + 1, s["detv"], s["ws"], st)
            plan.interp(s["detv"], q, q + 1, s["residues"][q * plan.C:(q + 1) * plan.C], s["ws"], st)
        return s["residues"]
    binding.mlp_forward(s["params"], s["x"], s["y"], s["act"], st)
    binding.mlp_backward(s["params"], s["x"], s["t"], s["y"], s["act"], s["delta"], s["grads"], s["loss"], st)
    s["step"] += 1
    binding.mlp_adam(s["params"], s["grads"], s["m"], s["v"], s["step"], LR, BETA1, BETA2, EPS, DECAY, st)
    return {k: s[k] for k in ("y", "loss", "grads", "params", "m", "v")}


# ---------------------------------------------------------------------------
# Necessary work
# ---------------------------------------------------------------------------
@lru_cache(maxsize=None)
def _primes():
    """The library's prime order: c 2^20 + 1 in (2^30, 2^31), those up to 1865126253 first, each group descending."""
    def prime(x):
        return all(x % d for d in range(3, math.isqrt(x) + 1, 2))
    every = [p for p in range((1 << 31) - (1 << 20) + 1, 1 << 30, -(1 << 20)) if prime(p)]
    return [p for p in every if p <= 1865126253] + [p for p in every if p > 1865126253]


def _limb_words(P):
    return (math.prod(_primes()[:P]).bit_length() + 31) // 32


def _updates(n):
    """Multiply-adds of one elimination."""
    return (n - 1) * n * (2 * n - 1) // 6


def _job_work(n, degs, P):
    G = math.prod(n * d + 1 for d in degs)
    E = math.prod(d + 1 for d in degs)
    return 4.0 * (n * n * E + G * _limb_words(P)), 2.0 * P * G * _updates(n)


def work(case):
    kind = case["kind"]
    if kind in ("call", "plain"):
        b, f = _job_work(case["n"], _ints(case["degs"]), _prime_counts(case)[0])
    elif kind == "batch":
        b = f = 0.0
        for pm, P in zip(_members(case, 0), _prime_counts(case)):
            x, y = _job_work(pm.n, pm.degs, P)
            b, f = b + x, f + y
    elif kind == "stream":
        n, P = case["m"] + case["l"], case["P"]
        df, dg = _ints(case["degs_f"]), _ints(case["degs_g"])
        G = math.prod(case["l"] * x + case["m"] * y + 1 for x, y in zip(df, dg))
        E = math.prod(max(x, y) + 1 for x, y in zip(df, dg))
        b, f = 4.0 * (E * (n + 2) + P * G), 2.0 * P * G * _updates(n)
    elif kind == "mlp":
        B, params = case["rows"], binding.MLP_PARAMS
        b = 4.0 * (7 * params + B * 12)  # params, m, v read and written, gradients written
        f = 6.0 * B * (8 * 64 + 64 * 64 + 64 * 2) + 12.0 * params
    else:
        n, degs, P = case["n"], _ints(case["degs"]), case["P"]
        C, E = math.prod(n * d + 1 for d in degs), math.prod(d + 1 for d in degs)
        G = math.prod(1 << (n * d).bit_length() for d in degs) if kind == "full" else C
        if kind == "eval":
            b, f = 4.0 * (n * n * E + P * n * n * G), 2.0 * P * n * n * G
        elif kind == "condense":
            b, f = 4.0 * P * G * (n * n + 1), 2.0 * P * G * _updates(n)
        elif kind == "full":
            b, f = 4.0 * (n * n * E + P * (n * n * G + G + C)), 2.0 * P * G * _updates(n)
        else:
            b = 4.0 * (2 * P * C + C * _limb_words(P))
            f = 2.0 * C * (P * sum(math.log2(n * d + 1) for d in degs) + P * (P + 1) / 2)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _det_mod(a, p):
    """Determinants mod p of a [n][n][nodes] int64 tensor of residues (Gaussian elimination with a row search)."""
    n, nodes = a.shape[0], a.shape[2]
    det = torch.ones(nodes, dtype=torch.int64, device=a.device)
    for c in range(n):
        row = (a[c:, c] != 0).to(torch.int8).argmax(0) + c  # first nonzero row of each node
        at = row.expand(1, n, nodes)
        top, other = a[c].clone(), a.gather(0, at)[0]
        a.scatter_(0, at, top[None])
        a[c] = other
        det = torch.where(row == c, det, (p - det) % p) * a[c, c] % p
        inv, base, e = torch.ones_like(det), a[c, c].clone(), p - 2
        while e:
            if e & 1:
                inv = inv * base % p
            base, e = base * base % p, e >> 1
        for i in range(c + 1, n):
            f = a[i, c] * inv % p
            a[i, c:] = (a[i, c:] + (p - f) * a[c, c:]) % p
    return det


def _exact_mlp(case, seed):
    s = prepare(case, seed)
    p = s["params"].double().requires_grad_(True)
    shapes, parts, at = ((64, 8), (64,), (64, 64), (64,), (2, 64), (2,)), [], 0
    for sh in shapes:
        parts.append(p[at:at + math.prod(sh)].reshape(sh))
        at += math.prod(sh)
    w1, b1, w2, b2, w3, b3 = parts
    h = torch.relu(s["x"].double() @ w1.T + b1)
    y = torch.relu(h @ w2.T + b2) @ w3.T + b3
    loss = 0.5 * (y - s["t"].double()).square().sum(1).mean()
    (g,) = torch.autograd.grad(loss, p)
    m, v, old = (1 - BETA1) * g, (1 - BETA2) * g * g, p.detach()
    new = old - LR * ((m / (1 - BETA1)) / ((v / (1 - BETA2)).sqrt() + EPS) + DECAY * old)
    return {"y": y.detach(), "loss": loss.detach().reshape(1), "grads": g, "params": new, "m": m, "v": v}


def exact(case, seed):
    """What run() returns, in 64-bit arithmetic: the predictor's step, and determinants mod p of moderate size.
    The other cases return exact integers of long chains (None)."""
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "condense" and case["n"] <= 24:
        n = case["n"]
        s = prepare(case, seed)
        G = s["plan"].G
        ev = s["evals"].reshape(case["P"], n, n, G)
        return torch.cat([_det_mod(ev[q].to(torch.int64), _primes()[q]) for q in range(case["P"])]).to(torch.int32)
    return None
