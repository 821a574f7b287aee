"""The calls by which this library's speed is judged: what a program that optimises with it does.

A case is a dict of plain values; `kind` says which entry points a pass goes through:

  solve     a whole solve of a small swarm: create, all iterations, gbest, destroy
  steps     a swarm that a program keeps: one step(iters) and the gbest it led to, or (read "each")
            step(1) with every step's gbest read one step later while the next one runs
  paper     the same in double precision (the paper's own workload and precision), a small swarm's whole
            population read at the end (in one dimension every run ends in the same maximum)
  batch     many independent swarms of uneven size in one call
  noalloc   one iteration on a swarm in the caller's own tensors
  resume    a checkpoint loaded, some iterations, the next checkpoint
  lsq       a least-squares swarm that a program keeps: iterations, gbest and its residual
  lsq_eval  the least-squares fitness of given positions

Problem data comes from the seed; the swarms' own draws are the library's Philox under that seed.
"""
import math

import numpy as np
import torch

from paper_2205_01313_gb300 import cupso as P
from paper_2205_01313_gb300 import workloads as W

L2_BYTES = 129 << 20
FIDS = {"sphere": 0, "rastrigin": 1, "ackley": 2, "rosenbrock": 3, "cubic_max": 4}
PRECISIONS = ("fp32", "bf16", "fp8", "fp64")


def listed():
    return [
        # a user's first program: a small textbook problem solved whole (the swarm fits one cluster's shared memory)
        {"name": "solve_sphere_1024x32", "kind": "solve", "fitness": "sphere", "N": 1024, "D": 32, "iters": 1000},
        # the smallest call: one iteration inside another framework's memory pool
        {"name": "noalloc_rosenbrock_3000x20", "kind": "noalloc", "fitness": "rosenbrock", "N": 3000, "D": 20},
        # a mid-size multimodal problem whose state fits in L2
        {"name": "steps_rastrigin_65536x128", "kind": "steps", "fitness": "rastrigin", "N": 65536, "D": 128,
         "iters": 100, "read": "end"},
        # the largest single swarm, streamed from HBM, every step's result read (the benchmark's default workload)
        {"name": "steps_rosenbrock_1048576x64", "kind": "steps", "fitness": "rosenbrock", "N": 1 << 20, "D": 64,
         "iters": 20, "read": "each"},
        # sizes as problems have them: no power of two, dimensions that no vector width divides
        {"name": "steps_ackley_20011x30", "kind": "steps", "fitness": "ackley", "N": 20011, "D": 30, "iters": 200,
         "read": "end"},
        # the paper's one-dimensional experiment (Table 3), FP64
        {"name": "paper_8192x1", "kind": "paper", "fitness": "cubic_max", "N": 8192, "D": 1, "iters": 2000,
         "read": "state"},
        # the paper's 120-dimensional experiment (Table 4), FP64
        {"name": "paper_16384x120", "kind": "paper", "fitness": "cubic_max", "N": 16384, "D": 120, "iters": 20,
         "read": "end"},
        # hyper-parameter or multi-start search: 512 uneven swarms at once
        {"name": "batch_512", "kind": "batch", "swarms": 512, "shapes": 1, "iters": 100},
        # a dense fitness on the tensor cores
        {"name": "lsq_bf16_8192x1024", "kind": "lsq", "precision": "bf16", "N": 8192, "D": 1024, "M": 4096, "iters": 16},
        # the same family where the fitness has to be plain FP32
        {"name": "lsq_fp32_2048x500", "kind": "lsq", "precision": "fp32", "N": 2048, "D": 500, "M": 2000, "iters": 2},
        # scoring a set of candidate solutions with the low-precision fitness
        {"name": "lsq_eval_fp8_8192x1000", "kind": "lsq_eval", "precision": "fp8", "N": 8192, "D": 1000, "M": 4000},
        # a preempted job: load the checkpoint, run on, write the next one
        {"name": "resume_rastrigin_20000x48", "kind": "resume", "fitness": "rastrigin", "N": 20000, "D": 48, "iters": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "steps", "steps", "paper", "batch", "noalloc", "resume", "lsq", "lsq", "lsq_eval"])
    fit = rng.choice(sorted(FIDS))
    if kind == "solve":
        return {"kind": kind, "fitness": fit, "N": _log(rng, 64, 4096), "D": _log(rng, 2, 96),
                "iters": _log(rng, 100, 1000)}
    if kind == "steps":
        D = _log(rng, 2, 256)
        if rng.random() < 0.5:
            D = max(16, D // 8 * 8)
        N = _log(rng, 1000, min(1 << 20, (1 << 26) // D))
        return {"kind": kind, "fitness": fit, "N": N, "D": D, "iters": max(1, min(100, (20 << 26) // (N * D))),
                "read": rng.choice(["end", "end", "each"])}
    if kind == "paper":
        D = rng.choice([1, 1, 2, 10, 30, 120])
        N = _log(rng, 32, 131072 if D < 120 else 32768)
        return {"kind": kind, "fitness": rng.choice(["cubic_max", "cubic_max", "sphere", "rosenbrock"]), "N": N, "D": D,
                "iters": max(10, min(2000, (1 << 26) // (max(N, 2048) * D))), "read": "state" if N * D <= 1 << 18 else "end"}
    if kind == "batch":
        return {"kind": kind, "swarms": _log(rng, 8, 384), "shapes": rng.randint(2, 1 << 20), "iters": _log(rng, 20, 100)}
    if kind == "noalloc":
        return {"kind": kind, "fitness": fit, "N": _log(rng, 500, 200000), "D": _log(rng, 2, 128)}
    if kind == "resume":
        D = rng.choice([8 * rng.randint(2, 16), rng.randint(2, 128)])
        return {"kind": kind, "fitness": fit, "N": _log(rng, 1000, (1 << 22) // D), "D": D, "iters": rng.randint(1, 10)}
    D = _log(rng, 16, 1024)
    M = max(8, min(4096, int(D * rng.choice([0.5, 2.0, 4.0, 8.0])) + rng.randint(0, 40)))
    N = _log(rng, 256, 8192)
    prec = rng.choice(PRECISIONS)
    if prec == "fp64":        # the reference precision: small problems
        N, D, M = min(N, 1500), min(D, 200), min(M, 600)
    if kind == "lsq_eval":
        return {"kind": kind, "precision": prec, "N": N, "D": D, "M": M}
    return {"kind": kind, "precision": prec, "N": N, "D": D, "M": M,
            "iters": rng.randint(8, 32) if prec in ("bf16", "fp8") else 2}


# ---------------------------------------------------------------------------
# What a program has in hand
# ---------------------------------------------------------------------------
def _bounds(c):
    return W.BOUNDS[FIDS[c["fitness"]]] if "fitness" in c else W.lsq_config()["bounds"]


def _lsq_data(c, seed):
    """A (unit-norm columns in expectation), b = A x* + noise, and positions in the search box."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(c["M"], c["D"], generator=g, device="cuda") / math.sqrt(c["M"])
    xs = torch.rand(c["D"], generator=g, device="cuda") * 2 - 1
    b = (A.double() @ xs.double()).float() + 1e-3 * torch.randn(c["M"], generator=g, device="cuda")
    lo, hi, _ = W.lsq_config()["bounds"]
    X = torch.rand(c["N"], c["D"], generator=g, device="cuda") * (hi - lo) + lo
    return A.contiguous(), b.contiguous(), X.contiguous()


def _swarm_data(c, seed):
    """A swarm in mid-run on the GPU, particle-major: pos, v, pbest_pos, pbest_fit (that of pbest_pos)."""
    lo, hi, vmax = _bounds(c)
    N, D = c["N"], c["D"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    pos = (torch.rand(N, D, generator=g, device="cuda") * (hi - lo) + lo).clamp(lo, hi)
    v = ((torch.rand(N, D, generator=g, device="cuda") * 2 - 1) * vmax).clamp(-vmax, vmax)
    pb = (pos + 0.3 * vmax * torch.randn(N, D, generator=g, device="cuda")).clamp(lo, hi)
    pf = _fitness(FIDS[c["fitness"]], pb.double()).float()
    return pos, v, pb, pf


def _swarm(c, seed):
    if c["kind"] == "paper":
        S = W.PAPER_SETTING
        b = S["bounds"] if c["fitness"] == "cubic_max" else _bounds(c)
        w, c1, c2 = (S["w"], S["c1"], S["c2"]) if c["fitness"] == "cubic_max" else (W.W_STD, W.C_STD, W.C_STD)
        return P.Swarm(c["D"], c["N"], b, w, c1, c2, c["fitness"], seed, dtype="f64")
    return P.Swarm(c["D"], c["N"], _bounds(c), W.W_STD, W.C_STD, W.C_STD, c.get("fitness", "lsq"), seed)


def _batch(c, seed):
    probs = W.batch_problems(n_swarms=c["swarms"], seed=c["shapes"])
    return [dict(p, seed=seed * 100003 + k) for k, p in enumerate(probs)]


def prepare(case, seed):
    c = case
    st = {"case": c, "seed": seed}
    if c["kind"] in ("steps", "paper"):
        st["swarm"] = _swarm(c, seed)
    elif c["kind"] == "batch":
        st["problems"] = _batch(c, seed)
    elif c["kind"] == "noalloc":
        pos, v, pb, pf = _swarm_data(c, seed)
        ld = (c["N"] + 127) // 128 * 128
        pad = torch.zeros(c["D"], ld, device="cuda")
        for name, a in (("pos", pos), ("v", v), ("pbest_pos", pb)):
            st[name] = pad.clone()
            st[name][:, :c["N"]] = a.t()
        st["pbest_fit"] = torch.full((ld,), math.inf, device="cuda")
        st["pbest_fit"][:c["N"]] = pf
        st["gbest_pos"] = pb[int(torch.argmin(pf))].clone()
        st["gbest_fit"] = torch.zeros(1, device="cuda")
        st["gbest_idx"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        st["ld"], st["t"] = ld, 0
    elif c["kind"] == "resume":
        st["checkpoint"] = [a.cpu().numpy() for a in _swarm_data(c, seed)]
        st["swarm"] = _swarm(c, seed)
    elif c["kind"] in ("lsq", "lsq_eval"):
        st["A"], st["b"], st["X"] = _lsq_data(c, seed)
        if c["kind"] == "lsq":
            st["X"] = None
            st["swarm"] = _swarm(c, seed)
            torch.cuda.synchronize()
            st["swarm"].set_lsq(st["A"].data_ptr(), st["b"].data_ptr(), c["M"], c["precision"])
        else:
            st["f"] = torch.empty(c["N"], device="cuda")
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _result(r):
    status, fit, idx, pos = r
    return {"status": status, "fit": np.asarray(fit, dtype=pos.dtype), "idx": idx, "pos": pos}


def run(state):
    st, c = state, state["case"]
    kind = c["kind"]
    if kind == "solve":
        with _swarm(c, st["seed"]) as s:
            s.step(c["iters"])
            return _result(s.gbest())
    if kind in ("steps", "paper"):
        s = st["swarm"]
        if c.get("read") == "each":
            for k in range(c["iters"]):
                s.step(1)
                s.gbest_post(k & 1)
                if k:
                    last = s.gbest_wait((k - 1) & 1)
            last = s.gbest_wait((c["iters"] - 1) & 1)
            return _result(last)
        s.step(c["iters"])
        if c["read"] == "state":
            return dict(_result(s.gbest()), population=s.state())
        return _result(s.gbest())
    if kind == "batch":
        status, out = P.cupso_solve_batch(st["problems"], c["iters"])
        return {"status": status, "fit": np.array([r["fit"] for r in out], np.float32),
                "idx": np.array([r["idx"] for r in out], np.int64), "pos": np.concatenate([r["pos"] for r in out])}
    if kind == "noalloc":
        st["t"] += 1
        P.cupso_tree_step_noalloc(c["D"], c["N"], _bounds(c), W.W_STD, W.C_STD, W.C_STD, FIDS[c["fitness"]], st["seed"], 0,
                                  st["t"], st["pos"].data_ptr(), st["v"].data_ptr(), st["pbest_pos"].data_ptr(),
                                  st["pbest_fit"].data_ptr(), st["ld"], st["gbest_pos"].data_ptr(),
                                  st["gbest_fit"].data_ptr(), st["gbest_idx"].data_ptr(), st["status"].data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
        n = c["N"]
        return {"pos": st["pos"][:, :n], "v": st["v"][:, :n], "pbest_pos": st["pbest_pos"][:, :n],
                "pbest_fit": st["pbest_fit"][:n], "gbest_pos": st["gbest_pos"], "gbest_fit": st["gbest_fit"],
                "gbest_idx": st["gbest_idx"], "status": st["status"]}
    if kind == "resume":
        s = st["swarm"]
        s.set_state(*st["checkpoint"], t=100)
        s.step(c["iters"])
        return s.state()
    if kind == "lsq":
        s = st["swarm"]
        s.step(c["iters"])
        out = _result(s.gbest())
        out["residual"] = np.float64(s.gbest_f64())
        return out
    P.cupso_lsq_eval(st["A"].data_ptr(), st["b"].data_ptr(), c["M"], c["D"], st["X"].data_ptr(), c["N"],
                     P.LSQ_PRECISIONS[c["precision"]], st["f"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    return st["f"]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _swarm_work(N, D, iters, esize):
    """Every iteration reads pos, v, pbest_pos and pbest_fit and writes pos and v (a swarm that the chip's L2 holds:
    in and out once a pass); about 16 operations per particle and dimension (Eq. 1, Eq. 2, a fitness term)."""
    state = 3 * esize * N * D + esize * N
    return {"bytes": 2 * state if state <= L2_BYTES else iters * (5 * esize * N * D + esize * N),
            "flops": 16 * N * D * iters}


def work(case):
    c = case
    if c["kind"] == "batch":
        pd = sum(p["N"] * p["D"] for p in W.batch_problems(n_swarms=c["swarms"], seed=c["shapes"]))
        return _swarm_work(pd, 1, c["iters"], 4)
    if c["kind"] == "lsq_eval":
        return {"bytes": 4 * (c["N"] * c["D"] + c["M"] * c["D"] + c["M"] + c["N"]), "flops": 2 * c["N"] * c["D"] * c["M"]}
    w = _swarm_work(c["N"], c["D"], c.get("iters", 1), 8 if c["kind"] == "paper" else 4)
    if c["kind"] == "lsq":
        w = {"bytes": w["bytes"] + 4 * c["M"] * c["D"], "flops": w["flops"] + 2 * c["N"] * c["D"] * c["M"] * c["iters"]}
    if c["kind"] == "resume":   # the checkpoint in and out
        w["bytes"] += 2 * (12 * c["N"] * c["D"] + 4 * c["N"])
    return w


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words."""
    m32 = 0xFFFFFFFF
    k0, k1 = seed & m32, (seed >> 32) & m32
    zero = torch.zeros_like(c0)
    c1, c2, c3 = c1 + zero, c2 + zero, c3 + zero
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & m32) ^ c1 ^ k0, p1 & m32, ((p0 >> 32) & m32) ^ c3 ^ k1, p0 & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c0, c1, c2, c3


def _uniforms(N, D, t, seed, f64):
    """r1, r2 [N][D] of iteration t: 24 bits each, two dimensions to a call; or 53 bits each, one to a call."""
    i = torch.arange(N, device="cuda").view(-1, 1)
    if f64:
        d = torch.arange(D, device="cuda").view(1, -1)
        w = _philox(d + 0 * i, i, torch.full_like(i, t), 0 * i, seed)
        return (((w[0] << 21) + (w[1] >> 11) + 1).double() * 2.0 ** -53,
                ((w[2] << 21) + (w[3] >> 11) + 1).double() * 2.0 ** -53)
    g = torch.arange((D + 1) // 2, device="cuda").view(1, -1)
    w = [((x >> 8) + 1).double() * 2.0 ** -24 for x in _philox(g + 0 * i, i, torch.full_like(i, t), 0 * i, seed)]
    return (torch.stack((w[0], w[2]), 2).view(N, -1)[:, :D], torch.stack((w[1], w[3]), 2).view(N, -1)[:, :D])


def _fitness(fid, x, A=None, b=None):
    D = x.shape[1]
    if A is not None:
        return (x @ A.double().t() - b.double()).square().sum(1)
    if fid == 0:
        return x.square().sum(1)
    if fid == 1:
        return (x.square() - 10 * torch.cos(2 * math.pi * x) + 10).sum(1)
    if fid == 2:
        return (-20 * torch.exp(-0.2 * x.square().mean(1).sqrt()) - torch.exp(torch.cos(2 * math.pi * x).mean(1))
                + 20 + math.e)
    if fid == 3:
        return (100 * (x[:, 1:] - x[:, :-1].square()).square() + (1 - x[:, :-1]).square()).sum(1) if D > 1 else 0 * x[:, 0]
    return -(((x - 0.8) * x - 1000) * x + 8000).sum(1)


def _simulate(c, seed, state=None, t0=0, A=None, b=None):
    """`iters` iterations from `state` (or from Step 1 of the method): pos, v, pbest_pos, pbest_fit, gbest index."""
    f64 = c["kind"] == "paper"
    real = float if f64 else lambda a: float(np.float32(a))
    if f64 and c["fitness"] == "cubic_max":
        S = W.PAPER_SETTING
        (lo, hi, vmax), w, c1, c2 = S["bounds"], S["w"], S["c1"], S["c2"]
    else:
        lo, hi, vmax = (real(a) for a in _bounds(c))
        w, c1, c2 = real(W.W_STD), real(W.C_STD), real(W.C_STD)
    fid, N, D = FIDS.get(c.get("fitness")), c["N"], c["D"]
    if state is None:
        u0, u1 = _uniforms(N, D, 0, seed, f64)
        x, v = (lo + u0 * (hi - lo)).clamp(lo, hi), (u1 * 2 * vmax - vmax).clamp(-vmax, vmax)
        pb, pf = x.clone(), _fitness(fid, x, A, b)
        g = int(torch.argmin(pf))
    else:
        x, v, pb, pf = (a.double() for a in state)
        g = int(torch.argmin(pf))
    for k in range(c.get("iters", 1)):
        r1, r2 = _uniforms(N, D, t0 + 1 + k, seed, f64)
        v = (w * v + c1 * r1 * (pb - x) + c2 * r2 * (pb[g] - x)).clamp(-vmax, vmax)
        x = (x + v).clamp(lo, hi)
        f = _fitness(fid, x, A, b)
        better = f < pf
        pb, pf = torch.where(better[:, None], x, pb), torch.where(better, f, pf)
        g = int(torch.argmin(pf))
    return x, v, pb, pf, g


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "lsq_eval":
        A, b, X = _lsq_data(c, seed)
        return _fitness(None, X.double(), A, b)
    # A swarm is chaotic: over many iterations a rounding decides which particles improve, and 64 bits run another
    # trajectory. The low-precision fitness decides by its own roundings from the first iteration on.
    if kind in ("solve", "batch") or c.get("precision") in ("bf16", "fp8") or c.get("iters", 1) > 20:
        return None
    if kind == "lsq":
        A, b, _ = _lsq_data(c, seed)
        x, v, pb, pf, g = _simulate(c, seed, A=A, b=b)
        return {"status": None, "fit": pf[g], "idx": None, "pos": pb[g], "residual": pf[g]}
    if kind in ("steps", "paper"):
        x, v, pb, pf, g = _simulate(c, seed)
        out = {"status": None, "fit": pf[g], "idx": None, "pos": pb[g]}
        if c["read"] == "state":
            out["population"] = {"pos": x, "v": v, "pbest_pos": pb, "pbest_fit": pf, "t": None}
        return out
    x, v, pb, pf, g = _simulate(c, seed, state=_swarm_data(c, seed), t0=100 if kind == "resume" else 0)
    if kind == "resume":
        return {"pos": x, "v": v, "pbest_pos": pb, "pbest_fit": pf, "t": None}
    return {"pos": x.t(), "v": v.t(), "pbest_pos": pb.t(), "pbest_fit": pf, "gbest_pos": pb[g], "gbest_fit": pf[g].view(1),
            "gbest_idx": None, "status": None}
