"""The work that a user of this library has it do, as cases that can be timed
and whose results can be compared.

Every case goes through the public entry points of
``paper_1507_07039_gb300.panda``.  A pass does not depend on the passes
before it: the static step works on copies of its networks, a kept context or
set is first put back to its start networks (``panda_set_state``), and the
whole-program case creates its own context.

Kinds of case:

* ``static``  one iteration in place on caller-owned device networks
  (``panda_step_static``, T and G up to 512, FP32);
* ``run``     a kept context: start networks in, ``iters`` iterations (or, with
  ``iters`` 0, up to 200 until h < 1e-3), the three networks out, all in device
  memory;
* ``set``     a kept set of uneven networks, each put back, iterated together
  and read out, in device memory;
* ``program`` a whole program on host data: create from expression data
  (Pearson prior and Z-score on the GPU), iterate, read back, destroy.

Networks are the library's synthetic ones (a Bernoulli motif prior, a
Bernoulli interaction prior, the correlation of a factor model's samples; or
identity priors), made here on the GPU and, where a context takes them as they
are, Z-scored in FP64.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1507_07039_gb300 import panda

ALPHA = 0.1
PREC = {"fp32": panda.PANDA_FP32, "bf16x3": panda.PANDA_BF16X3, "bf16x2": panda.PANDA_BF16X2,
        "fp8mix": panda.PANDA_FP8MIX}
MAX_ITER, TOL = 200, 1e-3


def listed():
    return [
        # one step of a small network (64 TFs x 256 genes) inside a program that owns its device
        # memory: the smallest call, launches and latency count
        {"name": "static_64x256", "kind": "static", "T": 64, "G": 256},
        # the paper's Table I: P = C = I, random W, FP32 (the library's default mode), to h < 1e-3;
        # its smallest size and one of its larger ones
        {"name": "table1_125", "kind": "run", "prec": "fp32", "T": 125, "G": 125, "identity": True, "iters": 0},
        {"name": "table1_1000", "kind": "run", "prec": "fp32", "T": 1000, "G": 1000, "identity": True, "iters": 0},
        # a bacterium-sized network with ragged edges, in the default mode and on the tensor cores
        {"name": "fp32_250x2100", "kind": "run", "prec": "fp32", "T": 250, "G": 2100, "identity": False, "iters": 10},
        {"name": "bf16x3_250x2100", "kind": "run", "prec": "bf16x3", "T": 250, "G": 2100, "identity": False,
         "iters": 10},
        # human TF count on the 5200 most variable genes, default mode
        {"name": "fp32_1000x5200", "kind": "run", "prec": "fp32", "T": 1000, "G": 5200, "identity": False, "iters": 6},
        # the human-sized network: the default mode, the headline mode, the fastest mode
        {"name": "fp32_1000x17000", "kind": "run", "prec": "fp32", "T": 1000, "G": 17000, "identity": False,
         "iters": 3},
        {"name": "bf16x3_1000x17000", "kind": "run", "prec": "bf16x3", "T": 1000, "G": 17000, "identity": False,
         "iters": 6},
        {"name": "fp8mix_1000x17000", "kind": "run", "prec": "fp8mix", "T": 1000, "G": 17000, "identity": False,
         "iters": 2},
        # the largest network that is benchmarked
        {"name": "bf16x3_1600x30000", "kind": "run", "prec": "bf16x3", "T": 1600, "G": 30000, "identity": False,
         "iters": 3},
        # networks of several conditions, of uneven sizes, iterated together
        {"name": "set12_bf16x3", "kind": "set", "prec": "bf16x3", "n": 12, "t_lo": 200, "t_hi": 1000, "g_lo": 2000,
         "g_hi": 8000, "iters": 6},
        # a whole program: expression data in host memory to networks in host memory
        {"name": "program_600x6000", "kind": "program", "prec": "bf16x3", "T": 600, "G": 6000, "samples": 120,
         "iters": 12},
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the same ranges."""
    kind = rng.choice(["static", "table1", "run", "run", "run", "set", "program"])
    if kind == "static":
        return {"kind": "static", "T": _log_int(rng, 16, 512), "G": _log_int(rng, 32, 512)}
    if kind == "table1":
        n = _log_int(rng, 125, 2000)
        return {"kind": "run", "prec": rng.choice(["fp32", "bf16x3"]), "T": n, "G": n, "identity": True, "iters": 0}
    if kind == "set":
        return {"kind": "set", "prec": "bf16x3", "n": rng.randint(3, 12), "t_lo": 100, "t_hi": _log_int(rng, 200, 1000),
                "g_lo": 500, "g_hi": _log_int(rng, 1000, 8000), "iters": rng.randint(2, 6)}
    if kind == "program":
        return {"kind": "program", "prec": rng.choice(["fp32", "bf16x3"]), "T": _log_int(rng, 60, 800),
                "G": _log_int(rng, 400, 7000), "samples": _log_int(rng, 20, 300), "iters": rng.randint(2, 12)}
    prec = rng.choice(["fp32", "fp32", "bf16x3", "bf16x3", "bf16x2", "fp8mix"])
    # FP32 up to the human-sized network, the tensor-core modes up to the largest
    T = _log_int(rng, 60, 1000 if prec == "fp32" else 1600)
    G = _log_int(rng, max(T, 250), 17000 if prec == "fp32" else 30000)
    most = 3 if G > 9000 else 10
    return {"kind": "run", "prec": prec, "T": T, "G": G, "identity": False,
            "iters": rng.randint(1, min(most, 2) if prec == "fp8mix" else most)}


# ---- inputs --------------------------------------------------------------------

def _generator(seed: int, k: int = 0) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (int(seed) + 1) + k)
    return g


def _rand_expression(g, G, samples):
    """Genes x samples from a tenth as many latent factors, plus noise."""
    k = max(2, samples // 10)
    L = torch.randn(G, k, generator=g, device="cuda")
    F = torch.randn(k, samples, generator=g, device="cuda")
    return L @ F + 0.5 * torch.randn(G, samples, generator=g, device="cuda")


def _rand_priors(g, T, G):
    W = (torch.rand(T, G, generator=g, device="cuda") < 0.05).float()
    up = (torch.rand(T, T, generator=g, device="cuda") < 0.02).float().triu_(1)
    P = up + up.T
    P.fill_diagonal_(1.0)
    return W, P


def _zscore(X):
    """One global mean and population standard deviation, in FP64, rounded once."""
    Y = X.double()
    Y -= Y.mean()
    Y /= Y.square().mean().sqrt()
    return Y.float()


def _networks(T, G, identity, seed, k=0):
    """Z-scored start networks (W, P, C) on the GPU, P and C exactly symmetric."""
    g = _generator(seed, k)
    W, P = _rand_priors(g, T, G)
    if identity:
        P, C = torch.eye(T, device="cuda"), torch.eye(G, device="cuda")
    else:
        X = _rand_expression(g, G, 100)
        X -= X.mean(1, keepdim=True)
        X /= X.norm(dim=1, keepdim=True)
        C = (X @ X.T).triu_(1)
        C = C + C.T
        C.fill_diagonal_(1.0)
    return _zscore(W), _zscore(P), _zscore(C)


def _set_sizes(case):
    """The uneven sizes of a set: a property of the case, not of the seed."""
    r = random.Random(1507)
    return [(r.randint(case["t_lo"], case["t_hi"]), r.randint(case["g_lo"], case["g_hi"])) for _ in range(case["n"])]


def _raw_program(case, seed):
    g = _generator(seed)
    W, P = _rand_priors(g, case["T"], case["G"])
    return W, P, _rand_expression(g, case["G"], case["samples"])


def _pinned(x):
    return x.cpu().pin_memory().numpy()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "static":
        return {"case": case, "nets": _networks(case["T"], case["G"], False, seed)}
    if kind == "run":
        nets = _networks(case["T"], case["G"], case["identity"], seed)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        ctx = panda.PandaContext(*nets, prec=PREC[case["prec"]], normalize=False, device=True,
                                 stream=stream.cuda_stream)
        return {"case": case, "nets": nets, "stream": stream, "ctx": ctx}
    if kind == "set":
        nets = [_networks(T, G, False, seed, k) for k, (T, G) in enumerate(_set_sizes(case))]
        batch = panda.PandaBatch([tuple(x.cpu().numpy() for x in n) for n in nets], prec=PREC[case["prec"]],
                                 normalize=False)
        return {"case": case, "nets": nets, "batch": batch, "handles": [batch.context(k) for k in range(len(nets))]}
    W, P, X = (_pinned(x) for x in _raw_program(case, seed))
    T, G = case["T"], case["G"]
    out = [torch.empty(s, pin_memory=True).numpy() for s in ((T, G), (T, T), (G, G))]
    return {"case": case, "W": W, "P": P, "X": X, "out": out}


# ---- one pass ------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "static":
        W, P, C = (x.clone() for x in state["nets"])
        h = panda.panda_step_static(case["T"], case["G"], W, P, C, ALPHA, 1,
                                    stream=torch.cuda.current_stream().cuda_stream)
        return {"W": W, "P": P, "C": C, "h": h}
    if kind == "run":
        ctx, nets = state["ctx"], state["nets"]
        panda.panda_set_state_device(ctx.h, *nets, 0)
        if case["iters"]:
            _, n, _ = ctx.run(ALPHA, 0.0, case["iters"])
        else:
            _, n, _ = ctx.run(ALPHA, TOL, MAX_ITER)
        out = [torch.empty_like(x) for x in nets]
        panda.panda_get_device(ctx.h, *out)
        return {"W": out[0], "P": out[1], "C": out[2], "iterations": n}
    if kind == "set":
        for h, nets in zip(state["handles"], state["nets"]):
            panda.panda_set_state_device(h, *nets, 0)
        _, n, _ = state["batch"].run(ALPHA, 0.0, case["iters"])
        outs = []
        for h, nets in zip(state["handles"], state["nets"]):
            out = [torch.empty_like(x) for x in nets]
            panda.panda_get_device(h, *out)
            outs.append(out)
        return {"networks": outs, "iterations": n}
    W, P, C = state["out"]
    with panda.PandaContext.from_expression(state["W"], state["P"], state["X"], prec=PREC[case["prec"]]) as ctx:
        _, n, _ = ctx.run(ALPHA, 0.0, case["iters"])
        panda.panda_get_into(ctx.h, W, P, C)
    return {"W": W, "P": P, "C": C, "iterations": n}


# ---- what a pass cannot do without ---------------------------------------------

def _iter_flops(T, G):
    # W.C and P.W, and the symmetric halves of W'^T.W' and W'.W'^T
    return 3.0 * T * G * G + 3.0 * T * T * G


def _net_bytes(T, G):
    return 4.0 * (T * G + T * T + G * G)


def work(case):
    kind = case["kind"]
    if kind == "set":
        sizes = _set_sizes(case)
        return {"bytes": 2 * sum(_net_bytes(T, G) for T, G in sizes),
                "flops": case["iters"] * sum(_iter_flops(T, G) for T, G in sizes)}
    T, G = case["T"], case["G"]
    if kind == "static":
        return {"bytes": 2 * _net_bytes(T, G), "flops": _iter_flops(T, G)}
    if kind == "run":
        # a run to convergence takes at least ten iterations on these networks
        return {"bytes": 2 * _net_bytes(T, G), "flops": (case["iters"] or 10) * _iter_flops(T, G)}
    return {"bytes": _net_bytes(T, G) + 4.0 * (T * G + T * T + G * case["samples"]),
            "flops": case["iters"] * _iter_flops(T, G) + 1.0 * G * G * case["samples"]}


# ---- the same in 64 bits -------------------------------------------------------

def _tan(num, nx, ny):
    """x.y / sqrt(|x|^2 + |y|^2 - |x.y|) in place of x.y (0 where both vectors are zero)."""
    den = (nx[:, None] + ny[None, :]).sub_(num.abs()).sqrt_()
    num.div_(den)
    return num.nan_to_num_(0.0, 0.0, 0.0)


def _eq5_eq6(X, S, alpha, mult, t):
    """The damped update of a symmetric network and its diagonal rule."""
    n = X.shape[0]
    dg = X.diagonal().clone()
    X = X.mul_(1.0 - alpha).add_(S, alpha=alpha)
    X.fill_diagonal_(0.0)
    if n > 2:
        mean = X.sum(1) / (n - 1)
        D = X - mean[:, None]
        D.fill_diagonal_(0.0)
        sigma = (D.square_().sum(1) / (n - 1)).sqrt()
    else:
        sigma = torch.zeros_like(dg)
    X.diagonal().copy_((1.0 - alpha) * dg + alpha * mult * sigma * math.exp(2.0 * alpha * t))
    return X


def _iterate(W, P, C, iters, tol=None):
    """Eqs. 2-7 in FP64 with one iteration after the other; (W, P, C, iterations, h)."""
    W, P, C = W.double(), P.double(), C.double()
    T, G = W.shape
    a = float(np.float32(ALPHA))
    h, t = 0.0, 0
    while t < iters:
        t += 1
        R = _tan(P @ W, P.square().sum(1), W.square().sum(0))
        A = _tan(W @ C, W.square().sum(1), C.square().sum(0))
        Wn = (1.0 - a) * W + 0.5 * a * (R + A)
        del R, A
        h = float((Wn - W).abs().mean())
        W = Wn
        r, c = W.square().sum(1), W.square().sum(0)
        P = _eq5_eq6(P, _tan(W @ W.T, r, r), a, float(G), t)
        C = _eq5_eq6(C, _tan(W.T @ W, c, c), a, float(T), t)
        if tol is not None and h < tol:
            break
    return W, P, C, t, h


def exact(case, seed):
    kind = case["kind"]
    if kind == "static":
        W, P, C, _, h = _iterate(*_networks(case["T"], case["G"], False, seed), 1)
        return {"W": W, "P": P, "C": C, "h": h}
    if kind == "run":
        T, G = case["T"], case["G"]
        nets = _networks(T, G, case["identity"], seed)
        W, P, C, n, _ = _iterate(*nets, *((case["iters"],) if case["iters"] else (MAX_ITER, TOL)))
        return {"W": W, "P": P, "C": C, "iterations": n}
    if kind == "set":
        outs, its = [], []
        for k, (T, G) in enumerate(_set_sizes(case)):
            W, P, C, n, _ = _iterate(*_networks(T, G, False, seed, k), case["iters"])
            outs.append([W, P, C])
            its.append(n)
        return {"networks": outs, "iterations": its}
    W, P, X = (x.double() for x in _raw_program(case, seed))
    X = X - X.mean(1, keepdim=True)
    X = X / X.norm(dim=1, keepdim=True)
    C = X @ X.T
    C.fill_diagonal_(1.0)

    def z(Y):
        Y = Y - Y.mean()
        return Y / Y.square().mean().sqrt()

    W, P, C, n, _ = _iterate(z(W), z(P), z(C), case["iters"])
    return {"W": W, "P": P, "C": C, "iterations": n}
