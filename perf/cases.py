"""Measured cases of the library: what a program that evaluates Boys functions
has it do, through the package's public calls.

Arguments are synthetic, in the laws of ``workloads.py`` and drawn on the GPU:

* ``parity``  90% log-uniform on [1e-8, 1e3], 5% zeros, 5% within 1e-12 of the
              two region boundaries (most arguments in region A);
* ``eri``     40% log-uniform on [1e-12, 1e2], 40% uniform on [0, 60],
              20% uniform on [60, 1e4] (all three regions in earnest);
* ``log``     log-uniform on [1e-10, 1e3].

A case is {"op", sizes, options}; ``op`` is one of

* ``eval``     boys_eval into the caller's buffer (FP64, order-major);
* ``f32``      boys_eval_f32 into the caller's buffer (FP32 tier);
* ``host``     boys_eval_host on pinned host buffers;
* ``fused``    boys_eval_fused (sum_k (-2 rho)^k F_k, one value per argument);
* ``grad``     boys() and its backward: F and dL/dx;
* ``ragged``   a batch of segments with a kmax each: boys_eval_ragged on the
               caller's output and workspace, or a RaggedPlan's launch;
* ``pairwise`` boys_pairwise (z_i = sum_l c_l sum_j F_l(x_i + x_j) y_j).
"""
import math

import torch

import paper_2512_10059_gb300 as boys
from paper_2512_10059_gb300 import workloads as W

DEV = "cuda:0"


def listed():
    return [
        # one batch of integrals as a direct SCF code hands it over: latency
        {"name": "eval_k4_n1000", "op": "eval", "kmax": 4, "n": 1000, "law": "parity"},
        # the parity workload's size: a batch of p/d shell quartets
        {"name": "eval_k8_n65536", "op": "eval", "kmax": 8, "n": 65536, "law": "parity"},
        # a middle batch of an odd size (odd row stride), first derivatives of f shells
        {"name": "eval_k16_n1000003", "op": "eval", "kmax": 16, "n": 1000003, "law": "eri"},
        # low angular momentum in bulk, the commonest kmax of a basis set
        {"name": "eval_k4_n2p25", "op": "eval", "kmax": 4, "n": 1 << 25, "law": "parity"},
        # the headline: every order up to 32, 17.7 GB written
        {"name": "eval_k32_n2p26", "op": "eval", "kmax": 32, "n": 1 << 26, "law": "eri"},
        # McMurchie-Davidson scaling consumed at once, nothing stored but the sum
        {"name": "fused_k32_n2p24", "op": "fused", "kmax": 32, "n": 1 << 24, "law": "eri"},
        # a differentiated call: forward and backward
        {"name": "grad_k16_n2p23", "op": "grad", "kmax": 16, "n": 1 << 23, "law": "log"},
        # shell quartets of mixed angular momentum, a new batch each time
        {"name": "ragged_4096seg", "op": "ragged", "nseg": 4096, "min_len": 32, "max_len": 65536, "plan": False},
        # a smaller batch whose plan a program keeps and replays
        {"name": "ragged_plan_512seg", "op": "ragged", "nseg": 512, "min_len": 32, "max_len": 4096, "plan": True},
        # the single-precision tier in bulk (screening, guesses)
        {"name": "f32_k12_n2p26", "op": "f32", "kmax": 12, "n": 1 << 26, "law": "parity"},
        # the paper's Algorithm 2 at its k, arguments sorted
        {"name": "pairwise_k12_n65536", "op": "pairwise", "k": 12, "n": 65536, "sort": True},
        # arguments and results in the caller's pinned host buffers
        {"name": "host_k8_n2p20", "op": "host", "kmax": 8, "n": 1 << 20, "law": "parity"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["eval"] * 6 + ["fused"] * 2 + ["grad"] * 2 + ["ragged"] * 4 + ["f32", "pairwise", "host"])
    law = rng.choice(["parity", "eri"])
    if op == "eval":
        kmax = rng.randint(0, 32)
        n = min(_log_int(rng, 500, 1 << 26), (33 << 26) // (kmax + 1))
        return {"op": op, "kmax": kmax, "n": n, "law": law}
    if op == "f32":
        return {"op": op, "kmax": rng.randint(0, 32), "n": _log_int(rng, 1000, 1 << 25), "law": law}
    if op == "host":
        return {"op": op, "kmax": rng.randint(0, 12), "n": _log_int(rng, 1000, 1 << 20), "law": law}
    if op == "fused":
        return {"op": op, "kmax": rng.randint(2, 32), "n": _log_int(rng, 1000, 1 << 24), "law": law}
    if op == "grad":
        return {"op": op, "kmax": rng.randint(1, 24), "n": _log_int(rng, 1000, 1 << 22), "law": rng.choice(["log", "eri"])}
    if op == "ragged":
        return {"op": op, "nseg": _log_int(rng, 16, 4096), "min_len": rng.randint(1, 64),
                "max_len": _log_int(rng, 256, 65536), "plan": rng.random() < 0.4}
    return {"op": op, "k": rng.randint(2, 20), "n": _log_int(rng, 500, 30000), "sort": rng.random() < 0.7}


# ------------------------------------------------------------------- inputs

def _gen(seed, dev=DEV):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    return g


def _uniform(n, g, dev=DEV):
    return torch.rand(n, dtype=torch.float64, device=dev, generator=g)


def _log_uniform(u, lo, hi):
    return torch.exp(math.log(lo) + u * (math.log(hi) - math.log(lo)))


def _arguments(law, n, g):
    u = _uniform(n, g)
    if law == "log":
        return _log_uniform(u, 1e-10, 1e3)
    c = _uniform(n, g)
    if law == "parity":
        edge = W.X0_PRINTED + (W.X1_PRINTED - W.X0_PRINTED) * (c < 0.975).double()
        near = edge + (2.0 * u - 1.0) * 1e-12
        return torch.where(c < 0.90, _log_uniform(u, 1e-8, 1e3), torch.where(c < 0.95, torch.zeros_like(u), near))
    return torch.where(c < 0.4, _log_uniform(u, 1e-12, 1e2), torch.where(c < 0.8, 60.0 * u, 60.0 + (1e4 - 60.0) * u))


def _segments(case, seed):
    """Lengths and kmax of the segments, on the host: one set of segments a
    case (so that every batch has the same sizes in all), in an order of the seed."""
    g = _gen(case["nseg"], "cpu")
    u = torch.rand(case["nseg"], dtype=torch.float64, generator=g)
    lens = _log_uniform(u, case["min_len"], case["max_len"] + 1).floor().long()
    lens = lens.clamp(case["min_len"], case["max_len"])
    p = torch.tensor([0.40, 0.30, 0.20, 0.08, 0.02])
    kmax = torch.multinomial(p.expand(case["nseg"], 5), 4, replacement=True, generator=g).sum(1)
    order = torch.randperm(case["nseg"], generator=_gen(seed, "cpu"))
    return lens[order], kmax.int()[order]


def _inputs(case, seed):
    """The tensors that the call reads, from the seed alone."""
    g, op = _gen(seed), case["op"]
    if op == "ragged":
        lens, kmax = _segments(case, seed)
        off = torch.zeros(case["nseg"] + 1, dtype=torch.int64)
        off[1:] = torch.cumsum(lens, 0)
        return {"x": _arguments("parity", int(off[-1]), g), "seg_off": off.to(DEV), "seg_kmax": kmax.to(DEV)}
    if op == "pairwise":
        x = 30.0 * _uniform(case["n"], g)
        x = torch.sort(x).values if case["sort"] else x
        y = torch.randn(case["n"], dtype=torch.float64, device=DEV, generator=g)
        c = torch.randn(case["k"] + 1, dtype=torch.float64, device=DEV, generator=g)
        return {"x": x, "y": y, "c": c}
    x = _arguments(case["law"], case["n"], g)
    if op == "f32":
        return {"x": x.float()}
    if op == "fused":
        return {"x": x, "rho": 0.1 + 9.9 * _uniform(case["n"], g)}
    if op == "grad":
        return {"x": x, "g": torch.randn((case["kmax"] + 1, case["n"]), dtype=torch.float64, device=DEV, generator=g)}
    return {"x": x}


def prepare(case, seed):
    s, op = dict(_inputs(case, seed), op=case["op"]), case["op"]
    if op in ("eval", "f32", "host", "fused", "grad"):
        s["kmax"] = case["kmax"]
    if op in ("eval", "f32"):
        s["out"] = torch.empty((case["kmax"] + 1, case["n"]), dtype=s["x"].dtype, device=DEV)
    elif op == "host":
        s["x"] = s["x"].cpu().pin_memory()
        s["out"] = torch.empty((case["kmax"] + 1, case["n"]), dtype=torch.float64, pin_memory=True)
    elif op == "fused":
        s["out"] = torch.empty_like(s["x"])
    elif op == "grad":
        s["x"].requires_grad_()
    elif op == "ragged":
        lens = s["seg_off"][1:] - s["seg_off"][:-1]
        sizes = (s["seg_kmax"].long() + 1) * lens
        s["out_off"] = (torch.cumsum(sizes, 0) - sizes).contiguous()
        s["out"] = torch.empty(int(sizes.sum()), dtype=torch.float64, device=DEV)
        if case["plan"]:
            s["plan"] = boys.RaggedPlan(s["x"], s["seg_off"], s["seg_kmax"], out=s["out"], out_off=s["out_off"])
    return s


def run(s):
    op = s["op"]
    if op == "eval":
        return boys.boys_eval(s["x"], s["kmax"], out=s["out"])
    if op == "f32":
        return boys.boys_eval_f32(s["x"], s["kmax"], out=s["out"])
    if op == "host":
        return boys.boys_eval_host(s["x"], s["kmax"], out=s["out"])
    if op == "fused":
        return boys.boys_eval_fused(s["x"], s["rho"], s["kmax"], out=s["out"])
    if op == "grad":
        f = boys.boys(s["x"], s["kmax"])
        (dx,) = torch.autograd.grad(f, s["x"], s["g"])
        return {"F": f.detach(), "dx": dx}
    if op == "ragged":
        if "plan" in s:
            return s["plan"].launch()
        return boys.boys_eval_ragged(s["x"], s["seg_off"], s["seg_kmax"], out=s["out"], out_off=s["out_off"])[0]
    return boys.boys_pairwise(s["x"], s["y"], s["c"])


# -------------------------------------------------------------------- work

# flops of one argument: the anchor's rational (about 17 multiply-adds), one
# exponential and three operations an order
def _flops(kmax):
    return 40 + 3 * kmax


def work(case):
    op = case["op"]
    if op == "ragged":
        lens, kmax = _segments(case, 0)
        orders, n = int((lens * (kmax + 1)).sum()), int(lens.sum())
        return {"bytes": 8 * (n + orders) + 20 * case["nseg"], "flops": 40 * n + 3 * orders}
    n = case["n"]
    if op == "pairwise":
        return {"bytes": 24 * n, "flops": n * n * (_flops(case["k"]) + 2 * case["k"])}
    k = case["kmax"]
    if op == "f32":
        return {"bytes": 4 * n * (k + 2), "flops": n * _flops(k)}
    if op == "fused":
        return {"bytes": 24 * n, "flops": n * (_flops(k) + 2 * k)}
    if op == "grad":  # F written; x and g read, dx written
        return {"bytes": 8 * n * (k + 2) + 8 * n * (k + 3), "flops": n * (_flops(k) + _flops(k + 1) + 2 * k)}
    return {"bytes": 8 * n * (k + 2), "flops": n * _flops(k)}


# ------------------------------------------------------------------- exact

def _boys64(x, kmax):
    """F_0..F_kmax(x), [kmax+1, n], in 64 bits from the definition's series:
    x < 30: F_kmax = e^-x sum_i (2x)^i / ((2k+1)(2k+3)...(2k+2i+1)), all terms
    positive, then downward; x >= 30: F_0 = sqrt(pi/x) erf(sqrt(x)) / 2, upward."""
    out = torch.empty((kmax + 1, x.numel()), dtype=torch.float64, device=x.device)
    step = 1 << 24
    for a in range(0, x.numel(), step):
        v = x[a:a + step].double()
        low = torch.clamp(v, max=30.0)
        e, two = torch.exp(-low), 2.0 * low
        term = torch.full_like(low, 1.0 / (2 * kmax + 1))
        total = term.clone()
        for i in range(1, 170):
            term *= two
            term /= 2 * kmax + 2 * i + 1
            total += term
        down = e * total
        high = torch.clamp(v, min=30.0)
        eh = torch.exp(-high)
        up = 0.5 * torch.sqrt(math.pi / high) * torch.erf(torch.sqrt(high))
        small = v < 30.0
        o = out[:, a:a + step]
        o[kmax] = down
        for k in range(kmax - 1, -1, -1):
            down = (two * down + e) / (2 * k + 1)
            o[k] = down
        for k in range(kmax + 1):
            o[k] = torch.where(small, o[k], up)
            up = ((2 * k + 1) * up - eh) / (2.0 * high)
    return out


def exact(case, seed):
    s, op = _inputs(case, seed), case["op"]
    if op in ("eval", "f32"):
        return _boys64(s["x"], case["kmax"])
    if op == "host":
        return _boys64(s["x"], case["kmax"]).cpu()
    if op == "fused":
        total = torch.zeros_like(s["x"])
        for k, f in reversed(list(enumerate(_boys64(s["x"], case["kmax"])))):
            total = f - 2.0 * s["rho"] * total
        return total
    if op == "grad":
        f = _boys64(s["x"], case["kmax"] + 1)
        return {"F": f[:-1], "dx": -(s["g"] * f[1:]).sum(0)}
    if op == "pairwise":
        # F_l(x) = int_0^1 t^2l e^(-x t^2) dt by Gauss-Legendre quadrature (exact to rounding for x <= 60)
        import numpy as np
        t, w = np.polynomial.legendre.leggauss(96)
        t, w = (torch.tensor(v, device=DEV) for v in (0.5 * (t + 1.0), 0.5 * w))
        l = torch.arange(case["k"] + 1, device=DEV)
        cl = (s["c"][None, :] * t[:, None] ** (2 * l)[None, :]).sum(1)
        e = torch.exp(-s["x"][:, None] * (t * t)[None, :])
        return e @ (w * cl * (s["y"] @ e))
    off, kmax = s["seg_off"].tolist(), s["seg_kmax"].tolist()
    parts = {}
    for k in set(kmax):
        segs = [i for i, v in enumerate(kmax) if v == k]
        cat = _boys64(torch.cat([s["x"][off[i]:off[i + 1]] for i in segs]), k)
        a = 0
        for i in segs:
            n = off[i + 1] - off[i]
            parts[i] = cat[:, a:a + n].reshape(-1)
            a += n
    return torch.cat([parts[i] for i in range(len(kmax))])
