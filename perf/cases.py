"""The work that a user of this package has it do, as cases that can be timed.

A case names one public entry point, a size and the options it is called with.
Bodies are the package's own workloads: Plummer spheres (one, two on an
approach, or a batch of uneven ones), G = 1.

The float32 modes, the tree code and the fast multipole method compute their
pair terms in float32 and hand the sums back in float64 arrays; a program that
picks them keeps accelerations and gradients in float32, and so do the cases.
The float64 and double-float modes' accelerations, and every integrated state
(which is float64 in each mode), stay float64.
"""
import math

import torch

from paper_1211_2292_gb300 import inputs, nbody, tune
from paper_1211_2292_gb300.autograd import rollout

G = 1.0
DEV = "cuda"


def listed():
    return [
        # one force evaluation of a small cluster: the latency of a call
        {"name": "force_1k", "kind": "force", "prec": "fp32_comp", "n": 1000, "eps": 0.01},
        # a simulation's inner loop at a few thousand bodies: leapfrog steps in one graph
        {"name": "step_4k", "kind": "step", "prec": "fp32_comp", "n": 4096, "eps": 0.01, "steps": 8},
        # a mid-sized system in the plain float32 mode, of ragged size
        {"name": "force_16k_plain", "kind": "force", "prec": "fp32", "n": 16411, "eps": 0.01},
        # a large direct sum, in Morton order: the two-sphere workload of the benchmark
        {"name": "force_256k", "kind": "force", "prec": "fp32_comp", "n": 262144, "eps": 0.002},
        # the float64 mode, which a run's accuracy is checked with, of ragged size
        {"name": "force_4k_fp64", "kind": "force", "prec": "fp64", "n": 4097, "eps": 0.01},
        # float64 accuracy at a mid size
        {"name": "force_16k_df64", "kind": "force", "prec": "df64", "n": 16384, "eps": 0.005},
        # many uneven systems in one launch: the benchmark's batch
        {"name": "batch_512", "kind": "batch", "prec": "fp32_comp", "nsys": 512, "lo": 64,
         "hi": 8192, "eps": 0.01},
        # a training step: rollout, loss and gradients at the differentiation workload's size
        {"name": "grad_16k", "kind": "grad", "prec": "fp32_comp", "n": 16384, "eps": 0.01,
         "steps": 4, "every": 2},
        # tree code on a small system, steps in one graph: the rebuild counts
        {"name": "tree_step_20k", "kind": "tree_step", "prec": "fp32_comp", "n": 20000, "eps": 0.01,
         "theta": 0.5, "leaf": 16, "group": 64, "steps": 4},
        # tree code at the benchmark's size
        {"name": "tree_1m", "kind": "tree", "prec": "fp32_comp", "n": 1048576, "eps": 0.002,
         "theta": 0.5, "leaf": 16, "group": 64},
        # fast multipole method on a small system of ragged size, lower order
        {"name": "fmm_30k", "kind": "fmm", "prec": "fp32_comp", "n": 30001, "eps": 0.005,
         "theta": 0.6, "order": 4, "leaf": 32},
        # fast multipole method at the benchmark's size
        {"name": "fmm_1m", "kind": "fmm", "prec": "fp32_comp", "n": 1048576, "eps": 0.002,
         "theta": 0.6, "order": 6, "leaf": 64},
    ]


def _size(rng, lo, hi):
    """A size in [lo, hi], spread over its logarithm; odd ones among them."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(["force", "force", "step", "batch", "grad", "tree", "tree_step", "fmm"])
    eps = rng.choice([0.002, 0.005, 0.01, 0.02])
    prec = rng.choice(["fp32_comp", "fp32_comp", "fp32"])
    if kind == "force":
        prec = rng.choice(["fp32_comp", "fp32_comp", "fp32", "fp64", "df64"])
        hi = {"fp64": 8192, "df64": 65536}.get(prec, 262144)
        return {"kind": kind, "prec": prec, "n": _size(rng, 64, hi), "eps": eps}
    if kind == "step":
        return {"kind": kind, "prec": prec, "n": _size(rng, 256, 32768), "eps": 0.01,
                "steps": rng.randint(1, 8)}
    if kind == "batch":
        lo = _size(rng, 16, 512)
        return {"kind": kind, "prec": prec, "nsys": _size(rng, 8, 512), "lo": lo,
                "hi": _size(rng, lo, 8192), "eps": 0.01}
    if kind == "grad":
        return {"kind": kind, "prec": prec, "n": _size(rng, 256, 16384), "eps": 0.01,
                "steps": rng.randint(1, 6), "every": rng.randint(1, 4)}
    theta, group = rng.choice([0.4, 0.5, 0.6, 0.7]), rng.choice([32, 64])
    if kind == "tree":
        return {"kind": kind, "prec": prec, "n": _size(rng, 2000, 1000000), "eps": eps,
                "theta": max(theta, 0.5), "leaf": rng.choice([8, 16, 32]), "group": group}
    if kind == "tree_step":
        return {"kind": kind, "prec": prec, "n": _size(rng, 2000, 100000), "eps": 0.01,
                "theta": theta, "leaf": rng.choice([8, 16, 32]), "group": group,
                "steps": rng.randint(1, 6)}
    return {"kind": kind, "prec": prec, "n": _size(rng, 3000, 1000000), "eps": eps,
            "theta": max(theta, 0.5), "order": rng.randint(3, 6), "leaf": rng.choice([32, 64])}


DT = 2.5e-4  # a step well inside the shortest orbit's period at these softenings


def _batch_sizes(case):
    """The sizes of a batch's systems, which belong to the case."""
    return inputs.batch_sizes(case["nsys"], case["lo"], case["hi"])


def _bodies(case, seed):
    """The case's bodies: two spheres for the large systems, else one."""
    if case["kind"] == "batch":
        return inputs.plummer_batch(sizes=_batch_sizes(case), seed=seed)
    n = case["n"]
    if n >= 131072:
        b = inputs.two_plummer((n + 1) // 2, seed=seed)
        return inputs.Bodies(b.pos[:n], b.vel[:n], b.mass[:n]), None
    return inputs.plummer(n, seed=seed), None


def _host(case, seed):
    """Host inputs; a training step's parameters are float32."""
    b, offsets = _bodies(case, seed)
    x, v, m = (torch.as_tensor(a, dtype=torch.float64).contiguous() for a in (b.pos, b.vel, b.mass))
    if case["kind"] == "grad":
        g = torch.Generator().manual_seed(seed)
        target = x + 1e-3 * torch.randn(x.shape, generator=g, dtype=torch.float64)
        return [t.float() for t in (x, v, m)] + [target], offsets
    return [x, v, m], offsets


def prepare(case, seed):
    arrays, offsets = _host(case, seed)
    arrays = [a.to(DEV) for a in arrays]
    s = {"case": case, "x": arrays[0], "v": arrays[1], "m": arrays[2]}
    nb = s["nb"] = nbody.NBody(arrays[2].shape[0], case["prec"])
    tune.apply(nb)
    kind, eps = case["kind"], case["eps"]
    if kind == "batch":
        nb.batch_plan(offsets)
    elif kind == "grad":
        s["target"] = arrays[3]
        for k in ("x", "v", "m"):
            s[k].requires_grad_()
    elif kind == "step":  # the force at the start, which a stepping loop carries along
        s["acc"] = nb.forces(s["x"], s["m"], G, eps)
    elif kind == "tree_step":
        s["acc"] = nb.tree_forces(s["x"], s["m"], G, eps, case["theta"], case["leaf"],
                                  group=case["group"])
    return s


def run(s):
    c, nb, x, v, m = s["case"], s["nb"], s["x"], s["v"], s["m"]
    kind, eps = c["kind"], c["eps"]
    if kind == "force":
        acc = nb.forces(x, m, G, eps)
        return acc if c["prec"] in ("fp64", "df64") else acc.float()
    if kind == "step":
        nb.step(x, v, m, G, eps, DT, c["steps"], s["acc"], acc_valid=True, graph=True)
        return x, v, s["acc"].float()
    if kind == "batch":
        return nb.forces_batched(x, m, G, eps).float()
    if kind == "grad":
        xe, ve = rollout(nb, x.double(), v.double(), m.double(), G, eps, 2 * DT, c["steps"],
                         c["every"])
        loss = (xe - s["target"]).square().sum(1).mean()
        return [xe.detach(), ve.detach(), loss.detach().float(),
                *torch.autograd.grad(loss, (x, v, m))]
    if kind == "tree":
        return nb.tree_forces(x, m, G, eps, c["theta"], c["leaf"], group=c["group"]).float()
    if kind == "tree_step":
        nb.tree_step(x, v, m, G, eps, c["theta"], c["leaf"], DT, c["steps"], s["acc"],
                     acc_valid=True, graph=True, group=c["group"])
        return x, v, s["acc"].float()
    return nb.fmm_forces(x, m, G, eps, c["theta"], c["order"], c["leaf"]).float()


def work(case):
    """20 flops per pair (the field's convention), 54 per pair of the force's
    gradient (its 26 float32 multiply-adds, and 2 for the product with the
    total), and the arrays of the call read and written once."""
    kind = case["kind"]
    if kind == "batch":
        sizes = [int(k) for k in _batch_sizes(case)]
        return {"bytes": 44 * sum(sizes), "flops": 20 * sum(k * k for k in sizes)}
    n = case["n"]
    if kind == "force":
        return {"bytes": (56 if case["prec"] in ("fp64", "df64") else 44) * n, "flops": 20 * n * n}
    if kind == "step":
        return {"bytes": 92 * n + 48 * n, "flops": 20 * n * n * case["steps"]}
    if kind == "grad":
        # forward, and backward with every position but the segments' ends evaluated again
        k = case["steps"]
        return {"bytes": 156 * n, "flops": n * n * (20 * (k + 1) + 54 * (k + 1))}
    if kind in ("tree", "tree_step"):
        # bodies and cells on a body's list: about 5700 at 2^20 bodies, theta 0.5, groups of 64
        theta = case["theta"] or 0.5
        inter = min(n, 290 * math.log2(n) * (0.5 / theta) ** 2)
        k = case.get("steps", 1)
        return {"bytes": (44 if kind == "tree" else 140) * n, "flops": 20 * n * inter * k}
    # expansions' multiply-adds and direct pairs, per body about 58 000 + 46 000 flops at
    # theta 0.6, order 6, leaves of up to 64
    p = case["order"]
    terms = math.comb(p + 6, 6) / math.comb(12, 6)
    leaf = case["leaf"] / 64
    return {"bytes": 44 * n, "flops": n * (0.6 / case["theta"]) ** 3 * (58000 * terms / leaf
                                                                        + 46000 * leaf)}


# ------------------------------------------------- the same in 64 bits, in plain torch
def _rows(n):
    return max(1, min(n, (1 << 27) // n))


def _force64(x, m, eps):
    n = x.shape[0]
    acc = torch.empty_like(x)
    for i in range(0, n, _rows(n)):
        d = [x[None, :, c] - x[i:i + _rows(n), c, None] for c in range(3)]
        w = d[0].square().addcmul_(d[1], d[1]).addcmul_(d[2], d[2]).add_(eps * eps).rsqrt_()
        w = w * w * w * m
        for c in range(3):
            acc[i:i + _rows(n), c] = (w * d[c]).sum(1)
    return acc.mul_(G)


class _Force(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, m, eps):
        ctx.save_for_backward(x, m)
        ctx.eps = eps
        return _force64(x, m, eps)

    @staticmethod
    def backward(ctx, lam):
        (x, m), n = ctx.saved_tensors, lam.shape[0]
        gx, gm = torch.zeros_like(x), torch.empty_like(m)
        for i in range(0, n, _rows(n)):
            k = slice(i, i + _rows(n))  # the bodies whose gradients are summed, against all j
            d = [x[None, :, c] - x[k, c, None] for c in range(3)]
            r = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + ctx.eps ** 2).rsqrt_()
            r3 = r * r * r
            w = [m[k, None] * lam[None, :, c] - m[None, :] * lam[k, c, None] for c in range(3)]
            dw = (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * r3 * r * r * 3
            for c in range(3):
                gx[k, c] = (w[c] * r3 - dw * d[c]).sum(1) * G
            dl = d[0] * lam[None, :, 0] + d[1] * lam[None, :, 1] + d[2] * lam[None, :, 2]
            gm[k] = -(dl * r3).sum(1) * G
        return gx, gm, None


def _leapfrog(x, v, m, acc, eps, dt, steps):
    for _ in range(steps):
        v = v + 0.5 * dt * acc
        x = x + dt * v
        acc = _Force.apply(x, m, eps)
        v = v + 0.5 * dt * acc
    return x, v, acc


def exact(case, seed):
    """What run() returns on a new state; the sums over all pairs also where
    the call approximates them.  None above 2^18 bodies."""
    kind, eps = case["kind"], case["eps"]
    if kind != "batch" and case["n"] > 262144:
        return None
    arrays, offsets = _host(case, seed)
    x, v, m = (a.to(DEV).double() for a in arrays[:3])
    if kind == "batch":
        out = torch.empty_like(x)
        for a, b in zip(offsets[:-1], offsets[1:]):
            out[a:b] = _force64(x[a:b], m[a:b], eps)
        return out
    if kind in ("step", "tree_step"):
        return _leapfrog(x, v, m, _force64(x, m, eps), eps, DT, case["steps"])
    if kind == "grad":
        for t in (x, v, m):
            t.requires_grad_()
        xe, ve, _ = _leapfrog(x, v, m, _Force.apply(x, m, eps), eps, 2 * DT, case["steps"])
        loss = (xe - arrays[3].to(DEV)).square().sum(1).mean()
        return [xe.detach(), ve.detach(), loss.detach(), *torch.autograd.grad(loss, (x, v, m))]
    return _force64(x, m, eps)
