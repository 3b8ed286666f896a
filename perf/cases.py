"""Workloads of the library as a user's program runs them, for timing and for comparing outputs.

Every case is one call (for the cost model, one training step) of the public
binding `paper_1609_01490_gb300.tri` on inputs that already live on the GPU.
Sizes are those of the repository's tests and benchmark, or generic odd ones.
"""
from __future__ import annotations

import math

import torch

from paper_1609_01490_gb300 import inputs, tri

_DEV = "cuda"
_MAPS = {"lambda": tri.MAP_LAMBDA, "bb": tri.MAP_BB, "rb": tri.MAP_RB, "table": tri.MAP_TET_TABLE}
_PREC = {"fp32": tri.FP32, "x3": tri.BF16X3, "x6": tri.BF16X6}
# birth and survival masks: Conway's rule, and HighLife as the rule that is not Conway's
_RULES = {"life": (tri.LIFE_BIRTH, tri.LIFE_SURVIVE), "highlife": ((1 << 3) | (1 << 6), (1 << 2) | (1 << 3))}


def listed():
    return [
        # the paper's own size (Section 5, test 2): a small triangle, where launch and latency count
        {"name": "edm-fp32-n2048-d3", "kind": "edm", "prec": "fp32", "n": 2048, "d": 3, "map": "lambda", "points": "uniform"},
        # low-dimensional points at the library's full size: 8.6 GB of distances
        {"name": "edm-fp32-n65536-d3", "kind": "edm", "prec": "fp32", "n": 65536, "d": 3, "map": "lambda", "points": "uniform"},
        # direct differences of feature vectors, sizes that no tile divides
        {"name": "edm-fp32-n20011-d100", "kind": "edm", "prec": "fp32", "n": 20011, "d": 100, "map": "lambda", "points": "normal"},
        # the headline workload: 65,536 feature vectors with 1% duplicates on tensor cores
        {"name": "edm-x6-n65536-d128", "kind": "edm", "prec": "x6", "n": 65536, "d": 128, "map": "lambda", "points": "normal"},
        # a mid-size odd triangle on tensor cores at the lower precision
        {"name": "edm-x3-n12345-d100", "kind": "edm", "prec": "x3", "n": 12345, "d": 100, "map": "lambda", "points": "normal"},
        # a thousand uneven triangles in one launch, with the tile that the autotuner picks for it
        {"name": "edm-batched-1000-d64", "kind": "batched", "count": 1000, "lo": 64, "hi": 8192, "d": 64, "rho": 16, "reg": 8},
        # one Life step of a full-size grid, the call's default tile
        {"name": "life-step-n16384", "kind": "ca", "n": 16384, "steps": 0, "rho": 16, "map": "lambda", "rule": "life"},
        # the Life workload: 100 steps of the full-size grid
        {"name": "life-run-n16384-s100", "kind": "ca", "n": 16384, "steps": 100, "rho": 32, "map": "lambda", "rule": "life"},
        # collision detection at the benchmark's size, and a smaller odd one in the plane
        {"name": "collide-n65536-3d", "kind": "collide", "n": 65536, "dim": 3, "kappa": 4.0, "map": "lambda"},
        {"name": "collide-n9001-2d", "kind": "collide", "n": 9001, "dim": 2, "kappa": 12.0, "map": "lambda"},
        # triplet energy at the benchmark's size
        {"name": "at-n1536-rho32", "kind": "at", "n": 1536, "rho": 32, "map": "table"},
        # one training step (gradient and Adam) of the cost model on the size of its sweep
        {"name": "cost-model-step-b391", "kind": "mlp", "batch": 391, "h1": 64, "h2": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp32-low", "fp32-high", "x6", "x3", "batched", "step", "run", "collide", "at", "mlp"])
    two_d = rng.choice(["lambda", "lambda", "rb", "bb"])
    if kind == "fp32-low":
        return {"kind": "edm", "prec": "fp32", "n": _log_int(rng, 700, 65536), "d": rng.randint(1, 8), "map": two_d,
                "points": "uniform"}
    if kind == "fp32-high":
        return {"kind": "edm", "prec": "fp32", "n": _log_int(rng, 700, 30000), "d": _log_int(rng, 16, 128), "map": two_d,
                "points": "normal"}
    if kind in ("x6", "x3"):
        return {"kind": "edm", "prec": kind, "n": _log_int(rng, 700, 60000), "d": rng.randint(32, 192 if kind == "x6" else 256),
                "map": rng.choice(["lambda", "lambda", "bb"]), "points": "normal"}
    if kind == "batched":
        hi = _log_int(rng, 512, 8192)
        return {"kind": "batched", "count": _log_int(rng, 10, 800), "lo": rng.randint(20, 100), "hi": hi,
                "d": rng.choice([3, 17, 32, 48, 64]), "rho": 16, "reg": rng.choice([0, 8])}
    if kind == "step":
        return {"kind": "ca", "n": _log_int(rng, 900, 30000), "steps": 0, "rho": rng.choice([16, 32]), "map": two_d,
                "rule": rng.choice(["life", "life", "highlife"])}
    if kind == "run":
        return {"kind": "ca", "n": _log_int(rng, 300, 16384), "steps": rng.randint(2, 100), "rho": 32, "map": two_d, "rule": "life"}
    if kind == "collide":
        return {"kind": "collide", "n": _log_int(rng, 1000, 65536), "dim": rng.randint(1, 3), "kappa": rng.choice([4.0, 8.0, 12.0]),
                "map": two_d}
    if kind == "at":
        return {"kind": "at", "n": _log_int(rng, 200, 1536), "rho": rng.choice([16, 32]), "map": rng.choice(["table", "lambda"])}
    return {"kind": "mlp", "batch": _log_int(rng, 64, 2048), "h1": rng.choice([32, 64, 128]), "h2": rng.choice([32, 64, 96])}


# -------------------------------------------------------------------- inputs --
def _gen(seed):
    return torch.Generator(device=_DEV).manual_seed(seed)


def _points(case, seed):
    """U[0,1)^d, or N(0,1) feature vectors of which 1% are copies of other rows (exact-zero distances)."""
    g, n, d = _gen(seed), case["n"], case["d"]
    if case["points"] == "uniform":
        return torch.rand(n, d, generator=g, device=_DEV)
    x = torch.randn(n, d, generator=g, device=_DEV)
    ndup = n // 100
    order = torch.randperm(n, generator=g, device=_DEV)
    x[order[:ndup]] = x[order[ndup:2 * ndup]]
    return x


def _sizes(case):
    """Instance sizes floor(exp(U(ln lo, ln hi))): part of the workload, the same for every seed."""
    return inputs.batched_sizes(case["count"], case["lo"], case["hi"])


def _batch(case, seed):
    """The sizes and N(0,1) points of every instance, concatenated."""
    n_k = torch.from_numpy(_sizes(case)).to(_DEV)
    return n_k, torch.randn(int(n_k.sum()), case["d"], generator=_gen(seed), device=_DEV)


def _spheres(case, seed):
    """Centres U[0,1)^dim, radii U[0, a) with about kappa contacts per sphere (Section 5, test 3)."""
    g, n, dim, kappa = _gen(seed), case["n"], case["dim"], case["kappa"]
    if dim == 1:
        a = kappa / (2.0 * (n - 1))
    elif dim == 2:
        a = math.sqrt(kappa / ((n - 1) * math.pi * 7.0 / 6.0))
    else:
        a = (kappa / ((n - 1) * (4.0 / 3.0) * math.pi * 1.5)) ** (1.0 / 3.0)
    return torch.rand(n, dim, generator=g, device=_DEV), torch.rand(n, generator=g, device=_DEV) * a


def _at_points(case, seed):
    """Unit density: n points in [0, n^(1/3))^3."""
    return torch.rand(case["n"], 3, generator=_gen(seed), device=_DEV) * case["n"] ** (1.0 / 3.0)


_F = tri.SELECT_FEATURES


def _mlp_state(case, seed):
    """Standardised features, targets, and a network and Adam moments in the middle of a training run."""
    g, B, h1, h2 = _gen(seed), case["batch"], case["h1"], case["h2"]
    def draw(*shape):
        return torch.randn(*shape, generator=g, device=_DEV)
    theta = torch.cat([draw(h1 * _F) * (2.0 / _F) ** 0.5, draw(h1) * 0.1, draw(h2 * h1) * (2.0 / h1) ** 0.5, draw(h2) * 0.1,
                       draw(h2) * (2.0 / h2) ** 0.5, draw(1) * 0.1])
    return theta, draw(B, _F), draw(B), draw(theta.numel()) * 0.05, draw(theta.numel()).square() * 0.01 + 1e-3


_ADAM = {"t": 50, "lr": 1e-3, "beta1": 0.9, "beta2": 0.999, "eps": 1e-8}


def _tri_count(n):
    return n * (n + 1) // 2


def prepare(case, seed):
    s = dict(case)
    kind = case["kind"]
    if kind == "edm":
        n, d = case["n"], case["d"]
        s["x"] = _points(case, seed)
        s["out"] = torch.zeros(_tri_count(n), device=_DEV)
        nbytes = tri.tri_edm_workspace_size(n, d, _PREC[case["prec"]])
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device=_DEV) if nbytes else None
    elif kind == "batched":
        n_k, s["x"] = _batch(case, seed)
        pairs = n_k * (n_k + 1) // 2
        s["pt_off"] = n_k.cumsum(0) - n_k
        s["out_off"] = pairs.cumsum(0) - pairs
        s["n_k"] = n_k.to(torch.int32)
        s["out"] = torch.zeros(int(pairs.sum()), device=_DEV)
        s["ws"] = torch.empty(tri.tri_edm_batched_workspace_size(case["count"]), dtype=torch.uint8, device=_DEV)
    elif kind == "ca":
        n = case["n"]
        ld = (n + 15) // 16 * 16
        s["grid"] = torch.randint(0, 2, (n, ld), generator=_gen(seed), device=_DEV, dtype=torch.uint8).tril_()
        s["out"] = torch.zeros_like(s["grid"])
        s["scratch"] = torch.zeros_like(s["grid"]) if case["steps"] > 1 else None
    elif kind == "collide":
        s["c"], s["r"] = _spheres(case, seed)
        s["n_pairs"] = torch.zeros(1, dtype=torch.int64, device=_DEV)
        s["count"] = torch.zeros(case["n"], dtype=torch.int32, device=_DEV)
    elif kind == "at":
        s["p"] = _at_points(case, seed)
        s["energy"] = torch.zeros(1, dtype=torch.float64, device=_DEV)
        nbytes = tri.tet_at_workspace_size(case["n"], case["rho"], _MAPS[case["map"]])
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device=_DEV)
    else:
        s["theta"], s["X"], s["y"], s["m"], s["v"] = _mlp_state(case, seed)
        s["grad"], s["loss"] = torch.zeros_like(s["theta"]), torch.zeros(1, device=_DEV)
        nbytes = tri.tri_mlp_workspace_size(case["batch"], case["h1"], case["h2"])
        s["ws"] = torch.empty(nbytes, dtype=torch.uint8, device=_DEV)
    return s


# ----------------------------------------------------------------------- run --
def run(s):
    kind = s["kind"]
    if kind == "edm":
        tri.tri_edm(s["x"], s["out"], map=_MAPS[s["map"]], prec=_PREC[s["prec"]], workspace=s["ws"])
        return s["out"]
    if kind == "batched":
        tri.tri_edm_batched(s["x"], s["pt_off"], s["n_k"], s["out"], s["out_off"], rho=s["rho"], reg=s["reg"], workspace=s["ws"])
        return s["out"]
    if kind == "ca":
        birth, survive = _RULES[s["rule"]]
        if s["steps"]:
            tri.tri_ca_run(s["grid"], s["out"], s["n"], s["steps"], scratch=s["scratch"], birth_mask=birth,
                           survive_mask=survive, map=_MAPS[s["map"]], rho=s["rho"])
        else:
            tri.tri_ca_step(s["grid"], s["out"], s["n"], birth_mask=birth, survive_mask=survive, map=_MAPS[s["map"]],
                            rho=s["rho"])
        return s["out"]
    if kind == "collide":
        # the pair list comes in no particular order: the counts are what can be compared
        tri.tri_collide(s["c"], s["r"], s["n_pairs"], count=s["count"], map=_MAPS[s["map"]])
        return {"n_pairs": s["n_pairs"], "count": s["count"]}
    if kind == "at":
        tri.tet_at_energy(s["p"], s["energy"], map=_MAPS[s["map"]], rho=s["rho"], workspace=s["ws"])
        return s["energy"]
    tri.tri_mlp_grad(s["theta"], s["X"], s["y"], s["loss"], s["grad"], s["h1"], s["h2"], s["ws"])
    tri.tri_mlp_adam(s["theta"], s["grad"], s["m"], s["v"], **_ADAM)
    return {"loss": s["loss"], "grad": s["grad"], "theta": s["theta"], "m": s["m"], "v": s["v"]}


# ---------------------------------------------------------------------- work --
def work(case):
    kind = case["kind"]
    if kind == "edm":
        n, d = case["n"], case["d"]
        # direct differences: subtract, multiply, add; tensor cores: the inner product
        return {"bytes": 4 * (_tri_count(n) + n * d), "flops": _tri_count(n) * d * (3 if case["prec"] == "fp32" else 2)}
    if kind == "batched":
        sizes = _sizes(case)
        pairs, points = int((sizes * (sizes + 1) // 2).sum()), int(sizes.sum())
        return {"bytes": 4 * (pairs + points * case["d"]), "flops": 3 * pairs * case["d"]}
    if kind == "ca":
        # a step: the eight neighbours' sum and the rule, ten operations on words of 32 cells
        cells = _tri_count(case["n"])
        return {"bytes": 2 * cells, "flops": 10 * max(1, case["steps"]) * cells / 32}
    if kind == "collide":
        n, dim = case["n"], case["dim"]
        return {"bytes": 4 * n * (dim + 2) + 8, "flops": (3 * dim + 1) * n * (n - 1) / 2}
    if kind == "at":
        n = case["n"]
        return {"bytes": 12 * n + 8, "flops": 40 * n * (n - 1) * (n - 2) / 6}
    B, h1, h2 = case["batch"], case["h1"], case["h2"]
    params = h1 * _F + h1 + h2 * h1 + 2 * h2 + 1
    return {"bytes": 4 * (B * (_F + 1) + 8 * params), "flops": 6 * B * params}


# --------------------------------------------------------------------- exact --
def _distances(x, out, rows=1024):
    """Packed lower triangle of Euclidean distances by direct differences, in 64 bits."""
    n, d = x.shape
    xt = x.double().t().contiguous()
    for r0 in range(0, n, rows):
        r1 = min(n, r0 + rows)
        acc = torch.zeros(r1 - r0, r1, dtype=torch.float64, device=x.device)
        diff = torch.empty_like(acc)
        for k in range(d):
            torch.sub(xt[k, r0:r1, None], xt[k, None, :r1], out=diff)
            acc.addcmul_(diff, diff)
        keep = torch.ones_like(acc, dtype=torch.bool).tril_(r0)
        out[_tri_count(r0):_tri_count(r1)] = acc.sqrt_()[keep]


def _axilrod_teller(p):
    """Sum over i > j > k of (1 + 3 cos cos cos) / (r_ij r_jk r_ki)^3, one i at a time."""
    p = p.double()
    d2 = (p[:, None, :] - p[None, :, :]).square().sum(-1)
    total = torch.zeros((), dtype=torch.float64, device=p.device)
    for i in range(2, p.shape[0]):
        c = d2[i, :i]
        a, b = c[:, None], d2[:i, :i]
        c = c[None, :]
        q = a * b * c
        term = (1 + 0.375 * (a + c - b) * (a + b - c) * (b + c - a) / q) / (q * q.sqrt())
        total += torch.where(torch.ones_like(b, dtype=torch.bool).tril_(-1), term, torch.zeros_like(term)).sum()
    return total.reshape(1)


def _training_step(case, seed):
    theta, X, y, m, v = (t.double() for t in _mlp_state(case, seed))
    h1, h2 = case["h1"], case["h2"]
    theta.requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(theta, [h1 * _F, h1, h2 * h1, h2, h2, 1])
    z = torch.relu(X @ W1.view(h1, _F).t() + b1)
    z = torch.relu(z @ W2.view(h2, h1).t() + b2)
    loss = (z @ W3 + b3 - y).square().mean()
    (g,) = torch.autograd.grad(loss, theta)
    b1, b2 = _ADAM["beta1"], _ADAM["beta2"]
    m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
    step = (m / (1 - b1 ** _ADAM["t"])) / ((v / (1 - b2 ** _ADAM["t"])).sqrt() + _ADAM["eps"])
    return {"loss": loss.detach().reshape(1), "grad": g, "theta": theta.detach() - _ADAM["lr"] * step, "m": m, "v": v}


def exact(case, seed):
    kind = case["kind"]
    if kind == "edm":
        out = torch.empty(_tri_count(case["n"]), dtype=torch.float64, device=_DEV)
        _distances(_points(case, seed), out)
        return out
    if kind == "batched":
        n_k, x = _batch(case, seed)
        sizes = n_k.tolist()
        out = torch.empty(sum(_tri_count(n) for n in sizes), dtype=torch.float64, device=_DEV)
        p = o = 0
        for n in sizes:
            _distances(x[p:p + n], out[o:o + _tri_count(n)], rows=4096)
            p, o = p + n, o + _tri_count(n)
        return out
    if kind == "at":
        return _axilrod_teller(_at_points(case, seed))
    if kind == "mlp":
        return _training_step(case, seed)
    return None  # cells and contact counts are whole numbers
