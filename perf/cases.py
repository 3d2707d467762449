"""Cases on which the time of this framework is measured, through its public entry points.

A case is one call that a program which rounds weight matrices under two-sided Hessian estimates makes: the set-up
of the feedback factors, the sweep, both for many small layers at once, the objective, and the storage and order
options of the sweep.  Sizes and input statistics are those of the configurations in ``workloads.py`` (64 x 64,
256 x 256, 1024 x 4096, 4096 x 4096, 8192 x 8192; Gaussian samples without and with channel scales, and a geometric
spectrum of condition 1e6), plus ragged sizes between them.  Inputs are made on the GPU from the seed alone.

The mode that computes in 32 bits is not among them: entries within its rounding of a tie fall either way with the
order of its sums, and each moves all that follow (two of its own kernels differ in 6 to 40 % of the integers at
1024 x 1024), so that two correct implementations cannot be told from wrong ones by their integers.
"""
import math

import torch

from paper_2607_27042_b200 import gptq2d as g

F64 = torch.float64


def listed():
    return [
        # one small matrix (the smallest configuration): nothing but launch, start-up and the dependent chain
        {"name": "sweep_64", "op": "sweep", "m": 64, "n": 64, "kind": "scaled", "E": True},
        # one layer of a transformer (down-projection shape), heavy-tailed channels, errors asked for as well
        {"name": "sweep_1024x4096_E", "op": "sweep", "m": 1024, "n": 4096, "kind": "scaled", "E": True},
        # ragged in both directions and odd leading dimensions, as a pruned or split layer gives
        {"name": "sweep_2999x1803_E", "op": "sweep", "m": 2999, "n": 1803, "kind": "scaled", "E": True},
        # a square layer with ill-conditioned Grams
        {"name": "sweep_4096_E", "op": "sweep", "m": 4096, "n": 4096, "kind": "spectrum", "E": True},
        # the largest configuration, integers only
        {"name": "sweep_8192", "op": "sweep", "m": 8192, "n": 8192, "kind": "plain", "E": False},
        # inputs and result in pinned host memory, as when layers are kept on the host and rounded one by one
        {"name": "sweep_host_4096", "op": "sweep_host", "m": 4096, "n": 4096, "kind": "plain", "E": False},
        # X and factors stored in 32 bits, last row and column first: the storage and order options
        {"name": "sweep_f32in_2048x3072_E", "op": "sweep_f32in", "m": 2048, "n": 3072, "kind": "plain", "E": True},
        # 64 heads or experts of one model in one launch, two shapes mixed
        {"name": "sweep_batch_64x256", "op": "sweep_batch", "m": 256, "n": 256, "count": 64, "kind": "scaled", "E": False},
        # their set-up: small bases, one call
        {"name": "setup_batch_128x96", "op": "setup_batch", "m": 96, "n": 96, "count": 128, "kind": "scaled"},
        # the set-up of one layer, ragged
        {"name": "setup_1100x4100", "op": "setup", "m": 1100, "n": 4100, "kind": "scaled"},
        # the set-up of the largest configuration
        {"name": "setup_8192", "op": "setup", "m": 8192, "n": 8192, "kind": "plain"},
        # what a rounding cost, evaluated after it
        {"name": "objective_4096", "op": "objective", "m": 4096, "n": 4096, "kind": "plain"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sweep", "sweep", "sweep", "setup", "setup", "objective", "sweep_host", "sweep_f32in",
                     "sweep_reverse", "sweep_batch", "setup_batch"])
    kind = rng.choice(["plain", "scaled", "spectrum"])
    if op in ("sweep_batch", "setup_batch"):
        m, n = _log(rng, 24, 512 if op == "sweep_batch" else 128), _log(rng, 24, 512 if op == "sweep_batch" else 128)
        c = {"op": op, "m": m, "n": n, "count": min(_log(rng, 4, 256), 2 ** 23 // (m * n)), "kind": kind}
        if op == "sweep_batch":
            c["E"] = rng.random() < 0.5
        return c
    top = 8192 if op in ("sweep", "setup", "objective") else 4096
    c = {"op": op, "m": _log(rng, 48, top), "n": _log(rng, 48, top), "kind": kind}
    if op.startswith("sweep"):
        c["E"] = op != "sweep_host" and rng.random() < 0.5
    return c


def _shapes(case):
    """The shapes of a batch: m x n and m x 2n in turn."""
    return [(case["m"], case["n"] * (1 + b % 2)) for b in range(case["count"])]


def _gram(gen, count, k, kind):
    """count Grams of order k: Gaussian samples with 1 % damping ("plain"), the same with log-normal channel scales
    ("scaled"), or a geometric spectrum of condition 1e6 ("spectrum")."""
    if kind == "spectrum":
        q, _ = torch.linalg.qr(torch.randn(count, k, k, dtype=F64, device="cuda", generator=gen))
        ev = torch.logspace(0, -6, k, dtype=F64, device="cuda")
        s = (q * ev) @ q.mT
    else:
        t = 2 * k
        s = torch.randn(count, k, t, dtype=F64, device="cuda", generator=gen)
        if kind == "scaled":
            s *= torch.exp(torch.randn(count, k, 1, dtype=F64, device="cuda", generator=gen))
        s = s @ s.mT / t
        s.diagonal(dim1=-2, dim2=-1).add_(0.01 * s.diagonal(dim1=-2, dim2=-1).mean(-1, keepdim=True))
    return 0.5 * (s + s.mT)


def _upper(s):
    """The upper triangular R with R^T R = s: how the configurations store a basis."""
    return torch.linalg.cholesky(s).mT.contiguous()


def _unit_lower(s):
    """(F, p^2) of s = P^T P, P lower triangular: F = P^-1 diag(P) (unit lower), and the squared diagonal."""
    p = torch.linalg.cholesky(s.flip(-1, -2)).flip(-1, -2).mT
    d = p.diagonal(dim1=-2, dim2=-1)
    eye = torch.eye(s.shape[-1], dtype=F64, device=s.device).expand_as(s)
    f = torch.linalg.solve_triangular(p.contiguous(), eye, upper=False) * d.unsqueeze(-2)
    return f.tril(-1) + eye, d * d


def _factors(case, gen, count, m, n):
    left = _unit_lower(_gram(gen, count, m, case["kind"]))[0]
    right = _unit_lower(_gram(gen, count, n, case["kind"]))[0].mT
    return left.contiguous(), right.contiguous()


def _x(case, gen, count, m, n):
    if case["kind"] == "spectrum":
        return 15.0 * torch.rand(count, m, n, dtype=F64, device="cuda", generator=gen) - 7.5
    return 4.0 * torch.randn(count, m, n, dtype=F64, device="cuda", generator=gen)


def _ws(nbytes):
    return torch.empty(max(int(nbytes), 256), dtype=torch.uint8, device="cuda")


def _views(shapes, dtype):
    """Zeroed matrices in one buffer, each on a boundary of 64 elements: (buffer, views)."""
    at, size = [], 0
    for shape in shapes:
        at.append(size)
        size += -(-math.prod(shape) // 64) * 64
    flat = torch.zeros(size, dtype=dtype, device="cuda")
    return flat, [flat[o:o + math.prod(shape)].view(shape) for o, shape in zip(at, shapes)]


def _laid_out(v):
    """Matrices copied into such a buffer."""
    flat, views = _views([tuple(t.shape) for t in v], v[0].dtype)
    for t, w in zip(v, views):
        w.copy_(t)
    return flat


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    op, m, n = case["op"], case["m"], case["n"]
    if op == "sweep_batch":
        xs, ls, us = [None] * case["count"], [None] * case["count"], [None] * case["count"]
        for par in range(2):
            own = list(range(par, case["count"], 2))
            if own:
                w = n * (1 + par)
                f, u = _factors(case, gen, len(own), m, w)
                x = _x(case, gen, len(own), m, w)
                for k, b in enumerate(own):
                    xs[b], ls[b], us[b] = x[k].clone(), f[k].clone(), u[k].clone()
        return {"X": xs, "L": ls, "U": us}
    if op == "setup_batch":
        a, b = [], []
        for _ in range(case["count"]):
            a.append(_upper(_gram(gen, 1, m, case["kind"]))[0])
            b.append(_upper(_gram(gen, 1, n, case["kind"]))[0])
        return {"A": a, "B": b}
    if op in ("setup", "objective"):
        s = {"A": _upper(_gram(gen, 1, m, case["kind"]))[0], "B": _upper(_gram(gen, 1, n, case["kind"]))[0]}
        if op == "objective":
            s["X"] = _x(case, gen, 1, m, n)[0]
            s["Z"] = torch.round(s["X"]).to(torch.int32)
        return s
    f, u = _factors(case, gen, 1, m, n)
    s = {"X": _x(case, gen, 1, m, n)[0], "L": f[0], "U": u[0]}
    if op == "sweep_f32in":
        s = {k: v.float() for k, v in s.items()}
    if op == "sweep_reverse":
        s["L"], s["U"] = s["L"].mT.contiguous(), s["U"].mT.contiguous()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    op, m, n = case["op"], case["m"], case["n"]
    s["op"] = op
    s["info"] = torch.zeros(4, dtype=torch.int32, device="cuda")
    i32 = {"dtype": torch.int32, "device": "cuda"}
    f64 = {"dtype": F64, "device": "cuda"}
    if op in ("sweep", "sweep_f32in", "sweep_reverse"):
        s["Z"] = torch.empty(m, n, **i32)
        s["E"] = torch.empty(m, n, **f64) if case["E"] else None
        s["ws"] = _ws({"sweep": g.gptq2d_round_workspace_bytes, "sweep_f32in": g.gptq2d_round_f32in_workspace_bytes,
                       "sweep_reverse": g.gptq2d_round_reverse_workspace_bytes}[op](m, n))
    elif op == "sweep_host":
        for k in "XLU":
            s[k] = s[k].cpu().pin_memory()
        s["Z"] = torch.empty(m, n, dtype=torch.int32).pin_memory()
        s["info"] = torch.zeros(4, dtype=torch.int32).pin_memory()
        s["ws"] = _ws(g.gptq2d_round_host_workspace_bytes(m, n))
    elif op == "sweep_batch":
        s["Z"], zs = _views(_shapes(case), torch.int32)
        s["E"], es = _views(_shapes(case), F64) if case["E"] else (None, None)
        s["problems"] = g.make_problems(s["X"], s["L"], s["U"], zs, es)
        s["ws"] = _ws(g.gptq2d_round_batched_workspace_bytes(problems=s["problems"]))
    elif op == "setup_batch":
        views = {}
        for k, shape in (("L", (m, m)), ("U", (n, n)), ("dL", (m,)), ("dU", (n,))):
            s[k], views[k] = _views([shape] * case["count"], F64)
        s["problems"] = g.make_factor_problems(s["A"], s["B"], views["L"], views["U"], views["dL"], views["dU"])
        s["ws"] = _ws(g.gptq2d_factor_batched_workspace_bytes(s["problems"]))
    elif op == "setup":
        s["L"], s["U"] = torch.empty(m, m, **f64), torch.empty(n, n, **f64)
        s["dL"], s["dU"] = torch.empty(m, **f64), torch.empty(n, **f64)
        s["ws"] = _ws(g.gptq2d_factor_workspace_bytes(m, n))
    else:
        s["obj"] = torch.empty(1, **f64)
        s["ws"] = _ws(g.gptq2d_objective_workspace_bytes(m, n))
    return s


def run(s):
    op = s["op"]
    if op in ("sweep", "sweep_f32in", "sweep_reverse"):
        call = {"sweep": g.gptq2d_round, "sweep_f32in": g.gptq2d_round_f32in, "sweep_reverse": g.gptq2d_round_reverse}[op]
        call(s["X"], s["L"], s["U"], Z=s["Z"], E=s["E"], workspace=s["ws"], info=s["info"])
        return {"Z": s["Z"], "info": s["info"]} if s["E"] is None else {"Z": s["Z"], "E": s["E"], "info": s["info"]}
    if op == "sweep_host":
        g.gptq2d_round_host(s["X"], s["L"], s["U"], hZ=s["Z"], workspace=s["ws"], hinfo=s["info"])
        return {"Z": s["Z"], "info": s["info"]}
    if op == "sweep_batch":
        g.gptq2d_round_batched(problems=s["problems"], workspace=s["ws"], info=s["info"])
        return {"Z": s["Z"], "info": s["info"]} if s["E"] is None else {"Z": s["Z"], "E": s["E"], "info": s["info"]}
    if op == "setup_batch":
        g.gptq2d_factor_batched(problems=s["problems"], workspace=s["ws"], info=s["info"])
        return {k: s[k] for k in ("L", "U", "dL", "dU", "info")}
    if op == "setup":
        g.gptq2d_factor(s["A"], s["B"], s["L"], s["U"], s["dL"], s["dU"], workspace=s["ws"], info=s["info"])
        return {k: s[k] for k in ("L", "U", "dL", "dU", "info")}
    return g.gptq2d_objective(s["X"], s["Z"], s["A"], s["B"], obj=s["obj"], workspace=s["ws"], info=s["info"])


def work(case):
    op, m, n = case["op"], case["m"], case["n"]
    if op == "setup_batch":
        k3 = case["count"] * (m ** 3 + n ** 3)
        return {"bytes": 16 * case["count"] * (m * m + n * n), "flops": 5 * k3 / 3}
    if op == "setup":
        # half a Gram product, a Cholesky factorisation and a triangular inverse a side; basis in, factor out
        return {"bytes": 16 * (m * m + n * n), "flops": 5 * (m ** 3 + n ** 3) / 3}
    if op == "objective":
        return {"bytes": 12 * m * n + 8 * (m * m + n * n), "flops": 2 * m * n * (m + n)}
    total = {"bytes": 0, "flops": 0}
    word = 4 if op == "sweep_f32in" else 8
    for (r, c) in (_shapes(case) if op == "sweep_batch" else [(m, n)]):
        total["bytes"] += r * c * (word + 4 + (8 if case["E"] else 0)) + word * (r * r + c * c) // 2
        total["flops"] += r * c * max(1, r + c - 2)
    return total


def tolerance(case):
    # Two correct fp64 sweeps or factorisations differ by their rounding times the condition of the Grams (seen against
    # exact(): sweeps 3e-14, set-ups 9e-14 with single entries 7e-12 off, objective 3e-16); integers differ only behind
    # an entry within that distance of a tie.
    if case["op"] == "objective":
        return {"rel": 1e-14, "max": 1e-14}
    if case["kind"] == "spectrum" and case["op"].startswith("setup"):
        return {"rel": 1e-10, "max": 1e-8, "differ": 1e-6}
    return {"rel": 4e-13, "max": 4e-11, "differ": 1e-6}


def _sweep64(x, f, u):
    """The rounding itself in plain torch, one anti-diagonal at a time, on a batch (count, m, n): (Z, E)."""
    count, m, n = x.shape
    f, ut = f.tril(-1), u.triu(1).mT.contiguous()
    et = torch.zeros(count, n, m, dtype=F64, device=x.device)
    c = torch.zeros(count, m, n, dtype=F64, device=x.device)
    z = torch.zeros(count, m, n, dtype=F64, device=x.device)
    ar = torch.arange(max(m, n), device=x.device)
    for d in range(m + n - 1):
        i0, i1 = max(0, d - n + 1), min(m, d + 1)
        i = ar[i0:i1]
        j = d - i
        jtop = d - i0 + 1
        down = (f[:, i0:i1, :i1] * et[:, :, :i1][:, j]).sum(-1)
        y = x[:, i, j] + (c[:, i0:i1, :jtop] * ut[:, :, :jtop][:, j]).sum(-1) + down
        r = torch.round(y)
        z[:, i, j] = r
        et[:, j, i] = r - y
        c[:, i, j] = down + (r - y)
    return z.to(torch.int32), et.mT.contiguous()


def exact(case, seed):
    op, m, n = case["op"], case["m"], case["n"]
    if op == "sweep_batch":
        if not case["E"]:
            return None
        s = _inputs(case, seed)
        out = [None] * case["count"]
        for par in range(2):
            own = list(range(par, case["count"], 2))
            if own:
                z, e = _sweep64(*(torch.stack([s[k][b] for b in own]) for k in "XLU"))
                for k, b in enumerate(own):
                    out[b] = (z[k], e[k])
        return {"Z": _laid_out([o[0] for o in out]), "E": _laid_out([o[1] for o in out]), "info": None}
    if op.startswith("sweep"):
        if not case["E"] or m * n > 4096 * 4096 + 1:
            return None
        s = {k: v.double().unsqueeze(0) for k, v in _inputs(case, seed).items()}
        if op == "sweep_reverse":
            z, e = _sweep64(*(s[k].flip(-1, -2) for k in "XLU"))
            z, e = z.flip(-1, -2).contiguous(), e.flip(-1, -2).contiguous()
        else:
            z, e = _sweep64(s["X"], s["L"], s["U"])
        return {"Z": z[0], "E": e[0], "info": None}
    s = _inputs(case, seed)
    if op == "objective":
        return (s["A"] @ ((s["Z"].double() - s["X"]) @ s["B"])).square().sum().reshape(1)
    pairs = list(zip(s["A"], s["B"])) if op == "setup_batch" else [(s["A"], s["B"])]
    out = []
    for a, b in pairs:
        f, dl = _unit_lower((a.mT @ a).unsqueeze(0))
        u, du = _unit_lower((b @ b.mT).unsqueeze(0))
        out.append((f[0], u[0].mT.contiguous(), dl[0], du[0]))
    if op == "setup_batch":
        return dict({k: _laid_out([o[q] for o in out]) for q, k in enumerate(("L", "U", "dL", "dU"))}, info=None)
    return {"L": out[0][0], "U": out[0][1], "dL": out[0][2], "dU": out[0][3], "info": None}
