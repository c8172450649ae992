"""The calls whose time matters: evaluation and differentiation at power series.

Every case goes through the public entry points with the plan a program keeps
between calls (job tables and workspace), its series in device memory.  Sizes
are those of the paper's polynomials, of the batched and the system workloads,
and ordinary or ragged ones between them; series are random k-doubles with
uniform leading limbs, or, for the system, exponential series with scalar
coefficients, whose coefficients span hundreds of bits.

Outputs are k-limb arrays, limb 0 carrying the value to double precision.  The
64-bit evaluation is laid out the same: its value in limb 0, zeros below.
"""
import itertools
import math

import numpy as np
import torch

from paper_2101_10881_gb300 import pes

KS = (1, 2, 3, 4, 5, 8, 10)
DEV = "cuda"


def listed():
    return [
        # the smallest call: all 1820 products of 4 of 16 variables, low degree, double double
        {"name": "p1_k2_d8", "kind": "poly", "supp": "all", "n": 16, "m": 4, "k": 2, "d": 8},
        # an ordinary small polynomial of one Newton step, ragged degree, quad double
        {"name": "small_k4_d37", "kind": "poly", "supp": "mix", "n": 10, "N": 60, "lo": 1, "m": 5, "k": 4, "d": 37},
        # the paper's second polynomial: 128 products of 64 of 128 variables, deca double
        {"name": "p2_k10_d152", "kind": "poly", "supp": "draw", "n": 128, "N": 128, "m": 64, "k": 10, "d": 152},
        # the paper's third polynomial, all pairs of 128 variables, double double
        {"name": "p3_k2_d152", "kind": "poly", "supp": "all", "n": 128, "m": 2, "k": 2, "d": 152},
        # the same in quad double, the forward and the backward pass of autograd
        {"name": "p3_grad_k4_d152", "kind": "grad", "supp": "all", "n": 128, "m": 2, "k": 4, "d": 152},
        # one long product: a dependency chain of 64 factors, latency rather than throughput
        {"name": "chain_k10_d152", "kind": "poly", "supp": "draw", "n": 64, "N": 1, "m": 64, "k": 10, "d": 152},
        # octo double at an odd degree, forward and backward
        {"name": "p1_grad_k8_d95", "kind": "grad", "supp": "all", "n": 12, "m": 4, "k": 8, "d": 95},
        # complex series, monomials with powers, triple double
        {"name": "complex_k3_d63", "kind": "complex", "supp": "draw", "n": 32, "N": 48, "m": 12, "k": 3, "d": 63},
        # a degree beyond whole series in shared memory
        {"name": "long_k10_d1023", "kind": "poly", "supp": "draw", "n": 32, "N": 8, "m": 16, "k": 10, "d": 1023},
        # a system and its Jacobian as one matrix per power of t: a Newton step on exponential series
        {"name": "system_k5_d63", "kind": "system", "n": 24, "P": 24, "N": 32, "m": 12, "k": 5, "d": 63},
        # many instances in one call: large ones of mixed degrees, and many small ones
        {"name": "batch_k2", "kind": "batch", "count": 24, "n": 128, "N": 2048, "m": 8, "d": 152, "k": 2},
        {"name": "batch_small_k2", "kind": "batch", "count": 768, "n": 16, "N": 32, "m": 4, "d": 31, "k": 2},
    ]


def draw(rng):
    most = 0.5 * _muls(listed()[2])
    while True:
        c = _drawn(rng)
        if _muls(c) <= most:
            return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def _drawn(rng):
    kind = rng.choice(["poly", "poly", "poly", "grad", "grad", "complex", "system", "batch"])
    k = rng.choice(KS)
    d = _log(rng, 4, 190)
    if kind == "batch":
        N = _log(rng, 16, 1024)
        return {"kind": kind, "count": _log(rng, 8, max(8, min(512, 32768 // N))), "n": _log(rng, 8, 128), "N": N,
                "m": rng.randint(2, 8), "d": d, "k": k}
    if kind == "system":
        n = _log(rng, 4, 48)
        return {"kind": kind, "n": n, "P": _log(rng, 2, 48), "N": _log(rng, 4, 96), "m": min(n, rng.randint(2, 16)),
                "k": k, "d": d}
    if kind == "complex":
        n = _log(rng, 4, 48)
        return {"kind": kind, "supp": "draw", "n": n, "N": _log(rng, 4, 256), "m": min(n, rng.randint(1, 16)), "k": k,
                "d": d}
    if kind == "poly" and rng.random() < 0.25:  # few monomials of a high degree
        n = rng.randint(6, 32)
        return {"kind": kind, "supp": "mix", "n": n, "N": rng.randint(2, 10), "lo": 2, "m": min(n, rng.randint(3, 16)),
                "k": k, "d": _log(rng, 200, 1500)}
    n = _log(rng, 4, 128)
    return {"kind": kind, "supp": "mix", "n": n, "N": _log(rng, 2, 4096), "lo": 1, "m": min(n, _log(rng, 2, 64)), "k": k,
            "d": d}


# ---------------------------------------------------------------------------
# structures (fixed by the case) and series (by the seed)
# ---------------------------------------------------------------------------

def _subsets(rng, n, N, lo, hi):
    return [sorted(int(v) for v in rng.choice(n, size=int(rng.integers(lo, hi + 1)), replace=False)) for _ in range(N)]


def _supports(c):
    if c["supp"] == "all":
        return [list(s) for s in itertools.combinations(range(c["n"]), c["m"])]
    return _subsets(np.random.default_rng(7), c["n"], c["N"], c.get("lo", c["m"]), c["m"])


def _exponents(supp):
    rng = np.random.default_rng(8)
    return [[int(e) for e in rng.integers(1, 4, size=len(s))] for s in supp]


def _system(c):
    rng = np.random.default_rng(7)
    return [_subsets(rng, c["n"], c["N"], min(2, c["m"]), c["m"]) for _ in range(c["P"])]


def _instances(c):
    rng = np.random.default_rng(7)
    out = []
    for _ in range(c["count"]):
        n = int(rng.integers(max(4, c["n"] // 16), c["n"] + 1))
        N = int(rng.integers(max(4, c["N"] // 128), c["N"] + 1))
        d = int(rng.choice([max(1, c["d"] // 10), max(1, c["d"] // 5), max(1, c["d"] * 2 // 5), c["d"]]))
        out.append((_subsets(rng, n, N, min(2, n), min(c["m"], n)), n, d))
    return out


def _limbs(lead, k, gen):
    """k-doubles with the given leading limbs: each further limb uniform within half an ulp of the one above."""
    out = torch.empty((k,) + tuple(lead.shape), dtype=torch.float64, device=DEV)
    out[0] = lead
    for l in range(1, k):
        ulp = torch.ldexp(torch.ones_like(lead), torch.frexp(out[l - 1]).exponent - 53)
        u = torch.rand(lead.shape, generator=gen, dtype=torch.float64, device=DEV) * 2 - 1
        out[l] = torch.where(out[l - 1] == 0, 0.0, 0.5 * u * ulp)
    return out


def _uniform(shape, k, gen):
    return _limbs(torch.rand(shape, generator=gen, dtype=torch.float64, device=DEV) * 2 - 1, k, gen)


def _exponential(n, d, k, gen):
    """exp(a t) with a uniform in (-1, 1): coefficients a^j / j!."""
    a = torch.rand((n, 1), generator=gen, dtype=torch.float64, device=DEV) * 2 - 1
    j = torch.arange(d + 1, dtype=torch.float64, device=DEV)
    lead = torch.exp(j * torch.log(a.abs()) - torch.lgamma(j + 1))
    return _limbs(torch.where((j % 2 == 1) & (a < 0), -lead, lead), k, gen)


def _series(c, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000003 * seed + 17)
    k = c["k"]
    if c["kind"] == "batch":
        inst = _instances(c)
        return {"inst": inst,
                "coeff": torch.cat([_uniform((len(s) + 1, d + 1), k, gen).reshape(-1) for s, n, d in inst]),
                "input": torch.cat([_uniform((n, d + 1), k, gen).reshape(-1) for s, n, d in inst])}
    n, S = c["n"], c["d"] + 1
    if c["kind"] == "system":
        polys = _system(c)
        coeff = torch.zeros((k, c["P"] * (c["N"] + 1), S), dtype=torch.float64, device=DEV)
        coeff[:, :, 0] = _uniform((c["P"] * (c["N"] + 1),), k, gen)
        return {"polys": polys, "coeff": coeff, "input": _exponential(n, c["d"], k, gen)}
    supp = _supports(c)
    one = lambda r: _uniform((r, S), k, gen)
    if c["kind"] == "complex":
        return {"supp": supp, "ex": _exponents(supp), "coeff": torch.stack([one(len(supp) + 1), one(len(supp) + 1)]),
                "input": torch.stack([one(n), one(n)])}
    out = {"supp": supp, "coeff": one(len(supp) + 1), "input": one(n)}
    if c["kind"] == "grad":
        out["up"] = _uniform((S,), k, gen)
    return out


def prepare(case, seed):
    s = _series(case, seed)
    kind, k = case["kind"], case["k"]
    if kind == "batch":
        s["plan"] = pes.Batch(s.pop("inst"), k)
        ln = s["plan"].lengths()
        for name in ("value", "grad"):
            s[name] = torch.empty(ln[name], dtype=torch.float64, device=DEV)
    elif kind == "system":
        s["plan"] = pes.System(s.pop("polys"), case["n"], case["d"], k, with_vjp=False)
    elif kind == "complex":
        s["plan"] = pes.Plan(s.pop("supp"), case["n"], case["d"], k, exponents=s.pop("ex"), complex_series=True,
                             with_vjp=False)
    else:
        s["plan"] = pes.Plan(s.pop("supp"), case["n"], case["d"], k, with_vjp=kind == "grad")
    s["kind"] = kind
    return s


def run(state):
    plan, kind = state["plan"], state["kind"]
    if kind == "batch":
        return plan.eval_grad(state["coeff"], state["input"], state["value"], state["grad"])
    if kind == "system":
        return plan.eval_system(state["coeff"], state["input"], layout="matrix")
    value, grad = plan.eval_grad(state["coeff"], state["input"])
    if kind == "grad":
        gi, gc = plan.vjp(state["coeff"], state["input"], state["up"], reuse_forward=True)
        return value, grad, gi, gc
    return value, grad


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _products(supp, ex=None):
    """Series products of the reverse mode: 3 n_m - 3 per monomial, one for n_m = 1, and those of its powers."""
    t = 0
    for i, s in enumerate(supp):
        t += 3 * len(s) - 3 if len(s) > 1 else 1
        if ex is not None:
            t += sum(1 for e in ex[i] if e > 1)
    return t


def _muls(c):
    """Products of doubles: k (k + 1) / 2 of them in a k-double product kept to k doubles."""
    per = lambda d: (d + 1) * (d + 2) // 2 * c["k"] * (c["k"] + 1) // 2
    if c["kind"] == "batch":
        return sum(_products(s) * per(d) for s, n, d in _instances(c))
    if c["kind"] == "system":
        return sum(_products(p) for p in _system(c)) * per(c["d"])
    supp = _supports(c)
    if c["kind"] == "complex":
        return 4 * _products(supp, _exponents(supp)) * per(c["d"])
    extra = len(supp) + c["n"] if c["kind"] == "grad" else 0
    return (_products(supp) + extra) * per(c["d"])


def work(case):
    k, d = case["k"], case["d"]
    if case["kind"] == "batch":
        words = sum((len(s) + 1 + n + 1 + n) * (di + 1) for s, n, di in _instances(case))
    elif case["kind"] == "system":
        P, n, N = case["P"], case["n"], case["N"]
        words = (P * (N + 1) + n + P + P * n) * (d + 1)
    else:
        N, n = len(_supports(case)), case["n"]
        words = (N + 1 + n + 1 + n) * (d + 1)
        if case["kind"] == "grad":
            words += (1 + n + N + 1) * (d + 1)
        if case["kind"] == "complex":
            words *= 2
    return {"bytes": 8 * k * words, "flops": 2 * _muls(case)}


# ---------------------------------------------------------------------------
# the same in plain 64-bit arithmetic
# ---------------------------------------------------------------------------

def _conv(x, y):
    """Truncated products of series, row by row."""
    z = torch.zeros_like(x)
    S = x.shape[-1]
    for i in range(S):
        z[..., i:] += x[..., i:i + 1] * y[..., :S - i]
    return z


def _corr(u, y):
    """sum_l u_l y_{l-j}, row by row."""
    return _conv(u.flip(-1).expand_as(y).contiguous(), y).flip(-1)


def _eval(items, a0, out_shape):
    """items: (value row, gradient rows, coefficient, factors, exponents) of every monomial; sums into rows."""
    res = torch.zeros(out_shape, dtype=a0.dtype, device=DEV)
    groups = {}
    for it in items:
        groups.setdefault(len(it[1]), []).append(it)
    for m, its in groups.items():
        a = torch.stack([t[2] for t in its])
        F = [torch.stack([t[3][i] for t in its]) for i in range(m)]
        E = torch.tensor([t[4] for t in its], dtype=torch.float64, device=DEV)
        base = a
        for e in range(2, int(E.max()) + 1):  # the common factors of powers go into the coefficient
            for i in range(m):
                sel = (E[:, i] >= e).nonzero().flatten()
                if sel.numel():
                    base = base.clone()
                    base[sel] = _conv(base[sel], F[i][sel])
        suffix = [None] * (m + 1)
        for i in range(m - 1, 0, -1):
            suffix[i] = F[i] if suffix[i + 1] is None else _conv(suffix[i + 1], F[i])
        pre = base
        for i in range(m):
            g = pre if suffix[i + 1] is None else _conv(pre, suffix[i + 1])
            rows = torch.tensor([t[1][i] for t in its], device=DEV)
            res.index_add_(0, rows, g * E[:, i:i + 1])
            pre = _conv(pre, F[i])
        res.index_add_(0, torch.tensor([t[0] for t in its], device=DEV), pre)
    return res


def _lead(t, k):
    """Values in limb 0 of a k-limb array."""
    out = torch.zeros((k,) + tuple(t.shape), dtype=torch.float64, device=DEV)
    out[0] = t
    return out


def _poly(supp, a, z, ex=None):
    n = z.shape[0]
    items = [(0, [1 + v for v in s], a[1 + i], [z[v] for v in s], ex[i] if ex else [1] * len(s))
             for i, s in enumerate(supp)]
    res = _eval(items, a, (n + 1, z.shape[1]))
    res[0] += a[0]
    return res[0], res[1:]


def exact(case, seed):
    s = _series(case, seed)
    kind, k, S = case["kind"], case["k"], case["d"] + 1
    if kind == "batch":
        value, grad, co, io = [], [], 0, 0
        if len(s["inst"]) > 64:
            return None  # hundreds of small evaluations one by one
        for supp, n, d in s["inst"]:
            nc, ni = k * (len(supp) + 1) * (d + 1), k * n * (d + 1)
            v, g = _poly(supp, s["coeff"][co:co + nc].view(k, len(supp) + 1, d + 1).sum(0),
                         s["input"][io:io + ni].view(k, n, d + 1).sum(0))
            value.append(_lead(v, k).reshape(-1))
            grad.append(_lead(g, k).reshape(-1))
            co, io = co + nc, io + ni
        return torch.cat(value), torch.cat(grad)
    if kind == "system":
        a, z = s["coeff"].sum(0), s["input"].sum(0)
        P, n, N = case["P"], case["n"], case["N"]
        items = []
        for p, poly in enumerate(s["polys"]):
            for i, m in enumerate(poly):
                items.append((p, [P + p * n + v for v in m], a[p * (N + 1) + 1 + i], [z[v] for v in m], [1] * len(m)))
        res = _eval(items, a, (P + P * n, S))
        res[:P] += a[::N + 1]
        return _lead(res[:P].t().contiguous(), k), _lead(res[P:].t().reshape(S, P, n), k)
    if kind == "complex":
        a, z = (torch.complex(s[t][0].sum(0), s[t][1].sum(0)) for t in ("coeff", "input"))
        v, g = _poly(s["supp"], a, z, s["ex"])
        both = lambda t: torch.stack([_lead(t.real, k), _lead(t.imag, k)])
        return both(v), both(g)
    a, z = s["coeff"].sum(0), s["input"].sum(0)
    v, g = _poly(s["supp"], a, z)
    if kind != "grad":
        return _lead(v, k), _lead(g, k)
    u = s["up"].sum(0)
    gi = _corr(u[None], g)
    gc = torch.empty_like(a)
    gc[0] = u
    prods = torch.empty_like(a[1:])
    by = {}
    for i, m in enumerate(s["supp"]):
        by.setdefault(len(m), []).append(i)
    for m, idx in by.items():
        rows = torch.tensor(idx, device=DEV)
        M = torch.stack([z[s["supp"][i][0]] for i in idx])
        for f in range(1, m):
            M = _conv(M, torch.stack([z[s["supp"][i][f]] for i in idx]))
        prods[rows] = M
    gc[1:] = _corr(u[None], prods)
    return _lead(v, k), _lead(g, k), _lead(gi, k), _lead(gc, k)
