"""Terms that reach no coefficient of a product (zero coefficients at either end, products far
below the largest) are left out by the tensor-core kernels: same results as the integer pipe
from every pattern of zeros and of falling magnitudes, and less time for short series.

Both pipes drop at most 2^-(53 k - 1) of the product of the largest coefficients per product;
2^24 above a k-double's last bit leaves room for sums over a few hundred terms and monomials
and for the cancellation between them."""
import itertools

import numpy as np
import pytest

from paper_2101_10881_gb300 import pes
from paper_2101_10881_gb300.synth import random_md
from tests.exact import normwise_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    pes.build()
    assert _t.cuda.is_available()
    return _t


def falling(a, bits):
    return a * 2.0 ** -np.minimum(bits * np.arange(a.shape[-1]), 900)


def only(a, lo, hi):
    b = np.zeros_like(a)
    b[:, :, lo:hi] = a[:, :, lo:hi]
    return b


PATTERNS = {
    "scalar coefficients, degree 1": lambda c, z: (only(c, 0, 1), only(z, 0, 2)),
    "middle": lambda c, z: (c, only(z, z.shape[-1] // 3, z.shape[-1] // 2)),
    "last": lambda c, z: (only(c, c.shape[-1] - 1, c.shape[-1]), z),
    "falling to zeros": lambda c, z: (only(c, 0, 1), only(falling(z, 11), 0, z.shape[-1] // 4)),
    "rising": lambda c, z: (c, falling(z, 5)[:, :, ::-1].copy()),
    "falling": lambda c, z: (falling(c, 3), falling(z, 9)),
    "zero": lambda c, z: (c, 0 * z),
}


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("k,d,n", [(10, 95, 30), (4, 152, 40), (8, 95, 32), (10, 600, 9)])
def test_ranges_match_the_integer_pipe(torch, k, d, n, pattern):
    rng = np.random.default_rng(d)
    supp = [list(s) for s in itertools.combinations(range(n), 2)]
    coeff, inputs = PATTERNS[pattern](random_md(rng, k, (len(supp) + 1, d + 1)), random_md(rng, k, (n, d + 1)))
    C, Z, U = (torch.from_numpy(np.ascontiguousarray(a)).cuda()
               for a in (coeff, inputs, random_md(rng, k, (d + 1,))))
    U[:, 5:] = 0  # an upstream series of few coefficients
    got, words = [], []
    for arith in ("auto", "int"):
        plan = pes.Plan(supp, n, d, k, arith=arith)
        got.append([*plan.eval_grad(C, Z), *plan.vjp(C, Z, U, reuse_forward=True)])
        plan.check()
        words.append(plan.info()["workspace_bytes"])
    assert words[0] != words[1]  # tensor cores, integer pipe
    for a, b in zip(*got):
        assert normwise_err(a.cpu().numpy(), b.cpu().numpy()) <= 2.0 ** -(53 * k - 24)


@pytest.mark.parametrize("k,d,n,parts", [(4, 152, 48, "both"), (10, 600, 12, "inputs")])
def test_short_series_take_less_time(torch, k, d, n, parts):
    rng = np.random.default_rng(1)
    supp = [list(s) for s in itertools.combinations(range(n), 2)]
    C = torch.from_numpy(random_md(rng, k, (len(supp) + 1, d + 1))).cuda()
    Z = torch.from_numpy(random_md(rng, k, (n, d + 1))).cuda()
    plan = pes.Plan(supp, n, d, k, with_vjp=False)
    best = {}
    for name, length in (("full", d + 1), ("short", 2)):
        c, z = C.clone(), Z.clone()
        if parts == "both":
            c[:, :, length:] = 0
        z[:, :, length:] = 0
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.eval_grad(c, z)
            b.record()
            b.synchronize()
            best[name] = min(best.get(name, 1e9), a.elapsed_time(b))
    assert best["short"] < (0.75 if parts == "both" else 0.5) * best["full"], best


@pytest.mark.parametrize("pattern", PATTERNS)
@pytest.mark.parametrize("k,d,n", [(10, 95, 8), (4, 152, 8), (8, 101, 8), (5, 67, 8)])
def test_tiles_have_the_bits_of_whole_series(torch, k, d, n, pattern):
    """The tiled kernel exchanges a product's operands by where their zeros lie and stages fewer
    chunks; whole series clip their terms: the same sums."""
    rng = np.random.default_rng(d)
    supp = [list(s) for m in (2, 3) for s in itertools.combinations(range(n), m)]
    coeff, inputs = PATTERNS[pattern](random_md(rng, k, (len(supp) + 1, d + 1)), random_md(rng, k, (n, d + 1)))
    C, Z, U = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (coeff, inputs, random_md(rng, k, (d + 1,))))
    U[:, 5:] = 0
    got = []
    for opts in ({}, {"tile": 16}, {"tile": 48}, {"split": 2, "staging": 2}):
        plan = pes.Plan(supp, n, d, k, arith="tensor", **opts)
        got.append([*plan.eval_grad(C, Z), *plan.vjp(C, Z, U, reuse_forward=True)])
        plan.check()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert torch.equal(a, b)
