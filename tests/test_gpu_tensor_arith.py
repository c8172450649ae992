"""arith="tensor" (PES_ARITH_TENSOR) by name, at every k and degree around the column tiles'
edges and for every kind of plan: the oracle's results within the tolerance of the other
arithmetics, the integer pipe's within what a product drops, and the same bits from every
plan given it, whatever shares the plan.

The 28-bit form drops at most 2^-(53 k - 1) of the product of the largest coefficients per
product (k = 10; less at the other k) and the tensor form less; 2^24 above a k-double's last
bit leaves room for sums over a few hundred terms and monomials and for the cancellation
between them."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2101_10881_gb300 import pes, synth
from paper_2101_10881_gb300.synth import random_md
from tests.exact import TOL, normwise_err

pytestmark = pytest.mark.gpu

KT = (4, 5, 8, 10)


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    pes.build()
    assert _t.cuda.is_available()
    return _t


def close(k):
    return 2.0 ** -(53 * k - 24)


def cuda(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("k", KT)
@pytest.mark.parametrize("d", [0, 1, 6, 7, 8, 23, 24, 33])
@pytest.mark.parametrize("opts", [{}, {"tile": 16}])
def test_degrees_match_oracle(torch, k, d, opts):
    rng = np.random.default_rng(100 * k + d)
    n = 7
    supp = synth.random_supports(rng, n, 12, 1, 5)
    ex = [[int(e) for e in rng.integers(1, 4, size=len(s))] for s in supp]
    coeff, inputs = random_md(rng, k, (len(supp) + 1, d + 1)), random_md(rng, k, (n, d + 1))
    u = random_md(rng, k, (d + 1,))
    plan = pes.Plan(supp, n, d, k, exponents=ex, arith="tensor", **opts)
    assert plan.arith() == "tensor" and plan.info()["arith_name"] == "int"
    C, Z, U = (cuda(torch, a) for a in (coeff, inputs, u))
    got = [*plan.eval_grad(C, Z), *plan.vjp(C, Z, U, reuse_forward=True)]
    plan.check()
    ref = [*O.eval_grad(supp, n, coeff, inputs, exponents=ex), *O.vjp(supp, n, coeff, inputs, u, exponents=ex)]
    other = pes.Plan(supp, n, d, k, exponents=ex, arith="int", **opts)
    assert other.arith() == "int"
    same = [*other.eval_grad(C, Z), *other.vjp(C, Z, U, reuse_forward=True)]
    for a, r, b in zip(got, ref, same):
        a = a.cpu().numpy()
        assert normwise_err(a, r) <= TOL[k]
        assert normwise_err(a, b.cpu().numpy()) <= close(k)


@pytest.mark.parametrize("k", KT)
def test_complex_powers_match_the_integer_pipe(torch, k):
    rng = np.random.default_rng(k)
    n, d = 6, 41
    supp = synth.random_supports(rng, n, 14, 1, 5)
    ex = [[int(e) for e in rng.integers(1, 4, size=len(s))] for s in supp]
    C, Z, U = (cuda(torch, np.stack([random_md(rng, k, shape), random_md(rng, k, shape)]))
               for shape in ((len(supp) + 1, d + 1), (n, d + 1), (d + 1,)))
    got = []
    for arith in ("tensor", "int"):
        plan = pes.Plan(supp, n, d, k, exponents=ex, complex_series=True, arith=arith)
        got.append([*plan.eval_grad(C, Z), *plan.vjp(C, Z, U, reuse_forward=True)])
        plan.check()
    for a, b in zip(*got):
        for part in (0, 1):
            assert normwise_err(a[part].cpu().numpy(), b[part].cpu().numpy()) <= close(k)


@pytest.mark.parametrize("k", KT)
def test_systems_and_batches_have_the_bits_of_single_plans(torch, k):
    """Polynomials of all widths, a constant one among them, and degrees on both sides of the
    column tiles."""
    rng = np.random.default_rng(10 + k)
    n, d = 8, 40
    polys = [synth.random_supports(rng, n, N, 1, 5) for N in (1, 9, 30)] + [[]]
    coeffs = [random_md(rng, k, (len(p) + 1, d + 1)) for p in polys]
    Z = cuda(torch, random_md(rng, k, (n, d + 1)))
    sysp = pes.System(polys, n, d, k, arith="tensor")
    v, jac = sysp.eval_system(cuda(torch, np.concatenate(coeffs, axis=1)), Z, layout="series")
    sysp.check()
    for p, (supp, coeff) in enumerate(zip(polys, coeffs)):
        pv, pg = pes.Plan(supp, n, d, k, with_vjp=False, arith="tensor").eval_grad(cuda(torch, coeff), Z)
        assert torch.equal(v[:, p], pv) and torch.equal(jac[:, p], pg), p

    inst = [(synth.random_supports(rng, n, N, 1, 5), n, dd) for N, dd in ((5, 3), (20, 47), (9, 40), (14, 8))]
    cs = [random_md(rng, k, (len(s) + 1, dd + 1)) for s, _, dd in inst]
    zs = [random_md(rng, k, (n, dd + 1)) for _, _, dd in inst]
    batch = pes.Batch(inst, k, arith="tensor")
    ln = batch.lengths()
    bv, bg = (torch.empty(ln[name], dtype=torch.float64, device="cuda") for name in ("value", "grad"))
    batch.eval_grad(cuda(torch, np.concatenate([c.reshape(-1) for c in cs])),
                    cuda(torch, np.concatenate([z.reshape(-1) for z in zs])), bv, bg)
    batch.check()
    vo = go = 0
    for (supp, _, dd), c, z in zip(inst, cs, zs):
        pv, pg = pes.Plan(supp, n, dd, k, with_vjp=False, arith="tensor").eval_grad(cuda(torch, c), cuda(torch, z))
        nv, ng = pv.numel(), pg.numel()
        assert torch.equal(bv[vo:vo + nv], pv.reshape(-1)) and torch.equal(bg[go:go + ng], pg.reshape(-1))
        vo, go = vo + nv, go + ng


def against_the_integer_pipe(torch, k, d, supp, n, coeff, inputs):
    C, Z, U = (cuda(torch, a) for a in (coeff, inputs, inputs[:, 0]))
    got, infos = [], []
    for arith in ("tensor", "int"):
        plan = pes.Plan(supp, n, d, k, arith=arith)
        got.append([*plan.eval_grad(C, Z), *plan.vjp(C, Z, U, reuse_forward=True)])
        plan.check()
        infos.append(plan.info())
    for a, b in zip(*got):
        assert normwise_err(a.cpu().numpy(), b.cpu().numpy()) <= close(k)
    return infos


@pytest.mark.parametrize("k,d,tile", [(8, 513, 0), (8, 514, 128), (5, 563, 0), (5, 564, 128), (4, 669, 0),
                                      (4, 670, 128), (10, 471, 0), (10, 472, 128)])
def test_whole_series_and_tiles(torch, k, d, tile):
    """The tiled kernel takes the degrees whose staged pairs do not fit in shared memory, also
    where 28-bit digits would."""
    rng = np.random.default_rng(d)
    info, _ = against_the_integer_pipe(torch, k, d, [[0, 1, 2], [1, 2]], 3, random_md(rng, k, (3, d + 1)),
                                       random_md(rng, k, (3, d + 1)))
    assert info["tile"] == tile


@pytest.mark.parametrize("k,d", [(10, 152), (10, 700), (10, 1300), (8, 300), (8, 2500), (5, 200), (4, 330), (4, 2500)])
def test_maximal_slices(torch, k, d):
    """Every slice of every coefficient near its largest value and of one sign: the
    accumulators' upper parts are moved as often as ever, and carried in mid-series beyond 563
    terms at k = 10 and 2339 at k = 8."""
    from fractions import Fraction
    W = 10 if k == 10 else 9
    f = sum(Fraction(2 ** (W - 1) - 1, 2 ** (W * p)) for p in range(1, 53 * k // W + 2))
    x = np.array(synth.round_fraction_to_limbs(f, k))
    coeff, inputs = np.zeros((k, 2, d + 1)), np.zeros((k, 2, d + 1))
    coeff[:] = inputs[:] = x[:, None, None]
    against_the_integer_pipe(torch, k, d, [[0, 1]], 2, coeff, inputs)


@pytest.mark.parametrize("k", KT)
def test_products_far_below_the_smallest_double(torch, k):
    """Running products down to 2^-1900000 come back to 1: series are taken for zero below
    2^-2800000 only, as on the integer pipe."""
    n, d = 3800, 1
    inputs = np.zeros((k, n, d + 1))
    inputs[0, :, 0] = np.where(np.arange(n) < n // 2, 2.0 ** -1000, 2.0 ** 1000)
    inputs[0, :, 1] = inputs[0, :, 0] * (1 + np.arange(n) % 7)
    coeff = np.zeros((k, 2, d + 1))
    coeff[0, 1, 0] = 1.0
    got = []
    for arith in ("tensor", "int"):
        plan = pes.Plan([list(range(n))], n, d, k, with_vjp=False, arith=arith)
        got.append([t.cpu().numpy() for t in plan.eval_grad(cuda(torch, coeff), cuda(torch, inputs))])
        plan.check()
    assert got[0][0][0, 0] == 1.0
    for a, b in zip(*got):
        assert normwise_err(a, b) <= close(k)


@pytest.mark.parametrize("k", KT)
def test_one_product_is_exact_to_the_last_limb(torch, k):
    """One product of two series against rationals: what the tensor form drops of a product and
    the rounding to k limbs together stay below 2^-(53 k - 2) of the sum of the terms'
    magnitudes (2^-(53 k) from the rounding, less than 2^-(53 k) dropped)."""
    from fractions import Fraction
    from tests.exact import series_fractions
    rng = np.random.default_rng(k)
    d = 40
    inputs = random_md(rng, k, (2, d + 1))
    coeff = np.zeros((k, 2, d + 1))
    coeff[0, 1, 0] = 1.0
    plan = pes.Plan([[0, 1]], 2, d, k, with_vjp=False, arith="tensor")
    v, _ = plan.eval_grad(cuda(torch, coeff), cuda(torch, inputs))
    plan.check()
    got = series_fractions(v.cpu().numpy())
    x, y = series_fractions(inputs)
    for j in range(d + 1):
        terms = [x[i] * y[j - i] for i in range(j + 1)]
        assert abs(got[j] - sum(terms)) <= sum(abs(t) for t in terms) * Fraction(1, 2 ** (53 * k - 2))
