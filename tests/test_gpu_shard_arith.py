"""Split polynomials, two of them such as a plan puts on the tensor cores: the ranks' plans of
the same options give one plan's bits, by default and for arith="auto", "tensor" and "int",
however few monomials a rank holds."""
import itertools

import numpy as np
import pytest

from paper_2101_10881_gb300 import pes, synth
from paper_2101_10881_gb300.shard import ShardPlan, combine_host
from paper_2101_10881_gb300.synth import random_md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    pes.build()
    assert _t.cuda.is_available()
    return _t


def cases():
    rng = np.random.default_rng(5)
    pairs = [list(s) for s in itertools.combinations(range(32), 2)]
    mixed = synth.random_supports(rng, 24, 300, 1, 5)
    powers = [[int(e) for e in rng.integers(1, 4, size=len(s))] for s in mixed]
    return {"pairs k=10": (pairs, 32, 95, 10, None), "pairs k=4": (pairs, 32, 152, 4, None),
            "powers k=8": (mixed, 24, 95, 8, powers)}


@pytest.mark.parametrize("case", ["pairs k=10", "pairs k=4", "powers k=8"])
@pytest.mark.parametrize("opts", [{}, {"arith": "auto"}, {"arith": "tensor"}, {"arith": "int"}])
@pytest.mark.parametrize("world", [2, 7])
def test_shards_have_the_whole_plans_bits(torch, case, opts, world):
    supports, n, d, k, ex = cases()[case]
    rng = np.random.default_rng(d)
    inputs = random_md(rng, k, (n, d + 1))
    inputs[:, ::3] *= 2.0 ** -np.minimum(5 * np.arange(d + 1), 900)  # sums on grids of their own
    C = torch.from_numpy(random_md(rng, k, (len(supports) + 1, d + 1))).cuda()
    Z = torch.from_numpy(np.ascontiguousarray(inputs)).cuda()
    whole = pes.Plan(supports, n, d, k, exponents=ex, with_vjp=False, **opts)
    v0, g0 = whole.eval_grad(C, Z)
    whole.check()
    name = opts.get("arith", "auto")
    assert whole.arith() == (pes.auto_arith(supports, d, k) if name == "auto" else name)
    shards = [ShardPlan(supports, n, d, k, world, r, exponents=ex, **opts) for r in range(world)]
    grids = [s.plan.partial_grids(s.coeff_of(C), Z).clone() for s in shards]
    common = grids[0]
    for g in grids[1:]:
        common = torch.maximum(common, g)
    accs = [s.plan.partial_sums(common).clone() for s in shards]
    total = sum(accs[1:], accs[0].clone())
    for s in shards:
        v, g = s.plan.round_sums(common, total)
        s.plan.check()
        assert torch.equal(v, v0) and torch.equal(g, g0)
    hv, hg = combine_host(k, n, d, [(common.cpu().numpy(), a.cpu().numpy()) for a in accs], arith=whole.arith())
    assert np.array_equal(hv, v0.cpu().numpy()) and np.array_equal(hg, g0.cpu().numpy())
