"""Job tables wide enough for the tensor cores (mma_takes): the smallest degree of each k,
ragged column tiles, parts, tiles and degrees beyond whole series, forward and backward,
against the oracle within the tolerance of the other paths, and the same bits from every
shape.  Half of the variables are exponential-like (magnitudes falling as 1/j!, terms on
grids far apart), one of them with zero coefficients, one identically zero."""
import itertools
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2101_10881_gb300 import pes
from paper_2101_10881_gb300.synth import random_md
from tests.exact import TOL, normwise_err

pytestmark = pytest.mark.gpu

# k, d, n (all pairs of n variables), shapes that must give the same bits
CASES = [(10, 56, 48, [{"split": 2}]), (8, 72, 38, [{"staging": 2}]), (4, 136, 27, [{"threads": 64}]),
         (5, 256, 16, [{"split": 4}]), (10, 95, 28, [{"tile": 48}, {"threads": 32}]), (4, 200, 20, [{"tile": 16}]),
         (8, 127, 22, [{"split": 16}]), (10, 480, 8, []), (4, 1000, 6, [])]


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    pes.build()
    assert _t.cuda.is_available()
    return _t


@pytest.mark.parametrize("k,d,n,shapes", CASES)
def test_wide_tables_match_oracle(torch, k, d, n, shapes):
    rng = np.random.default_rng(7 * k + d)
    supp = [list(s) for s in itertools.combinations(range(n), 2)]
    coeff = random_md(rng, k, (len(supp) + 1, d + 1))
    inputs = random_md(rng, k, (n, d + 1))
    fall = np.array([2.0 ** -min(300, int(math.lgamma(j + 1) / math.log(2))) for j in range(d + 1)])
    inputs[:, n // 2:] *= fall
    inputs[:, n - 2, 1::3] = 0.0
    inputs[:, 0] = 0.0
    u = random_md(rng, k, (d + 1,))
    C, Z, U = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (coeff, inputs, u))
    plan = pes.Plan(supp, n, d, k)
    v, g = plan.eval_grad(C, Z)
    gi, gc = plan.vjp(C, Z, U, reuse_forward=True)
    plan.check()
    # (the series take other words in the workspace than the integer pipe's)
    other = pes.Plan(supp, n, d, k, arith="int")
    assert plan.info()["workspace_bytes"] != other.info()["workspace_bytes"]
    rv, rg = O.eval_grad(supp, n, coeff, inputs)
    ri, rc = O.vjp(supp, n, coeff, inputs, u)
    for got, ref in ((v, rv), (g, rg), (gi, ri), (gc, rc)):
        assert normwise_err(got.cpu().numpy(), ref) <= TOL[k]
    for opts in shapes:
        plan = pes.Plan(supp, n, d, k, **opts)
        v2, g2 = plan.eval_grad(C, Z)
        gi2, gc2 = plan.vjp(C, Z, U, reuse_forward=True)
        plan.check()
        for a, b in ((v, v2), (g, g2), (gi, gi2), (gc, gc2)):
            assert torch.equal(a, b), opts
