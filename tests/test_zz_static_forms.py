"""pes_eval_grad_static holds its series in the form a plan takes (tensor cores for wide
tables) while they fit the 64 MiB array, and in the integer pipe's shorter form when only
that fits: what fits the array as 28-bit digits is never refused."""
import numpy as np
import pytest

from paper_2101_10881_gb300 import pes, synth
from paper_2101_10881_gb300.synth import random_md
from tests.test_zz_no_alloc import outputs, static_call, static_rc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    pes.build()
    assert _t.cuda.is_available()
    return _t


# random monomials of 4 of 64 variables: 10 series each, beside a_0 and the inputs
@pytest.mark.parametrize("k,d,N,form", [(8, 95, 560, "auto"), (8, 95, 700, "int"), (4, 152, 700, "int"),
                                        (5, 256, 400, "int"), (8, 95, 900, None)])
def test_static_takes_the_longest_form_that_fits(torch, k, d, N, form):
    rng = np.random.default_rng(N)
    n = 64
    supp = [sorted(int(v) for v in rng.choice(n, 4, replace=False)) for _ in range(N)]
    coeff, inputs = random_md(rng, k, (N + 1, d + 1)), random_md(rng, k, (n, d + 1))
    prob = synth.Problem("static", n, d, k, supp, coeff, inputs)
    C, Z = torch.from_numpy(coeff).cuda(), torch.from_numpy(inputs).cuda()
    v, g = outputs(torch, prob)
    if form is None:
        assert static_rc(torch, prob, C, Z, v, g) == 7
        return
    sv, sg = static_call(torch, prob, C, Z, v, g)
    plan = pes.Plan(supp, n, d, k, with_vjp=False, arith=form)
    pv, pg = plan.eval_grad(C, Z)
    plan.check()
    assert np.array_equal(sv, pv.cpu().numpy()) and np.array_equal(sg, pg.cpu().numpy())
