"""The full-size polynomials on the tensor cores, which a plan takes by default, and on the
integer pipe: the same values and derivatives to 2^24 above the last bit of a k-double (both
forms drop at most 2^-(53 k - 1) of the product of the largest coefficients per product)."""
import numpy as np
import pytest

from paper_2101_10881_gb300 import pes, synth
from tests.exact import normwise_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [synth.config1, synth.config2], ids=["p2 k=10 d=152", "p3 k=4 d=152"])
def test_full_size_forms_agree(make):
    import torch
    pes.build()
    prob = make()
    C, Z = torch.from_numpy(prob.coeff).cuda(), torch.from_numpy(prob.inputs).cuda()
    got = []
    for arith in ("auto", "int"):
        plan = pes.Plan(prob.supports, prob.n, prob.d, prob.k, arith=arith)
        assert plan.arith() == ("tensor" if arith == "auto" else "int")
        v, g = plan.eval_grad(C, Z)
        gi, gc = plan.vjp(C, Z, v, reuse_forward=True)
        plan.check()
        got.append([t.cpu().numpy() for t in (v, g[:, ::16], gi[:, ::16], gc[:, :: max(1, prob.N // 8)])])
        del plan
    for a, b in zip(*got):
        assert normwise_err(np.ascontiguousarray(a), np.ascontiguousarray(b)) <= 2.0 ** -(53 * prob.k - 24)
