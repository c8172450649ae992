"""A plan, batch or single rank whose series fit the device memory as 28-bit digits only is built for the
integer pipe, where the automatic arithmetic would take the longer series of the tensor cores."""
import itertools

import pytest

from paper_2101_10881_gb300 import pes
from paper_2101_10881_gb300.shard import ShardPlan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    pes.build()
    assert _t.cuda.is_available()
    return _t


@pytest.mark.parametrize("kind", ["plan", "batch", "rank"])
def test_falls_back_to_the_integer_pipe(torch, kind):
    batch = kind == "batch"
    k, d, n = 5, 270, 200
    supp = [list(s) for s in itertools.combinations(range(n), 2)]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    series = []
    for rows in (len(supp) + 1, n):
        a = torch.zeros((k, rows, d + 1), dtype=torch.float64, device="cuda")
        a[0] = torch.rand(a.shape[1:], generator=gen, dtype=torch.float64, device="cuda") - 0.5
        series.append(a.reshape(-1) if batch else a)

    def build(arith):
        if batch:
            return pes.Batch([(supp, n, d)], k, arith=arith)
        if kind == "rank":
            return ShardPlan(supp, n, d, k, 1, 0, arith=arith).plan
        return pes.Plan(supp, n, d, k, with_vjp=False, arith=arith)

    v, g = (torch.empty((k, rows, d + 1), dtype=torch.float64, device="cuda") for rows in (1, n))
    v, g = (v.reshape(-1), g.reshape(-1)) if batch else (v[:, 0].contiguous(), g)
    plan = build("int")
    plan.eval_grad(*series, v, g)
    plan.check()
    want = (v.clone(), g.clone())
    short = plan.info()["workspace_bytes"]
    del plan
    plan = build("auto")
    long = plan.info()["workspace_bytes"]
    del plan
    assert long > 1.5 * short > 1.5e9
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    rest = torch.empty(free - (short + long) // 2, dtype=torch.uint8, device="cuda")
    try:
        plan = build("auto")
        assert plan.info()["workspace_bytes"] == short
        plan.eval_grad(*series, v, g)
        plan.check()
        assert torch.equal(v, want[0]) and torch.equal(g, want[1])
    finally:
        del rest
        torch.cuda.empty_cache()
