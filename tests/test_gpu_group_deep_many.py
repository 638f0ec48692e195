"""More groups than the single-block scan takes (8,192), a few of them deep (their sums
go another way above 1,024 regions): every group is bit for bit what it is alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8100, 8300])
def test_deep_groups_among_many(n):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    lm = torch.as_tensor(W.all_pairs(9)[:5], dtype=torch.int32, device="cuda")
    rng = np.random.default_rng(n)
    q = [torch.as_tensor(rng.uniform(-np.pi, np.pi, (m, 2)), device="cuda") for m in (n, 3)]
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, rule_n=4, cover=1.0, eval_fp32=1)
    b = [dict(kind=P.PH, T=1.0, q=q[0], lm=lm, rel_tol=1e-2),
         dict(kind=P.PP, T=0.02, q=q[1], lm=lm, rel_tol=1e-6)]
    many, deep = ctx.integrate_multi(b, pool_capacity=1500000)
    assert ctx.last_rc == 0 and int(deep.regions.max()) > 1024
    for r, k, i in ((many, 0, 0), (many, 0, n - 1), (deep, 1, 0), (deep, 1, 2)):
        one = ctx.integrate_multi([dict(b[k], q=q[k][i:i + 1].contiguous())])[0]
        for x in ("values", "errors", "regions", "status"):
            assert torch.equal(getattr(r, x).reshape(len(q[k]), -1)[i], getattr(one, x)), (k, i, x)
    ctx.close()
