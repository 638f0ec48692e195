"""One partition per (kind, q): groups of a large call read the first energy's half of
the kernel F from tables of the regions that they meet at the same temperature.  A
group's result must not depend on that: bit for bit what a call too small to share
gives, also when most regions are met once and the tables run out of room."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(torch, ctx, batches, **kw):
    out = ctx.integrate_multi(batches, **kw)
    assert ctx.last_rc == 0
    return [[x.cpu() for x in (r.values, r.errors, r.regions, r.status)] for r in out]


@pytest.mark.parametrize("many", [False, True])
@pytest.mark.parametrize("rule_n", [6, 12])
@pytest.mark.parametrize("fp32", [0, 1])
def test_a_group_is_the_same_in_a_small_and_a_large_call(fp32, rule_n, many):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    lmd = torch.as_tensor(W.all_pairs(9), dtype=torch.int32, device="cuda")
    rel = 1e-6 if rule_n == 12 else 1e-5
    if many:   # a temperature of its own for every four groups
        q = torch.as_tensor(W.q_grid_bz(2), device="cuda")
        batches = [dict(kind=P.PP if i % 2 else P.PH, T=float(T), q=q, lm=lmd, rel_tol=rel)
                   for i, T in enumerate(np.geomspace(0.05, 0.2, 40))]
    else:
        q = torch.as_tensor(W.q_grid_bz(6), device="cuda")
        batches = [dict(kind=k, T=T, q=q, lm=lmd, rel_tol=rel)
                   for k in (P.PH, P.PP) for T in (0.05, 0.09)]
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, eval_fp32=fp32, rule_n=rule_n, cover=1.0)
    every = _run(torch, ctx, batches, pool_capacity=60000 if many and rule_n == 12 else None)
    for b, got in zip(batches, every):
        nq, step = len(q), 18
        for i in range(0, nq, step):
            (one,) = _run(torch, ctx, [dict(b, q=q[i:i + step].contiguous())])
            for x, y in zip(got, one):
                x = x.reshape(nq, -1)[i:i + step].reshape(-1)
                assert torch.equal(torch.nan_to_num(x.double()), torch.nan_to_num(y.double())), b["T"]
    ctx.close()
