"""One partition per integral: the kernel F is evaluated once for all pairs of a q
that meet a region.  An integral's result must not depend on that: bit for bit what
a call with its pair alone gives (nothing is shared there), whatever the pool's size
(a tight pool has no room for part of the shared values) and beside other kinds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(torch, ctx, batches, **kw):
    out = ctx.integrate_multi(batches, **kw)
    assert ctx.last_rc == 0
    return [[x.cpu() for x in (r.values, r.errors, r.regions, r.status)] for r in out]


@pytest.mark.parametrize("rule_n", [4, 6])
@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("tight", [False, True])
def test_an_integral_is_the_same_alone_and_shared(rule_n, fp32, tight):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    rng = np.random.default_rng(rule_n + 10 * fp32)
    q = torch.as_tensor(np.concatenate([rng.uniform(-3, 3, (3, 2)), [[0.0, 0.0]]]), device="cuda")
    lm = W.all_pairs(9)[[0, 1, 9, 10, 20, 30, 44, 57, 66, 73, 80]]
    lm = np.concatenate([lm, [[3, 12]]])       # an invalid pair
    lmd = torch.as_tensor(lm, dtype=torch.int32, device="cuda")
    ctx = P.Context(*W.LATTICE, ffset=9, rule_n=rule_n, cover=1.0, eval_fp32=fp32)
    kinds = (P.PH, P.PP, P.OVERLAP)
    batches = [dict(kind=k, T=0.2, q=q, lm=lmd) for k in kinds]
    n = len(q) * len(lm) * len(kinds)
    every = _run(torch, ctx, batches, pool_capacity=300 * n if tight else None)
    for k, got in zip(kinds, every):
        got = [x.reshape(len(q), len(lm)) for x in got]
        for p in range(len(lm)):
            (one,) = _run(torch, ctx, [dict(kind=k, T=0.2, q=q, lm=lmd[p:p + 1].contiguous())])
            for a, b in zip(got, one):
                assert torch.equal(torch.nan_to_num(a[:, p].double()),
                                   torch.nan_to_num(b.double())), (k, p)
    ctx.close()


@pytest.mark.parametrize("init_level", [0, 1, 3])
def test_start_levels(init_level):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    q = torch.as_tensor(W.q_grid_bz(2), device="cuda")
    lmd = torch.as_tensor(W.all_pairs(9)[::5], dtype=torch.int32, device="cuda")
    ctx = P.Context(*W.LATTICE, ffset=9, init_level=init_level)
    (every,) = _run(torch, ctx, [dict(kind=P.PP, T=0.3, q=q, lm=lmd)])
    for p in range(len(lmd)):
        (one,) = _run(torch, ctx, [dict(kind=P.PP, T=0.3, q=q, lm=lmd[p:p + 1].contiguous())])
        for a, b in zip(every, one):
            assert torch.equal(a.reshape(len(q), -1)[:, p], b), p
    ctx.close()
