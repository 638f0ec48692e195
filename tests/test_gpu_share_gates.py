"""One partition per integral: F is read from the tables where the pairs of a q repeat
the regions of a round often enough, and evaluated in place elsewhere; an integral's
result is the same bit for bit either way.  paid_last_sharing shows which way a call
went.  Calls that start at the uniform level 4 and end after one round have 256
regions an integral, distinct by q."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _batch(torch, W, kind, nq, pairs, T=0.1, rel_tol=0.0, abs_tol=1e9, seed=0):
    lm = W.all_pairs(9)[np.random.default_rng(seed).permutation(81)[:pairs]]
    q = np.random.default_rng(seed + 1).uniform(-3, 3, (nq, 2))
    return dict(kind=kind, T=T, q=torch.as_tensor(q, device="cuda"), rel_tol=rel_tol,
                lm=torch.as_tensor(lm, dtype=torch.int32, device="cuda"), abs_tol=abs_tol)


def _call(ctx, batches, seeded=True, **kw):
    out = (ctx.integrate_multi_seeded(batches, None, 1.0, **kw) if seeded
           else ctx.integrate_multi(batches, **kw))
    assert ctx.last_rc == 0
    return [[x.cpu() for x in (r.values, r.errors, r.regions, r.status)] for r in out]


def _check(torch, ctx, batches, got, seeded=True):
    """every pair against a call of its own, in which nothing can share"""
    for b, r in zip(batches, got):
        nq, pairs = len(b["q"]), len(b["lm"])
        for p in range(pairs):
            (one,) = _call(ctx, [dict(b, lm=b["lm"][p:p + 1].contiguous())], seeded)
            assert not any(ctx.last_sharing().values())
            for x, y in zip(r, one):
                assert torch.equal(x.reshape(nq, pairs)[:, p], y), p


@pytest.mark.parametrize("rule_n", [4, 6])
@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("pairs,nq", [(2, 3), (2, 200), (3, 70), (9, 30)])
def test_pairs_of_a_q_share(fp32, rule_n, pairs, nq):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, eval_fp32=fp32, rule_n=rule_n)
    b = [_batch(torch, W, P.PP, nq, pairs)]
    got = _call(ctx, b, pool_capacity=40000 * nq * pairs)   # room for every distinct region
    assert ctx.last_sharing() == dict(rounds=1, entries=256 * nq * pairs, distinct=256 * nq,
                                      unplaced=0, roomless=0, skipped=0)
    _check(torch, ctx, b, got)
    ctx.close()


@pytest.mark.parametrize("rule_n", [4, 6])
@pytest.mark.parametrize("fp32", [0, 1])
def test_single_pairs_and_test_kinds_stay_out(fp32, rule_n):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, eval_fp32=fp32, rule_n=rule_n)
    b = [_batch(torch, W, P.PH, 1, 2), _batch(torch, W, P.PP, 300, 1, seed=5),
         _batch(torch, W, P.OVERLAP, 4, 3, seed=6)]
    got = _call(ctx, b)
    # less than a quarter of the integrals beside another pair: no passes
    assert not any(ctx.last_sharing().values())
    _check(torch, ctx, b, got)
    # the test kind's regions share nothing and do not count
    b = [_batch(torch, W, P.PH, 20, 4), _batch(torch, W, P.OVERLAP, 20, 4, seed=6),
         _batch(torch, W, P.PP, 20, 1, seed=5)]
    got = _call(ctx, b, pool_capacity=40000 * 180)
    s = ctx.last_sharing()
    assert (s["rounds"], s["entries"], s["distinct"]) == (1, 256 * 100, 256 * 40), s
    _check(torch, ctx, b, got)
    ctx.close()


@pytest.mark.parametrize("rule_n", [4, 6])
@pytest.mark.parametrize("fp32", [0, 1])
def test_a_pool_without_room_for_the_tables(fp32, rule_n):
    """room for F of (2 capacity - entries / 2) / nodes distinct regions: for all of
    them, for more than half (the rest in place), for less (all in place)"""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, eval_fp32=fp32, rule_n=rule_n)
    b = [_batch(torch, W, P.PH, 32, 2)]
    n, d, nodes = 256 * 64, 256 * 32, (2 * rule_n + 1) ** 2
    for part, rounds in ((1.1, 1), (0.7, 1), (0.3, 0)):
        cap = int((part * d * nodes + n / 2) / 2)
        got = _call(ctx, b, pool_capacity=max(n, cap))
        s = ctx.last_sharing()
        assert (s["rounds"], s["skipped"]) == (rounds, 1 - rounds), (part, s)
        assert (s["roomless"] > 0) == (part == 0.7), (part, s)
        _check(torch, ctx, b, got)
    ctx.close()


@pytest.mark.parametrize("nq,skipped", [(13, 1), (40, 0)])
def test_rounds_of_few_repeats_leave_the_tables_out(nq, skipped):
    """N = 4, FP32: nq momenta with four pairs beside 144 with one, so that (nq + 144) of
    every (4 nq + 144) regions are distinct: 0.80 with 13, above both classes' lines
    (1/2 and 3/4); 0.61 with 40, below float-float's"""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, eval_fp32=1, rule_n=4)
    b = [_batch(torch, W, P.PH, nq, 4), _batch(torch, W, P.PP, 144, 1, seed=5)]
    got = _call(ctx, b, pool_capacity=40000 * 304)
    s = ctx.last_sharing()
    assert (s["rounds"], s["skipped"]) == (1 - skipped, skipped), s
    _check(torch, ctx, b, got)
    ctx.close()


@pytest.mark.parametrize("pairs,nq,shared", [(2, 256, True), (2, 257, False), (3, 171, False),
                                            (4, 300, True)])
def test_fp32_calls_that_gain_nothing(pairs, nq, shared):
    """N = 4: up to three pairs share F only in calls of at most 512 integrals"""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, eval_fp32=1, rule_n=4)
    b = [_batch(torch, W, P.PH, nq, pairs)]
    got = _call(ctx, b, pool_capacity=40000 * nq * pairs)
    assert (ctx.last_sharing()["rounds"] == 1) == shared
    _check(torch, ctx, b, got)
    ctx.close()
