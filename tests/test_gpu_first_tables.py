"""Group mode: the first-energy tables are built where the regions of a round repeat
often enough and the pool has room for them, and left out elsewhere; a group's result
is the same bit for bit either way.  paid_last_sharing shows which way a call went.
The calls start at the uniform level 4 and end after one round, so that their entries,
and how many of them are distinct, are known exactly: 256 regions a group, distinct by
temperature."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

#: temperatures and groups at each of them (momenta), per batch
EVERY = [(T, 1) for T in np.linspace(0.05, 0.2, 40)]


def _batches(torch, P, W, spec, npairs=7):
    lm = torch.as_tensor(W.all_pairs(9)[:npairs], dtype=torch.int32, device="cuda")
    rng = np.random.default_rng(len(spec))
    return [dict(kind=P.PP if i % 2 else P.PH, T=float(T), lm=lm, rel_tol=0.0, abs_tol=1e9,
                 q=torch.as_tensor(rng.uniform(-3, 3, (nq, 2)), device="cuda"))
            for i, (T, nq) in enumerate(spec)]


def _call(ctx, batches, **kw):
    out = ctx.integrate_multi_seeded(batches, None, 1.0, **kw)
    assert ctx.last_rc == 0 and ctx.last_stats()["rounds"] == 1
    return [[x.cpu() for x in (r.values, r.errors, r.regions, r.status)] for r in out]


def _check(torch, ctx, batches, got):
    """every group against calls of at most 20 groups, too small for tables"""
    for b, r in zip(batches, got):
        nq = len(b["q"])
        for i in sorted({0, nq // 2, max(0, nq - 20)}):
            part = dict(b, q=b["q"][i:i + 20].contiguous())
            (one,) = _call(ctx, [part])
            assert ctx.last_sharing()["rounds"] == ctx.last_sharing()["skipped"] == 0
            for x, y in zip(r, one):
                assert torch.equal(x.reshape(nq, -1)[i:i + 20].reshape(-1), y), b["T"]


@pytest.mark.parametrize("fp32,rule_n,spec,want", [
    # one group at each temperature: nothing can repeat, no passes over the list
    (1, 12, [(T, 1) for T in np.linspace(0.05, 0.2, 160)], "none"),
    (0, 12, EVERY, "none"),
    # four at each: the least that pays at N = 12 on the FP32 pipe; eight at N = 8
    (1, 12, [(T, 4) for T in np.linspace(0.05, 0.2, 40)], "tables"),
    (1, 10, [(T, 2) for T in (0.05, 0.1, 0.15, 0.2)] * 40, "tables"),
    (1, 8, [(T, 4) for T in np.linspace(0.05, 0.2, 40)], "none"),
    (1, 8, [(T, 8) for T in np.linspace(0.05, 0.2, 20)], "tables"),
    (1, 6, [(T, 16) for T in np.linspace(0.05, 0.2, 10)], "tables"),
    (1, 4, [(0.1, 160)], "none"),          # N = 4: never on the FP32 pipe
    (0, 12, [(T, 2) for T in np.linspace(0.05, 0.2, 20)], "tables"),
    (0, 4, [(T, 2) for T in np.linspace(0.05, 0.2, 20)], "tables"),
    # one temperature with many groups among single ones: counted, and not enough
    (1, 12, EVERY * 1 + [(T, 1) for T in np.linspace(0.3, 0.4, 80)] + [(0.25, 20)], "skipped"),
    (0, 12, EVERY + [(0.25, 8)], "skipped"),
    # ... and enough; the test kind among them shares nothing
    (1, 12, EVERY + [(0.25, 260)], "tables"),
    (0, 8, EVERY + [(0.25, 80)], "tables"),
])
def test_tables_where_regions_repeat(fp32, rule_n, spec, want):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, eval_fp32=fp32, rule_n=rule_n)
    batches = _batches(torch, P, W, spec)
    got = _call(ctx, batches)
    s = ctx.last_sharing()
    n, d = 256 * sum(m for _, m in spec), 256 * len({T for T, _ in spec})
    assert n > 6000
    if want == "tables":
        assert s == dict(rounds=1, entries=n, distinct=d, unplaced=0, roomless=0, skipped=0), s
    else:
        assert (s["rounds"], s["skipped"]) == (0, int(want == "skipped")), s
    _check(torch, ctx, batches, got)
    ctx.close()


@pytest.mark.parametrize("fp32", [0, 1])
def test_entries_that_cannot_share_do_not_count(fp32):
    """the overlap kind's regions are no repeats of anything: 40 temperatures with two
    groups each stay below the FP32 pipe's line and above FP64's, whatever is beside"""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, eval_fp32=fp32, rule_n=12)
    batches = _batches(torch, P, W, [(T, 2) for T in np.linspace(0.05, 0.2, 40)] + [(0.07, 8)])
    over = dict(_batches(torch, P, W, [(0.1, 600)])[0], kind=P.OVERLAP)
    got = _call(ctx, batches + [over])
    s = ctx.last_sharing()
    assert (s["rounds"], s["skipped"]) == ((0, 1) if fp32 else (1, 0)), s
    if not fp32:
        assert (s["entries"], s["distinct"]) == (256 * 88, 256 * 41), s
    _check(torch, ctx, batches, got)
    ctx.close()


@pytest.mark.parametrize("fp32,rule_n", [(0, 12), (1, 12), (0, 4)])
def test_a_pool_without_room_for_the_tables(fp32, rule_n):
    """N = 12: 10,400 bytes of tables a distinct region, 972 bytes of room a region of
    the pool; the distinct regions of one temperature's 256 fit in 2,740, 40 times as
    many in 109,600."""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, eval_fp32=fp32, rule_n=rule_n)
    block = 32 * (rule_n + 1) * (2 * rule_n + 1)
    batches = _batches(torch, P, W, [(T, 8) for T in np.linspace(0.05, 0.2, 40)])
    n, d = 256 * 320, 256 * 40
    need = -(-d * block // 972) + 40   # both vector arrays hold whole blocks
    for cap, room in ((max(n, need), True), (n, n >= need)):
        got = _call(ctx, batches, pool_capacity=cap)
        s = ctx.last_sharing()
        assert s["rounds"] == int(room) and s["skipped"] == 1 - int(room), (cap, s)
        assert s["roomless"] == 0
        _check(torch, ctx, batches, got)
    ctx.close()


def test_entries_whose_probes_run_out():
    """a pool just below a power of two halves the hash table, two thirds of whose
    places are then taken: some entries find none within 32 probes and are evaluated
    whole"""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, eval_fp32=0, rule_n=4)
    spec = [(T, 1 + i % 2) for i, T in enumerate(np.linspace(0.05, 0.2, 170))]   # 255 groups
    batches = _batches(torch, P, W, spec, npairs=2)
    got = _call(ctx, batches, pool_capacity=65535)
    s = ctx.last_sharing()
    assert s["rounds"] == 1 and s["entries"] == 255 * 256 and s["unplaced"] > 0, s
    assert s["distinct"] <= 170 * 256
    _check(torch, ctx, batches[:4] + batches[-4:], got[:4] + got[-4:])
    ctx.close()


@pytest.mark.parametrize("fp32", [0, 1])
def test_the_allocation_free_call_shares_too(fp32):
    """paid_integrate_batch_static decides as the other entry points do"""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, eval_fp32=fp32, rule_n=12, cover=1.0)
    q = torch.as_tensor(W.q_grid_bz(28), device="cuda")
    lm = torch.as_tensor(W.all_pairs(9)[:5], dtype=torch.int32, device="cuda")
    r = ctx.integrate_batch_static(P.PP, q, lm, 0.3, 1e-4)
    assert ctx.last_rc == 0 and ctx.last_sharing()["rounds"] > 0
    for i in (0, 100, 764):
        one = ctx.integrate_batch_static(P.PP, q[i:i + 20].contiguous(), lm, 0.3, 1e-4)
        assert ctx.last_sharing()["rounds"] == 0
        for x in ("values", "errors", "regions", "status"):
            got = getattr(r, x).reshape(784, -1)[i:i + 20].reshape(-1)
            assert torch.equal(got, getattr(one, x)), x
    ctx.close()
