"""The group mode's pool kernels treat every group alike, whatever else the call
holds: a group's values, errors, region counts and statuses are bit for bit those
of a call of its own, from a handful of regions to deep partitions (the deep
slots' route starts above 1,024 regions) and from one slot to more than the
single-block scan takes (8,192)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _call(ctx, torch, kind, T, q, rel_tol, **kw):
    from paper_1610_09991_gb300 import workloads as W
    lm = torch.as_tensor(W.all_pairs(9), dtype=torch.int32, device="cuda")
    b = dict(kind=kind, T=T, q=torch.as_tensor(np.ascontiguousarray(q), device="cuda"), lm=lm,
             rel_tol=rel_tol)
    (r,) = ctx.integrate_multi([b], **kw)
    return [x.reshape(len(q), -1).cpu() for x in (r.values, r.errors, r.regions, r.status)]


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("T,rel_tol,nq,deep", [(0.01, 1e-6, 5, True), (0.2, 1e-6, 13, False),
                                              (0.05, 1e-5, 20, False)])
def test_a_group_is_the_same_alone_and_among_others(mode, T, rel_tol, nq, deep):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    q = W.q_grid_bz(nq)
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=mode, rule_n=8, cover=1.0, eval_fp32=1)
    for kind in (P.PH, P.PP):
        every = _call(ctx, torch, kind, T, q, rel_tol)
        assert int(every[3].max()) == 0
        assert int(every[2].max()) > 1024 or not deep
        order = np.argsort(every[2][:, 0].numpy())
        for i in sorted({0, *order[:2], *order[-3:], len(q) // 2}):
            one = _call(ctx, torch, kind, T, q[i:i + 1], rel_tol)
            for a, b in zip(every, one):
                assert torch.equal(a[i], b[0]), (kind, i)
    ctx.close()


@pytest.mark.parametrize("n", [1023, 1025, 8192, 8193])
def test_slot_counts_around_the_scan_blocks(n):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    q = np.random.default_rng(n).uniform(-np.pi, np.pi, (n, 2))
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, rule_n=4, cover=1.0, eval_fp32=1)
    every = _call(ctx, torch, P.PH, 1.0, q, 1e-2, pool_capacity=64 * n)
    for i in (0, 1022, n - 1):
        one = _call(ctx, torch, P.PH, 1.0, q[i:i + 1], 1e-2)
        for a, b in zip(every, one):
            assert torch.equal(a[i], b[0]), i
    ctx.close()


@pytest.mark.parametrize("capacity", [None, 40000])
@pytest.mark.parametrize("fp32", [1, 0])
def test_groups_that_share_their_first_energy(capacity, fp32):
    """400 groups a batch and rounds of more than 6,000 regions: x1 and exp(-|x1|) come
    from tables keyed by temperature and region.  Two temperatures, both kinds and the
    test kind in one call, and a pool whose tables run out of room."""
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    lm = torch.as_tensor(W.all_pairs(9)[::4], dtype=torch.int32, device="cuda")
    q = torch.as_tensor(W.q_grid_bz(20), device="cuda")
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, rule_n=12, cover=1.0, eval_fp32=fp32)
    bs = [dict(kind=k, T=T, q=q, lm=lm, rel_tol=1e-5)
          for T in (0.05, 0.06) for k in (P.PH, P.PP)] + [dict(kind=P.OVERLAP, T=0.05, q=q, lm=lm)]
    every = ctx.integrate_multi(bs, pool_capacity=capacity)
    assert ctx.last_rc == 0
    for b, r in zip(bs, every):
        for i in (0, 1, 77, 210, 399):
            one = ctx.integrate_batch(b["kind"], q[i:i + 1].contiguous(), lm, b["T"],
                                      b.get("rel_tol", 1e-6))
            for x in ("values", "errors", "regions", "status"):
                got = getattr(r, x).reshape(400, -1)[i]
                assert torch.equal(got, getattr(one, x)), (b["kind"], b["T"], i, x)
    ctx.close()
