"""The FP32-pipe group kernel at the edges of its blocks: any count of regions,
any position in the list, every rule order and kind, against the same regions
one by one and against the FP64 group kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

#: regions per block of the kernel (N: R)
BLOCK = {4: 12, 6: 9, 8: 14, 10: 14, 12: 12}


def _regions(n, seed):
    rng = np.random.default_rng(seed)
    level = rng.integers(0, 9, n)
    ij = (rng.random((n, 2)) * 2.0 ** level[:, None]).astype(int)
    return np.concatenate([level[:, None], ij], 1).astype(np.int32)


@pytest.mark.parametrize("N", sorted(BLOCK))
@pytest.mark.parametrize("kind", ["ph", "pp", "overlap", "flow_ph", "flow_pp"])
def test_block_edges_do_not_change_a_region(N, kind):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    k = {"ph": P.PH, "pp": P.PP, "overlap": P.OVERLAP, "flow_ph": P.FLOW_PH,
         "flow_pp": P.FLOW_PP}[kind]
    T = 0.05
    lm = torch.as_tensor(W.all_pairs(9), dtype=torch.int32, device="cuda")
    q = torch.tensor([0.9, -2.1], dtype=torch.float64, device="cuda")
    R = BLOCK[N]
    reg = torch.as_tensor(_regions(3 * R + 2, N), device="cuda")
    opts = dict(ffset=9, group_mode=1, rule_n=N)
    ff = P.Context(*W.LATTICE, eval_fp32=1, **opts)
    d = P.Context(*W.LATTICE, eval_fp32=0, **opts)
    one = [torch.cat(x) for x in zip(*(ff.rule_regions(k, q, lm, T, reg[i:i + 1].contiguous())
                                       for i in range(len(reg))))]
    for n in (1, 2, R - 1, R, R + 1, 2 * R, 3 * R + 2):
        for o in {0, len(reg) - n}:
            got = ff.rule_regions(k, q, lm, T, reg[o:o + n].contiguous())
            for g, r in zip(got, one):
                assert torch.equal(g, r[o:o + n]), (n, o)
    # the float-float values against FP64: 2e-12 (1 + 0.05 / T) of the region's
    # largest pair value (the kernel's documented bound); the flow kernel's
    # three terms cancel by up to 19 (3 + 10 + 6 against 1 at |e| = 0)
    q2, dq = d.rule_regions(k, q, lm, T, reg)
    scale = q2.abs().amax(1, keepdim=True)
    for g, r in zip(one, (q2, dq)):
        rel = 2e-12 * (1 + 0.05 / T) * (19 if kind.startswith("flow") else 1)
        assert ((g - r).abs() <= rel * scale + 1e-20).all()
    ff.close()
    d.close()
