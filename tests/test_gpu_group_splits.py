"""The two splits of the FP32-pipe group kernel (nodes up to 6,000 regions of a launch,
rows above) with several regions a block and ragged ends: a region's values are bit for
bit those it has in a launch of a few regions, for every rule order and kind, at any
place of the list.  (Launches of a few regions are held to the oracle and to FP64 by
the other tests.)  The lists repeat 97 regions, so that the places in a block vary."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

#: regions per block of the rows split and resident blocks per SM
ROWS = {4: (12, 7), 6: (9, 9), 8: (14, 5), 10: (14, 4), 12: (12, 4)}


@pytest.mark.parametrize("N", sorted(ROWS))
@pytest.mark.parametrize("kind", ["ph", "pp", "overlap", "flow_ph", "flow_pp"])
def test_a_region_is_the_same_in_every_split(N, kind):
    import torch
    from paper_1610_09991_gb300 import paid as P
    from paper_1610_09991_gb300 import workloads as W
    k = {"ph": P.PH, "pp": P.PP, "overlap": P.OVERLAP, "flow_ph": P.FLOW_PH,
         "flow_pp": P.FLOW_PP}[kind]
    R, B = ROWS[N]
    rng = np.random.default_rng(N)
    level = rng.integers(0, 9, 97)
    ij = (rng.random((97, 2)) * 2.0 ** level[:, None]).astype(int)
    base = torch.as_tensor(np.concatenate([level[:, None], ij], 1).astype(np.int32), device="cuda")
    lm = torch.as_tensor(W.all_pairs(9), dtype=torch.int32, device="cuda")
    q = torch.tensor([0.9, -2.1], dtype=torch.float64, device="cuda")
    ctx = P.Context(*W.LATTICE, ffset=9, group_mode=1, rule_n=N, eval_fp32=1)
    one = [torch.cat(x) for x in zip(*(ctx.rule_regions(k, q, lm, 0.05, base[i:i + 1].contiguous())
                                       for i in range(97)))]
    # nodes: one, two and more regions a block, the last block short; rows: its edges
    for n in (152 * B - 1, 152 * B + 1, 2 * 152 * B + 1, 5999, 6000, 6001, 6000 + R - 1, 6000 + R,
              6000 + R + 1, 152 * B * R + 1):
        at = torch.arange(n, device="cuda") % 97
        got = ctx.rule_regions(k, q, lm, 0.05, base[at].contiguous())
        for g, r in zip(got, one):
            assert torch.equal(g, r[at]), n
    ctx.close()
