"""The proposal network's kernels at the edges of their tiles and clusters: a row's
output does not depend on how many rows a call has (128 rows a CTA; clusters of 8, 4,
2 and 1 CTAs from 1, 2,049, 4,865 and 9,729 rows), an input that allows no 16-byte
loads gives the same bits, and gradients of ragged row counts match FP64."""
import pytest

pytestmark = pytest.mark.gpu


def _rows(torch, n, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((n, 32), generator=g, device="cuda").to(torch.bfloat16)
    t = torch.randn((n, 256), generator=g, device="cuda")
    return x, t


def test_a_row_is_the_same_in_calls_of_any_size():
    import torch
    from paper_1610_09991_gb300 import paid as P
    net = P.Proposal(seed=3)
    x, _ = _rows(torch, 9729)
    want = net.forward(x)
    assert torch.isfinite(want).all()
    for n in (1, 127, 128, 129, 2048, 2049, 4864, 4865, 9728):
        assert torch.equal(net.forward(x[:n].contiguous()), want[:n]), n


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 65, 777, 1024, 1025, 2049])
def test_gradients_of_ragged_row_counts(n):
    import torch
    from paper_1610_09991_gb300 import paid as P
    net = P.Proposal(seed=4)
    x, t = _rows(torch, n, n)
    g, loss = net.grad(x, t)
    g, loss = g.clone(), float(loss)
    # the same rows two bytes off any 16-byte boundary
    y = torch.empty(n * 32 + 1, dtype=torch.bfloat16, device="cuda")[1:].view(n, 32)
    y.copy_(x)
    if n <= 2048:   # more rows are summed with atomics
        assert torch.equal(net.grad(y, t)[0], g)
    p = net.params.double()
    shapes, o, ws = [(32, 256)] + [(256, 256)] * 4, 0, []
    for k, m in shapes:   # BF16 weights, FP32 biases
        ws += [p[o:o + k * m].view(k, m).float().bfloat16().double().requires_grad_(True),
               p[o + k * m:o + k * m + m].clone().requires_grad_(True)]
        o += k * m + m
    h = x.double()
    for i in range(5):
        h = h @ ws[2 * i] + ws[2 * i + 1]
        if i < 4:
            h = torch.nn.functional.gelu(h)
    ref = (h - t).square().mean()
    want = torch.cat([a.reshape(-1) for a in torch.autograd.grad(ref, ws)])
    # activations and gradients are rounded to BF16 (2^-9) in every layer: the
    # network's tests allow 5 % in the 2-norm
    assert abs(loss - ref.item()) <= 0.01 * ref.item()
    assert (g.double() - want).norm() <= 0.05 * want.norm()
