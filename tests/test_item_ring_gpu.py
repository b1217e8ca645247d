"""The persistent sparse kernels hand out their work items through a ring of 16 slots a CTA.  A layer with more
items per CTA than slots, whose key side is nearly all empty (every query block keeps key block 0), lets the
producer run far ahead of the warps that write the empty blocks' gradients."""
import pytest
import torch

from paper_2609_06712_gb300 import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,nB", [(40, 96), (3, 5)])
def test_every_query_block_keeps_block_zero(H, nB):
    from paper_2609_06712_gb300 import rola as rl
    cfg = configs.get("tiny", T=nB, Hh=8, Ww=8, H=H, keep=0.5 / nB, r=16)
    N = cfg["N"]
    g = torch.Generator(device="cuda").manual_seed(nB)
    shape = (1, H, N, 128)
    q, k, v, dO = (torch.randn(shape, generator=g, device="cuda") for _ in range(4))
    q, k = 0.1 * q, 0.1 * k
    q[..., 126] = 4.0                        # the slowest pair: block 0's scores stand out by far
    k[..., 126] = 0.0
    k[:, :, :64, 126] = 4.0
    q, k, v, dO = (t.bfloat16() for t in (q, k, v, dO))
    P = torch.zeros((H, 16, 128), dtype=torch.bfloat16, device="cuda")      # no low-rank part
    c = rl.make_config(cfg)
    assert rl.num_keep(c) == 1 and (H * nB > 16 * 152) == (H == 40)

    def step():
        leaves = [t.clone().requires_grad_() for t in (q, k, v)]
        out = rl.RoLAFunction.apply(c, *leaves, P, P, None)
        return torch.autograd.grad(out, leaves, dO)

    _, dk, dv = step()
    # nothing but block 0 was attended to
    assert (dk[:, :, 64:] == 0).all() and (dv[:, :, 64:] == 0).all()
    # the softmax weights of a query add up to 1, so the columns of dv over block 0 add up to those of dO:
    # each weight and each entry of dv rounds once to 8 bits of mantissa
    got, want = dv[:, :, :64].double().sum(2), dO.double().sum(2)
    tol = 2.0 ** -8 * (dO.double().abs().sum(2) + dv[:, :, :64].double().abs().sum(2))
    assert ((got - want).abs() <= tol).all()
    again = step()
    assert all(torch.equal(a, b) for a, b in zip((dk, dv), again[1:]))
