"""The sums over tokens of the low-rank gradients, where a CTA adds several chunks up: each chunk is added in fp32,
so a chunk 2^20 below the sum so far still counts."""
import pytest
import torch

from paper_2609_06712_gb300 import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [16, 32, 64])
def test_a_small_chunk_after_a_large_one(r):
    from paper_2609_06712_gb300 import rola as rl
    # 40 heads of 92 chunks: a CTA takes two consecutive chunks of a head.  No feature map and no rotation, so
    # dP_k[a] = sum_t (dC[a] . v_t) k_t with dC and dC . v_t in bf16
    H, nB = 40, 92
    cfg = configs.get("tiny", T=nB, Hh=8, Ww=8, H=H, keep=0.5 / nB, r=r, lowrank_act="identity", lowrank_rope=2)
    N = cfg["N"]
    g = torch.Generator(device="cuda").manual_seed(r)
    q, k, v, dO = (torch.zeros((1, H, N, 128), dtype=torch.bfloat16, device="cuda") for _ in range(4))
    q[..., 2:] = 0.1 * torch.randn((1, H, N, 126), generator=g, device="cuda").bfloat16()
    dO.copy_(torch.randn(dO.shape, generator=g, device="cuda"))
    # v along one axis and k along another, in powers of two: every product and chunk sum is exact
    v[:, :, :64, 7], k[:, :, :64, 0] = 2.0 ** 10, 2.0 ** 10          # 64 tokens of 2^20: 2^26 in all
    v[:, :, 64:128, 7], k[:, :, 64:128, 0] = 1.0, 1.0                # 64 in all
    k[:, :, 0, 1] = 1.0                                              # token 0 alone: 2^10
    P_q, P_k = (torch.randn((H, r, 128), generator=g, device="cuda").bfloat16() for _ in range(2))
    C = torch.randn((1, H, r, 128), generator=g, device="cuda")
    kv = torch.arange(nB, dtype=torch.int32, device="cuda").expand(1, H, nB).contiguous()
    lse = torch.full((1, H, N), 5.0, device="cuda")
    c = rl.make_config(cfg)
    assert rl.num_keep(c) == 1
    out = [torch.empty_like(q) for _ in range(3)] + [torch.empty((H, r, 128), device="cuda") for _ in range(2)]
    ws = rl.backward_workspace(c)
    rl.backward(c, q, k, v, P_q, P_k, None, kv, torch.zeros_like(q), lse, C, dO, *out, None, ws)
    torch.cuda.synchronize()
    assert rl.get_device_status(ws) == rl.ROLA_OK
    dP_k = out[4].double()
    unit = dP_k[..., 1] / 2.0 ** 10                                  # dC[a] . e_7 in bf16
    assert (unit != 0).float().mean() > 0.9
    want = unit * (2.0 ** 26 + 64)
    # one rounding to 24 bits; without the small chunk the sum is off by 2^-20
    assert ((dP_k[..., 0] - want).abs() <= 2.0 ** -23 * want.abs()).all()
