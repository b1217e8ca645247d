"""Gradients under masks whose query blocks mostly agree: nearly every key block is kept by no query block, and the
few others by one to four, so that a CTA meets work items of a few tiles between long runs of empty ones."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_06712_gb300 import configs
from parity_util import assert_close_grad, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nB,every", [(600, 23), (600, 151), (150, 40)])
def test_short_lists_between_empty_key_blocks(nB, every):
    from paper_2609_06712_gb300 import rola as rl
    H, r = 40, 16
    cfg = configs.get("tiny", T=nB, Hh=8, Ww=8, H=H, keep=0.5 / nB, r=r)
    one = dict(cfg, H=1)
    N = cfg["N"]
    kept = np.zeros(nB, np.int32)
    for n, j in enumerate(range(7, nB - 4, every)):
        kept[j:j + 1 + n % 4] = j                        # kept by 1, 2, 3, 4, 1 ... query blocks
    g = torch.Generator().manual_seed(nB + every)
    x = [torch.randn((1, 1, N, 128), generator=g).mul(s).bfloat16() for s in (0.5, 0.5, 1.0, 1.0)]
    h = [t.float().numpy() for t in x]
    zero = np.zeros((1, r, 128), np.float32)             # no low-rank part
    want = O.backward(one, h[0], h[1], h[2], zero, zero, None, kept[None, None, :, None], h[3])

    # the log-sum-exp of every query over its block's keys, from the rotated rows in their storage type
    qr, kr = (torch.from_numpy(O.rope_full(one, a)).bfloat16().double().view(nB, 64, 128) for a in h[:2])
    lse = torch.logsumexp(qr @ kr[torch.from_numpy(kept).long()].transpose(1, 2) / np.sqrt(128.0), -1).float()

    heads = lambda t: t.cuda().expand(1, H, *t.shape[2:]).contiguous()  # noqa: E731
    q, k, v, dO = (heads(t) for t in x)
    lse = heads(lse.view(1, 1, N))
    kv = heads(torch.from_numpy(kept).view(1, 1, nB, 1))
    c = rl.make_config(cfg)
    assert rl.num_keep(c) == 1
    ws, bws = rl.workspace(c), rl.backward_workspace(c)
    o_s, dq, dk, dv = (torch.empty_like(q) for _ in range(4))
    rl.sparse_attn(c, q, k, v, kv, o_s, ws)
    P = torch.zeros((H, r, 128), dtype=torch.bfloat16, device="cuda")
    dP = [torch.empty((H, r, 128), device="cuda") for _ in range(2)]
    rl.backward(c, q, k, v, P, P, None, kv, o_s, lse, torch.zeros((1, H, r, 128), device="cuda"), dO, dq, dk, dv, *dP,
                None, bws)
    torch.cuda.synchronize()
    assert rl.get_device_status(ws) == rl.ROLA_OK and rl.get_device_status(bws) == rl.ROLA_OK
    lists = np.bincount(kept, minlength=nB).repeat(64)   # per key row: how many query blocks kept its block
    for name, t in (("dq", dq), ("dk", dk), ("dv", dv)):
        assert all(torch.equal(t[:, 0], t[:, i]) for i in range(1, H)), name
        got, ref = to_np(t[0, 0]), want[name][0, 0]
        if name == "dq":
            assert_close_grad(got, ref, True, name)
            continue
        assert (got[lists == 0] == 0).all(), name
        short = (lists > 0) & (lists <= 4)
        assert_close_grad(got[short], ref[short], True, f"{name}, short lists")
        assert_close_grad(got[lists > 4], ref[lists > 4], True, f"{name}, block 0")
