"""The readout's SiLU where its denominator 1 + e^-u lies past 2^126: the features are tiny but not zero, and bf16
has the exponents for them, so against a large C they still give the whole low-rank output."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_06712_gb300 import configs
from parity_util import assert_close, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rope", [0, 2])
@pytest.mark.parametrize("r", [16, 40, 128])
def test_features_of_a_large_denominator(r, rope):
    from paper_2609_06712_gb300 import rola as rl
    cfg = configs.get("tiny", T=2, Hh=5, Ww=9, H=2, r=r, lowrank_rope=rope, gate_bias=1.0)
    N = cfg["N"]
    g = torch.Generator().manual_seed(r)
    q = torch.zeros((1, 2, N, 128)).bfloat16()
    q[..., 5] = 1.0
    P = torch.zeros((2, r, 128)).bfloat16()
    P[..., 5] = -88.0                                   # u = -88: 1 + e^88 = 1.65e38, silu(u) = -5.3e-37
    C = 1e36 * torch.randn((1, 2, r, 128), generator=g).bfloat16().float()
    o_s = torch.randn((1, 2, N, 128), generator=g).bfloat16()
    c = rl.make_config(cfg)
    o = torch.empty_like(o_s, device="cuda")
    ws = rl.workspace(c)
    rl.lowrank_apply(c, q.cuda(), P.cuda(), C.cuda(), None, o_s.cuda(), o, ws)
    torch.cuda.synchronize()
    assert rl.get_device_status(ws) == rl.ROLA_OK
    want = O.lowrank_apply(cfg, q.float().numpy(), P.float().numpy(), C.numpy(), None, o_s.float().numpy(), rope_mode=rope)
    want = want[0] if isinstance(want, tuple) else want
    assert np.abs(want - o_s.float().numpy()).max() > 0.5      # the low-rank part is there
    assert_close(to_np(o), want, True, f"o[r={r}, rope={rope}]")
