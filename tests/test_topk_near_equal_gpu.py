"""Block selection on rows whose scores agree to all but their last bits (a static scene, a constant frame): the
kept ids bit for bit against the oracle's fp32 decision, every row written."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_06712_gb300 import configs

pytestmark = pytest.mark.gpu


def select(cfg, dtype, q, k):
    """The kept ids of the kernels and of the oracle's fp32 decision."""
    from paper_2609_06712_gb300 import rola as rl
    q, k = (torch.from_numpy(x).to(dtype) for x in (q, k))
    c = rl.make_config(cfg, rl.ROLA_FP32 if dtype == torch.float32 else rl.ROLA_BF16)
    kv = torch.full((1, cfg["H"], rl.num_blocks(c), rl.num_keep(c)), -1, dtype=torch.int32, device="cuda")
    rl.block_mask(c, q.cuda(), k.cuda(), kv, rl.workspace(c))
    torch.cuda.synchronize()
    return kv.cpu().numpy(), O.block_mask_f32(cfg, q.float().numpy(), k.float().numpy())[0]


@pytest.mark.parametrize("ulps", [1, 3, 16, 60])
@pytest.mark.parametrize("base", [1.2200117, -0.9535515, 0.3333])
@pytest.mark.parametrize("nB,keep", [(39, 0.1), (64, 0.1), (64, 0.5), (128, 0.2), (512, 0.9), (1280, 0.95), (1281, 0.95)])
def test_scores_a_few_last_bits_apart(nB, keep, base, ulps):
    # one column: the column axis does not rotate, so the score of blocks i and j is a_i c_j / sqrt(d)
    cfg = configs.get("tiny", T=nB, Hh=64, Ww=1, H=2, keep=keep, r=16)
    rng = np.random.default_rng(1000 * nB + ulps)
    n_keep = O.num_keep(cfg)
    q = np.zeros((1, 2, nB, 64, 128), np.float32)
    k = np.zeros_like(q)
    q[..., 126] = 1.0
    for h in range(2):
        # head 0: fewer raised scores than are kept, so the lowest ones decide; head 1: raised ones decide
        raised = rng.permutation(nB)[:n_keep // 2 if h == 0 else min(nB - 1, n_keep + 3)]
        c = np.full(nB, np.float32(base)).view(np.int32)
        c[raised] += np.sign(base).astype(np.int32) * rng.integers(1, ulps + 1, len(raised)).astype(np.int32)
        if nB > 128:                      # the lowest scores: few enough to be ranked against each other
            c[rng.permutation(nB)[:100]] = np.float32(base).view(np.int32) - np.sign(base).astype(np.int32)
        k[0, h, :, :, 126] = c.view(np.float32)[:, None]
    got, want = select(cfg, torch.float32, q.reshape(1, 2, -1, 128), k.reshape(1, 2, -1, 128))
    assert (got == want).all()


@pytest.mark.parametrize("nB", [53, 78])
@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("factor", [0.99, 1.01])
def test_one_token_differs_in_bf16(nB, seed, factor):
    # one frame of one row, the default rotary split, constant tokens, one of them 1 % off in a coordinate
    cfg = configs.get("tiny", T=1, Hh=1, Ww=64 * nB, H=1, keep=0.1, r=16, rope_split=(44, 42, 42))
    rng = np.random.default_rng(seed)
    x = {}
    for name in ("q", "k"):
        x[name] = np.tile(rng.standard_normal(128).astype(np.float32), (1, 1, 64 * nB, 1))
        x[name][..., 86:] = 0.0           # nothing on the column axis: the frame's tokens rotate alike
    x["k"][0, 0, 64 * 7 + 5, 3] *= factor
    got, want = select(cfg, torch.bfloat16, x["q"], x["k"])
    assert (got == want).all()
