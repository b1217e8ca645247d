"""The block mask's selection kernel on rows that take each of its paths (the linear histogram, the radix
select, all scores equal) and at the edges of its row lengths, bit for bit against the oracle's fp32 decision."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2609_06712_gb300 import configs

pytestmark = pytest.mark.gpu


def values(kind, n, rng):
    """Per-block magnitudes: block i's tokens all hold values[i] in one coordinate, so score ij is a_i c_j const."""
    if kind == "normal":
        return rng.standard_normal(n)
    if kind == "ties":                       # four distinct scores a row: bins far over what is ranked directly
        return rng.integers(0, 4, n).astype(np.float64)
    if kind == "outlier":                    # one score a million times the others: nearly all in one bin
        return np.where(np.arange(n) == n // 3, 1e6, rng.standard_normal(n))
    if kind == "pairs":                      # every score twice: ties inside the bin that is ranked directly
        return np.repeat(rng.standard_normal(-(-n // 2)), 2)[:n]
    if kind == "infinite":                   # scores that overflow to +-inf
        return np.where(rng.random(n) < 0.2, 1e30, rng.standard_normal(n))
    return np.zeros(n)                       # all equal


@pytest.mark.parametrize("kind", ["normal", "ties", "outlier", "pairs", "infinite", "equal"])
@pytest.mark.parametrize("nB", [1, 31, 33, 512, 513, 1280, 1281])
def test_selection_paths(kind, nB):
    from paper_2609_06712_gb300 import rola as rl
    # one 8 x 8 plane of tokens a block, so every block sees the same row and column positions
    cfg = configs.get("tiny", T=nB, Hh=8, Ww=8, H=1, keep=0.1, r=16)
    rng = np.random.default_rng(nB)
    x = {}
    for name in ("q", "k"):
        t = np.zeros((1, 1, nB, 64, 128), np.float32)
        t[0, 0, :, :, 126] = values(kind, nB, rng)[:, None]      # the column axis's slowest pair
        x[name] = t.reshape(1, 1, nB * 64, 128)
    c = rl.make_config(cfg, rl.ROLA_FP32)
    kv = torch.empty((1, 1, nB, rl.num_keep(c)), dtype=torch.int32, device="cuda")
    rl.block_mask(c, *(torch.from_numpy(x[n]).cuda() for n in ("q", "k")), kv, rl.workspace(c))
    torch.cuda.synchronize()
    want, _ = O.block_mask_f32(cfg, x["q"], x["k"])
    assert (kv.cpu().numpy() == want).all()
