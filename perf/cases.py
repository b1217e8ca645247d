"""Performance cases of the RoLA attention library: what its users run, and how long that takes is what counts.

A case is one call (or the few calls that belong together) of the public binding ``paper_2609_06712_gb300.rola`` on
layers shaped like the named configurations and the tests' layers.  ``kind`` says which entry point:

  forward   RoLAAttention (rola_forward): the hybrid attention module at inference; the default 64-token query blocks,
            128-token query chunks (qblock=128) or 4x4x4 cube blocks (geometry="cube")
  block     attention_block: token gate, module and output projection in one call
  train     RoLAFunction forward and backward: one step of the single-stage fine-tune
  mask      block_mask alone: a caller that keeps its own sparse engine
  lowrank   lowrank_summary then lowrank_apply: the global branch beside a caller's own sparse output

``exact`` evaluates the paper's formulas in plain torch in 64 bits.  The block mask is by definition an fp32 decision
with every rounding fixed (see include/rola.h, rola_block_mask), so ``exact`` takes that one decision in fp32 too.
"""
import math

import torch
from torch.utils.checkpoint import checkpoint

D_H, BLOCK, THETA, SPLIT = 128, 64, 10000.0, (44, 42, 42)
EPS = 1e-6
GATE_BIAS = -1.946

_DEFAULTS = dict(kind="forward", B=1, H=12, T=21, Hh=30, Ww=52, keep=0.1, r=32, qblock=64, geometry="flat",
                 act="silu", dtype="bf16", dist="normal", gate=True, d_model=0)


def _case(name, **kw):
    c = dict(_DEFAULTS, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest layer (1024 tokens, 2 heads, 16 key blocks): every kernel is a few microseconds, launches count
        _case("tiny_forward", H=2, T=4, Hh=16, Ww=16, keep=0.125, r=16, gate=False),
        # a short ragged clip in training, batch 2 (1170 tokens: the last block holds 18)
        _case("clip_train", kind="train", B=2, H=12, T=5, Hh=13, Ww=18, keep=0.3, r=24),
        # the fp32 validation mode: what a user checks a port of the layer against
        _case("fp32_forward", H=4, T=6, Hh=15, Ww=26, keep=0.2, r=32, dtype="fp32"),
        # Wan2.1-1.3B layer at 480p, inference
        _case("wan13b_480p_forward", dist="rmsnorm", gate=False),
        # Wan2.1-1.3B layer at 480p, one fine-tuning step
        _case("wan13b_480p_train", kind="train", dist="rmsnorm"),
        # Wan2.1-14B at 480p: the attention block after the QKV projection (gate, module, output projection)
        _case("wan14b_480p_block", kind="block", H=40, d_model=5120, dist="rmsnorm_gain"),
        # Wan2.1-14B at 480p with cube blocks (grid edges give ragged cubes)
        _case("wan14b_480p_cube", H=40, geometry="cube", dist="rmsnorm_gain", gate=False),
        # the headline: Wan2.1-14B layer at 720p, inference
        _case("wan14b_720p_forward", H=40, Hh=45, Ww=80),
        # the same layer with the mask chosen per 128-token query chunk
        _case("wan14b_720p_q128", H=40, Hh=45, Ww=80, qblock=128),
        # the largest: one fine-tuning step of the 14B layer at 720p
        _case("wan14b_720p_train", kind="train", H=40, Hh=45, Ww=80),
        # the block mask alone at 720p
        _case("wan14b_720p_mask", kind="mask", H=40, Hh=45, Ww=80, gate=False),
        # the low-rank branch alone at 720p, a rank of the upper half of the sweep
        _case("wan14b_720p_lowrank_r64", kind="lowrank", H=40, Hh=45, Ww=80, r=64),
    ]


def draw(rng):
    """One more layer: a latent grid of 300 to 75600 tokens, 1 to 40 heads, ranks 8 to 128, 80 to 95 % sparsity."""
    kind = rng.choice(["forward", "forward", "forward", "block", "train", "train", "mask", "lowrank"])
    dtype = "fp32" if kind == "forward" and rng.random() < 0.15 else "bf16"
    most = 6000 if dtype == "fp32" else 75600
    while True:
        n = math.exp(rng.uniform(math.log(300), math.log(most)))
        T = max(1, min(41, round(math.exp(rng.uniform(0.0, math.log(41))))))
        plane = n / T
        Hh = max(2, round(math.sqrt(plane * rng.uniform(0.4, 1.0))))
        Ww = max(2, round(plane / Hh))
        if 300 <= T * Hh * Ww <= most:
            break
    c = _case(None, kind=kind, dtype=dtype, T=T, Hh=Hh, Ww=Ww)
    c["B"] = rng.choice([1, 1, 1, 2])
    c["H"] = round(math.exp(rng.uniform(0.0, math.log((8 if dtype == "fp32" else 40) / c["B"]))))
    c["keep"] = rng.choice([0.05, 0.1, 0.1, 0.2])
    c["r"] = rng.choice([8, 16, 16, 32, 32, 32, 48, 64, 64, 128])
    c["act"] = rng.choice(["silu"] * 7 + ["identity", "tanh", "relu", "gelu"])
    c["dist"] = rng.choice(["normal", "normal", "rmsnorm", "rmsnorm_gain"])
    c["gate"] = rng.random() < 0.6
    if kind in ("forward", "train", "mask") and rng.random() < 0.25:
        c["geometry"] = "cube"
    elif kind in ("forward", "block", "mask") and rng.random() < 0.3:
        c["qblock"] = 128
    if kind == "block":
        c["d_model"] = 64 * rng.randint(1, 2 * c["H"])
    largest = _flops(listed()[9])
    while _flops(c) > largest:
        c["keep"] /= 2
    return c


# ------------------------------------------------------------------ sizes and work

def _tokens(c):
    return c["T"] * c["Hh"] * c["Ww"]


def _blocks(c):
    """(key blocks, query blocks, kept key blocks of a query block)"""
    if c["geometry"] == "cube":
        nk = nq = -(-c["T"] // 4) * -(-c["Hh"] // 4) * -(-c["Ww"] // 4)
    else:
        nk, nq = -(-_tokens(c) // BLOCK), -(-_tokens(c) // c["qblock"])
    keep = float(torch.tensor(c["keep"], dtype=torch.float32))
    return nk, nq, min(nk, max(1, int(math.floor(keep * nk + 0.5))))


def _parts(c):
    """Operations of the sparse branch, the low-rank branch, the block scores and the projections (forward)."""
    n, bh = _tokens(c), c["B"] * c["H"]
    nk, nq, kept = _blocks(c)
    sparse = 4.0 * D_H * bh * n * (kept * n / nk)
    lowrank = 8.0 * bh * n * D_H * c["r"]
    scores = 2.0 * D_H * bh * nq * nk
    proj = c["d_model"] * c["B"] * n * (2.0 * D_H * c["H"] + 2.0)
    return sparse, lowrank, scores, proj


def _flops(c):
    sparse, lowrank, scores, proj = _parts(c)
    return {"forward": sparse + lowrank + scores, "block": sparse + lowrank + scores + proj,
            "train": 3.5 * sparse + 3.75 * lowrank + scores, "mask": scores, "lowrank": lowrank}[c["kind"]]


def work(case):
    c = case
    n, bh, e = _tokens(c), c["B"] * c["H"], 4 if c["dtype"] == "fp32" else 2
    rows, P = e * bh * n * D_H, 2 * e * c["H"] * c["r"] * D_H
    _, nq, kept = _blocks(c)
    mask, gate = 4 * bh * nq * kept, 4 * c["B"] * n if c["gate"] else 0
    if c["kind"] == "forward":
        b = 4 * rows + P + mask + gate
    elif c["kind"] == "block":
        b = 4 * rows + P + mask + 4 * c["B"] * n + 2 * e * c["B"] * n * c["d_model"] + e * c["d_model"] * D_H * c["H"]
    elif c["kind"] == "train":
        b = 8 * rows + 2 * P + 2 * gate
    elif c["kind"] == "mask":
        b = 2 * rows + mask
    else:
        b = 5 * rows + P + gate + 4 * bh * c["r"] * D_H
    return {"bytes": float(b), "flops": _flops(c)}


# ------------------------------------------------------------------ inputs

def _inputs(c, seed):
    """Layer activations as the backbone hands them over: q, k normalised as the model does, a token gate around 1/8."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    f32 = dict(dtype=torch.float32, device="cuda", generator=g)
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    shape = (c["B"], c["H"], _tokens(c), D_H)
    x = {}
    for name in ("q", "k", "v"):
        t = torch.randn(shape, **f32)
        if name != "v" and c["dist"] != "normal":
            t = t * torch.rsqrt(t.square().mean(-1, keepdim=True))
            if c["dist"] == "rmsnorm_gain":
                t = t * (0.5 + torch.rand((c["H"], 1, D_H), **f32))
        x[name] = t.to(dt)
    for name in ("P_q", "P_k"):
        x[name] = (torch.randn((c["H"], c["r"], D_H), **f32) / math.sqrt(D_H)).to(dt)
    x["gate"] = torch.sigmoid(GATE_BIAS + 0.5 * torch.randn(shape[0:1] + shape[2:3], **f32)) if c["gate"] else None
    if c["kind"] == "train":
        x["dO"] = torch.randn(shape, **f32).to(dt)
    if c["kind"] == "lowrank":
        x["o_s"] = (0.3 * torch.randn(shape, **f32)).to(dt)   # the spread of a softmax average over a few dozen values
    if c["kind"] == "block":
        dm = c["d_model"]
        x["X"] = torch.randn((c["B"], _tokens(c), dm), **f32).to(dt)
        x["w_g"] = (torch.randn((dm,), **f32) / math.sqrt(dm)).to(dt)
        x["W_o"] = (torch.randn((dm, c["H"] * D_H), **f32) / math.sqrt(c["H"] * D_H)).to(dt)
        x["b_o"] = 0.1 * torch.randn((dm,), **f32)
    return x


def prepare(case, seed):
    from paper_2609_06712_gb300 import rola
    c = case
    x = _inputs(c, seed)
    layer = dict(B=c["B"], H=c["H"], N=_tokens(c), T=c["T"], Hh=c["Hh"], Ww=c["Ww"], keep=c["keep"], r=c["r"],
                 lowrank_act=c["act"], block_geometry=c["geometry"], qblock=c["qblock"], gate_bias=GATE_BIAS)
    dtype = rola.ROLA_FP32 if c["dtype"] == "fp32" else rola.ROLA_BF16
    st = {"c": c, "x": x, "rola": rola}
    empty = lambda *s, dt=torch.float32: torch.empty(s, dtype=dt, device="cuda")  # noqa: E731
    nk, nq, kept = _blocks(c)
    if c["kind"] == "forward":
        st["attn"] = rola.RoLAAttention(layer, dtype)
        # the mask has a row per query block (128-token chunks: half as many as the handle's default buffer)
        st["kv_idx"] = empty(c["B"], c["H"], nq, kept, dt=torch.int32)
        return st
    st["cfg"] = rola.make_config(layer, dtype)
    if c["kind"] == "train":
        for name in ("q", "k", "v", "P_q", "P_k") + (("gate",) if c["gate"] else ()):
            x[name].requires_grad_()
        return st
    st["ws"] = rola.workspace(st["cfg"])
    if c["kind"] in ("block", "mask"):
        st["kv_idx"] = empty(c["B"], c["H"], nq, kept, dt=torch.int32)
    if c["kind"] == "block":
        st["gate"] = empty(c["B"], _tokens(c))
        st["o"] = torch.empty_like(x["q"])
        st["Y"] = torch.empty_like(x["X"])
    if c["kind"] == "lowrank":
        st["C"] = empty(c["B"], c["H"], c["r"], D_H)
        st["o"] = torch.empty_like(x["q"])
    return st


def run(state):
    c, x, rola = state["c"], state["x"], state["rola"]
    if c["kind"] == "forward":
        o, kv = state["attn"](x["q"], x["k"], x["v"], x["P_q"], x["P_k"], x["gate"], kv_idx=state["kv_idx"])
        return {"o": o, "kv_idx": kv}
    cfg = state["cfg"]
    if c["kind"] == "train":
        o = rola.RoLAFunction.apply(cfg, x["q"], x["k"], x["v"], x["P_q"], x["P_k"], x["gate"])
        names = ["q", "k", "v", "P_q", "P_k"] + (["gate"] if c["gate"] else [])
        grads = torch.autograd.grad(o, [x[n] for n in names], x["dO"])
        return {"o": o, **{"d" + n: g for n, g in zip(names, grads)}}
    ws = state["ws"]
    if c["kind"] == "block":
        rola.attention_block(cfg, x["X"], x["w_g"], GATE_BIAS, x["q"], x["k"], x["v"], x["P_q"], x["P_k"], x["W_o"],
                             x["b_o"], state["gate"], state["o"], state["Y"], state["kv_idx"], ws)
        return {"gate": state["gate"], "o": state["o"], "Y": state["Y"], "kv_idx": state["kv_idx"]}
    if c["kind"] == "mask":
        rola.block_mask(cfg, x["q"], x["k"], state["kv_idx"], ws)
        return {"kv_idx": state["kv_idx"]}
    rola.lowrank_summary(cfg, x["k"], x["v"], x["P_k"], state["C"], None, ws)
    rola.lowrank_apply(cfg, x["q"], x["P_q"], state["C"], x["gate"], x["o_s"], state["o"], ws)
    return {"C": state["C"], "o": state["o"]}


# ------------------------------------------------------------------ the same in 64 bits

def _cos_sin(c):
    """cos and sin of every (token, pair)'s rotation angle: 22 / 21 / 21 pairs on t / row / column, theta^(-2i/d_axis)."""
    T, Hh, Ww = c["T"], c["Hh"], c["Ww"]
    n = torch.arange(_tokens(c), device="cuda")
    pos = (n // (Hh * Ww), n // Ww % Hh, n % Ww)
    ang = []
    for p, d in zip(pos, SPLIT):
        i = torch.arange(d // 2, device="cuda", dtype=torch.float64)
        ang.append(p.double()[:, None] * torch.pow(torch.tensor(THETA, dtype=torch.float64, device="cuda"), -2.0 * i / d))
    ang = torch.cat(ang, 1)
    return ang.cos(), ang.sin()


def _rotate(x, cs):
    """(x0, x1) -> (x0 cos - x1 sin, x0 sin + x1 cos) on the adjacent pairs of the last axis."""
    c, s = cs
    a, b = x[..., 0::2], x[..., 1::2]
    m = a.shape[-1]
    return torch.stack((a * c[:, :m] - b * s[:, :m], a * s[:, :m] + b * c[:, :m]), -1).flatten(-2)


def _members(c, size):
    """Token of every slot of every block [blocks, size]; _tokens(c) where the slot is empty."""
    n = _tokens(c)
    if c["geometry"] != "cube":
        m = torch.arange(-(-n // size) * size, device="cuda").view(-1, size)
        return torch.where(m < n, m, n)
    T, Hh, Ww = c["T"], c["Hh"], c["Ww"]
    i = torch.arange(64, device="cuda")
    grids = torch.meshgrid(*(torch.arange(-(-a // 4), device="cuda") * 4 for a in (T, Hh, Ww)), indexing="ij")
    t, x, y = (g.reshape(-1, 1) + o for g, o in zip(grids, (i // 16, i // 4 % 4, i % 4)))
    return torch.where((t < T) & (x < Hh) & (y < Ww), (t * Hh + x) * Ww + y, n)


def _means32(x, cs32, members):
    """fp32 block means of one head's rotated rows, each rounding as the mask's definition has it."""
    c, s = cs32
    a, b = x[:, 0::2], x[:, 1::2]
    fma = lambda u, w, add: (u.double() * w.double() + add.double()).float()  # noqa: E731
    y = torch.stack((fma(a, c, -(b * s)), fma(a, s, b * c)), -1).flatten(-2)
    y = torch.cat((y, y.new_zeros(1, D_H)))[members]
    while y.shape[1] > 1:
        y = y[:, 0::2] + y[:, 1::2]
    return y[:, 0] / (members < x.shape[0]).sum(1, keepdim=True).float()


def _mask(c, q, k, cs, kept):
    """[kept ids of every query block] of one head, as the fp32 decision that defines it."""
    cs32 = (cs[0].float(), cs[1].float())
    qm = _means32(q.float(), cs32, _members(c, c["qblock"] if c["geometry"] == "flat" else BLOCK)).double()
    km = _means32(k.float(), cs32, _members(c, BLOCK)).double()
    acc = torch.zeros(qm.shape[0], km.shape[0], dtype=torch.float32, device="cuda")
    for d in range(D_H):
        acc = torch.addcmul(acc.double(), qm[:, d, None], km[None, :, d]).float()
    scores = acc * torch.tensor(1.0 / math.sqrt(D_H), dtype=torch.float32, device="cuda")
    return torch.sort(scores, dim=1, descending=True, stable=True)[1][:, :kept].sort(1)[0]


def _feature(x, P, cs, act):
    u = x @ P.T
    f = {"silu": torch.nn.functional.silu, "identity": lambda t: t, "tanh": torch.tanh, "relu": torch.relu,
         "gelu": torch.nn.functional.gelu}[act]
    return _rotate(f(u), cs)


def _sparse(c, qr, kr, v, kv, rows_at_once):
    """Softmax attention of one head over the kept key blocks."""
    n = qr.shape[0]
    km, qm = _members(c, BLOCK), _members(c, c["qblock"] if c["geometry"] == "flat" else BLOCK)
    pad = lambda t: torch.cat((t, t.new_zeros(1, D_H)))  # noqa: E731
    qp, kp, vp = pad(qr), pad(kr), pad(v)

    def some(qp, kp, vp, i):
        keys = km[kv[i:i + rows_at_once]].flatten(1)
        s = qp[qm[i:i + rows_at_once]] @ kp[keys].transpose(1, 2) / math.sqrt(D_H)
        s = s.masked_fill((keys == n)[:, None, :], -math.inf)
        return torch.softmax(s, -1) @ vp[keys]

    outs = [checkpoint(some, qp, kp, vp, i, use_reentrant=False) if qr.requires_grad else some(qp, kp, vp, i)
            for i in range(0, qm.shape[0], rows_at_once)]
    return torch.zeros(n + 1, D_H, dtype=torch.float64, device="cuda").index_copy(0, qm.flatten(), torch.cat(outs).flatten(0, 1))[:n]


def _fuse(o_s, y, gate):
    o_lr = y / torch.sqrt(y.square().mean(-1, keepdim=True) + EPS)
    r = torch.sqrt(o_s.square().mean(-1, keepdim=True) + EPS)
    return (o_s / r + gate[:, None] * o_lr) * r


def exact(case, seed):
    c = case
    kind, n = c["kind"], _tokens(c)
    # 64-bit products run at about one TFLOP/s here
    if kind in ("forward", "block", "train") and (_flops(c) > 6e12 or (kind == "train" and _parts(c)[0] > 1.2e12)):
        return None
    x = _inputs(c, seed)
    cs = _cos_sin(c)
    nk, nq, kept = _blocks(c)
    q, k, P_q, P_k, gate = (x[m] for m in ("q", "k", "P_q", "P_k", "gate"))
    B, H = c["B"], c["H"]
    heads = [(b, h) for b in range(B) for h in range(H)]
    if kind == "mask":
        return {"kv_idx": torch.stack([_mask(c, q[b, h], k[b, h], cs, kept) for b, h in heads]).view(B, H, nq, kept)}
    v = x["v"]
    res = {}
    if kind == "block":
        gate = torch.sigmoid(x["X"].double() @ x["w_g"].double() + GATE_BIAS)
        res["gate"] = gate
    if gate is None:
        gate = torch.full((B, n), 1.0 / (1.0 + math.exp(-GATE_BIAS)), dtype=torch.float64, device="cuda")
    train = kind == "train"
    leaf = lambda t: t.double().detach().requires_grad_(train)  # noqa: E731
    o = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    kvs, Cs = [], []
    grads = {m: torch.zeros(t.shape, dtype=torch.float64, device="cuda")
             for m, t in (("q", q), ("k", k), ("v", v), ("P_q", P_q), ("P_k", P_k), ("gate", gate))} if train else {}
    at_once = max(1, int(2e9 // (kept * BLOCK * (D_H + c["qblock"]) * 16)))
    for b, h in heads:
        leaves = dict(q=leaf(q[b, h]), k=leaf(k[b, h]), v=leaf(v[b, h]), P_q=leaf(P_q[h]), P_k=leaf(P_k[h]), gate=leaf(gate[b]))
        if kind == "lowrank":
            o_s = x["o_s"][b, h].double()
        else:
            kvs.append(_mask(c, q[b, h], k[b, h], cs, kept))
            o_s = _sparse(c, _rotate(leaves["q"], cs), _rotate(leaves["k"], cs), leaves["v"], kvs[-1], at_once)
        C = _feature(leaves["k"], leaves["P_k"], cs, c["act"]).T @ leaves["v"]
        out = _fuse(o_s, _feature(leaves["q"], leaves["P_q"], cs, c["act"]) @ C, leaves["gate"])
        o[b, h] = out.detach()
        Cs.append(C.detach())
        if train:
            for (m, _), g in zip(leaves.items(), torch.autograd.grad(out, list(leaves.values()), x["dO"][b, h].double())):
                at = {"P_q": h, "P_k": h, "gate": b}.get(m, (b, h))
                grads[m][at] += g
    if kind == "lowrank":
        return {"C": torch.stack(Cs).view(B, H, c["r"], D_H), "o": o}
    res["o"] = o
    if train:
        if not c["gate"]:
            grads.pop("gate")
        return {**res, **{"d" + m: g for m, g in grads.items()}}
    res["kv_idx"] = torch.stack(kvs).view(B, H, nq, kept).to(torch.int32)
    if kind == "block":
        res["Y"] = o.transpose(1, 2).reshape(B, n, H * D_H) @ x["W_o"].double().T + x["b_o"].double()
    return res
