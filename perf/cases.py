"""The calls this library is timed on: single MoSA layers through the binding,
from one short fp32 forward to the long bf16 training layers, hybrid layers
and TopK alone.

A case is a dict of plain values:
  op        "train"   forward + backward of one layer
            "infer"   forward only
            "topk"    TopK alone on given router scores
  dtype     storage, "bf16" or "f32"
  B, T, d   sequences, tokens per sequence, model width
  H, hp, k  MoSA heads, head size, tokens kept per head
  dense     dense (window 0) or local heads beside the MoSA heads (0: none)
  window    block length of the local heads
  first     every head keeps token 0 (Sec. 3.2)
  rope      rotary position encoding of Q and K (Sec. 2.2)

Inputs are the seeded Gaussian stand-ins of ``workloads.py`` (X ~ N(0,1),
weights ~ N(0,1/d), dY ~ N(0,1), a planted router margin so that the selected
set does not hang on the last bit of a score), drawn on the GPU.  Buffers
(workspace, outputs) are allocated once, as a training loop keeps them.
"""
import math

import torch

import paper_2505_00315_gb300 as mosa
from paper_2505_00315_gb300 import flops as F

MARGIN = 0.05   # raises the kept tokens' router logits, as workloads.PLANT_DELTA


def _case(name, op, dtype, B, T, d, H, hp, k, dense=0, window=0, first=False, rope=False):
    c = {"op": op, "dtype": dtype, "B": B, "T": T, "d": d, "H": H, "hp": hp, "k": k,
         "dense": dense, "window": window, "first": first, "rope": rope}
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest layer: one short fp32 sequence, forward only (a unit test, a
        # notebook, a small model's scoring call); launches and latency
        _case("f32_infer_B1_T256_H4_k64", "infer", "f32", 1, 256, 128, 4, 32, 64),
        # scoring one prompt of ragged length with a small language model's layer:
        # k from the adaptive rule max(T / 16, 2), first token kept, RoPE
        _case("infer_B1_T1531_H12_k95", "infer", "bf16", 1, 1531, 768, 12, 64, 95, 0, 0, True,
              True),
        # a training step of the paper's small models (T = 1024, d = 512, sparsity 8)
        _case("train_B8_T1024_d512_H16_k128", "train", "bf16", 8, 1024, 512, 16, 64, 128),
        # the IsoFLOP hybrid of Sec. 3.2: the same layer beside 4 dense heads, with
        # RoPE and the first token kept, as the paper trains it
        _case("train_hybrid_B8_T1024_H16_k128_dense4", "train", "bf16", 8, 1024, 512, 16, 64, 128,
              4, 0, True, True),
        # many small heads at high sparsity (16)
        _case("train_B16_T1024_H64_k64", "train", "bf16", 16, 1024, 1024, 64, 64, 64),
        # a long sequence at sparsity 32 (Sec. 3.4)
        _case("train_B2_T8192_H32_k256", "train", "bf16", 2, 8192, 1024, 32, 64, 256),
        # the long-sequence hybrid of Sec. 3.4: MoSA heads beside local heads of
        # 512 tokens, RoPE, at the paper's T = 2048
        _case("train_hybrid_B4_T2048_H60_k64_local4", "train", "bf16", 4, 2048, 1024, 60, 64, 64,
              4, 512, False, True),
        # both ends of the sparsity sweep at B4 T4096 d1024: few heads that keep
        # half of the tokens (the most work), and very many that keep 1/64
        _case("train_B4_T4096_H8_k2048", "train", "bf16", 4, 4096, 1024, 8, 64, 2048),
        _case("train_B4_T4096_H256_k64", "train", "bf16", 4, 4096, 1024, 256, 64, 64),
        # training in fp32 storage (a reference run, a small model) at ragged sizes
        _case("f32_train_B4_T1000_d768_H12_k125", "train", "f32", 4, 1000, 768, 12, 64, 125, 0, 0,
              False, True),
        # a model with heads of 128, the other common head size
        _case("train_hp128_B4_T1024_d1024_H16_k128", "train", "bf16", 4, 1024, 1024, 16, 128,
              128),
        # TopK alone (an external router), scores as they come, no margin
        _case("topk_64x8192_k256", "topk", "f32", 2, 8192, 8, 32, 64, 256),
    ]


def _flops(c):
    if c["op"] == "topk":
        return 0
    w = F.hybrid_work(c["B"], c["T"], c["d"], c["H"], c["hp"], c["k"], c["dense"], c["window"],
                      2 if c["dtype"] == "bf16" else 4)
    return w["forward_flops"] + (w["backward_flops"] if c["op"] == "train" else 0)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A call from the ranges the listed ones stand for, at any size in them."""
    kind = rng.choice(["train", "train", "train", "train", "hybrid", "infer", "f32", "f32_infer",
                       "heads", "topk"])
    # no drawn call costs more than the largest listed one of its storage and head size
    limit = {"f32": 7.5e9, "f32_infer": 7.5e9, "heads": 2.68e10}.get(kind, 1.63e11)
    while True:
        first, rope = rng.random() < 0.4, rng.random() < 0.5
        if kind == "topk":
            T = _log_int(rng, 64, 8192)
            rows = _log_int(rng, 1, 1024)
            k = max(1, min(T, int(T / math.exp(rng.uniform(0.1, math.log(128))))))
            if rows * T > (1 << 22):
                continue
            return _case(None, "topk", "f32", 1, T, 8, rows, 64, k)
        B = rng.randint(1, 16)
        T = _log_int(rng, 128, 8192)
        d = 8 * _log_int(rng, 16, 128)
        H = _log_int(rng, 2, min(256, d // 4))
        sparsity = math.exp(rng.uniform(math.log(2), math.log(64)))
        k = max(2, min(T, int(T / sparsity)))
        dense = window = 0
        hp = 64
        dtype = "bf16"
        op = "infer" if kind in ("infer", "f32_infer") else "train"
        if kind == "hybrid":
            T = 64 * max(2, T // 64)
            k = min(k, T)
            dense = rng.randint(1, 6)
            window = rng.choice([0] + [w for w in (64, 128, 256, 512) if T % w == 0])
        if kind in ("f32", "f32_infer"):
            dtype, hp = "f32", rng.choice([32, 64])
        if kind == "heads":
            hp = rng.choice([32, 128])
        c = _case(None, op, dtype, B, T, d, H, hp, k, dense, window, first, rope)
        if B * T <= 16384 and H * k <= 4 * T and B * H * T <= (1 << 22) and 1e6 < _flops(c) <= limit:
            return c


def _topk_indices(r, k, first):
    """[.., T] scores -> ascending indices of the k largest (ties: lower index)."""
    if first:
        r = r.clone()
        r[..., 0] = float("inf")
    order = torch.sort(r, dim=-1, descending=True, stable=True).indices
    return torch.sort(order[..., :k], dim=-1).values


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)

    if c["op"] == "topk":
        rows, T, k = c["B"] * c["H"], c["T"], c["k"]
        return {"case": c, "scores": torch.sigmoid(normal(rows, T)),
                "out": {"I": torch.empty((rows, k), dtype=torch.int32, device="cuda"),
                        "r_sel": torch.empty((rows, k), dtype=torch.float32, device="cuda")}}
    B, T, d, H, hp, k = (c[n] for n in ("B", "T", "d", "H", "hp", "k"))
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    s = 1.0 / math.sqrt(d)
    X = normal(B, T, d).to(dt)
    Wr = (normal(d, H) * s).to(dt)
    Wq, Wk, Wv = ((normal(H, d, hp) * s).to(dt) for _ in range(3))
    Wo = (normal(H, hp, d) * s).to(dt)
    dY = normal(B, T, d).to(dt)
    # the planted margin: X + G pinv(W_r), G = MARGIN on each head's k best tokens
    W64 = Wr.double()
    logits = (X.float() @ Wr.float()).transpose(1, 2)
    I = _topk_indices(logits, k, c["first"])
    raised = torch.zeros((B, H, T), dtype=torch.float64, device="cuda").scatter_(2, I, MARGIN)
    X = (X.double() + raised.transpose(1, 2) @ torch.linalg.solve(W64.T @ W64, W64.T)).to(dt)
    st = {"case": c, "X": X.contiguous(), "W": [Wr, Wq, Wk, Wv, Wo], "dY": dY, "D": []}
    if c["dense"]:
        n = c["dense"]
        st["D"] = [(normal(n, d, hp) * s).to(dt) for _ in range(3)] + [(normal(n, hp, d) * s).to(dt)]
        shape = mosa.make_hybrid_shape(X, Wq, k, n, c["window"], c["first"], c["rope"])
        st["ws"] = mosa.alloc_hybrid_workspace(shape, X.device)
    else:
        st["ws"] = mosa.alloc_workspace(mosa.make_shape(X, Wq, k, c["first"], c["rope"]), X.device)
    st["out"] = {"Y": torch.empty((B, T, d), dtype=torch.float32, device="cuda"),
                 "I": torch.empty((B, H, k), dtype=torch.int32, device="cuda"),
                 "r_sel": torch.empty((B, H, k), dtype=torch.float32, device="cuda")}
    if c["op"] == "train":
        names = ("dX", "dW_r", "dW_q", "dW_k", "dW_v", "dW_o", "dD_q", "dD_k", "dD_v", "dD_o")
        like = [X, Wr, Wq, Wk, Wv, Wo] + st["D"]
        st["grads"] = {n: torch.empty(t.shape, dtype=torch.float32, device="cuda")
                       for n, t in zip(names, like)}
    return st


def run(state):
    c = state["case"]
    if c["op"] == "topk":
        I, rs = mosa.mosa_topk(state["scores"], c["k"], out=state["out"])
        return {"I": I, "r_sel": rs}
    X, W, D, k = state["X"], state["W"], state["D"], c["k"]
    if D:
        Y, I, rs, ws = mosa.mosa_hybrid_forward(X, *W, *D, k, window=c["window"],
                                                workspace=state["ws"], out=state["out"],
                                                first_token=c["first"], rope=c["rope"])
    else:
        Y, I, rs, _, ws = mosa.mosa_forward(X, *W, k, workspace=state["ws"], out=state["out"],
                                            first_token=c["first"], rope=c["rope"])
    got = {"Y": Y, "I": I, "r_sel": rs}
    if c["op"] == "train":
        if D:
            got.update(mosa.mosa_hybrid_backward(X, *W, *D, I, rs, state["dY"], ws,
                                                 window=c["window"], out=state["grads"],
                                                 rope=c["rope"]))
        else:
            got.update(mosa.mosa_backward(X, *W, I, rs, state["dY"], ws, out=state["grads"],
                                          rope=c["rope"]))
    return got


def work(case):
    c = case
    B, T, d, H, hp, k, n = (c[x] for x in ("B", "T", "d", "H", "hp", "k", "dense"))
    if c["op"] == "topk":
        return {"bytes": B * H * (T + 2 * k) * 4, "flops": 0}
    e = 2 if c["dtype"] == "bf16" else 4
    weights = d * H + 4 * (H + n) * d * hp
    b = B * T * d * e + weights * e + B * T * d * 4 + 2 * B * H * k * 4   # in; Y, I, r_sel out
    if c["op"] == "train":
        b += B * T * d * e + B * T * d * 4 + weights * 4                   # dY in; gradients out
    return {"bytes": b, "flops": _flops(c)}


def _turn(x, pos):
    """RoPE on [.., tokens, h']: pairs (2p, 2p+1) of the first h'/2 dimensions."""
    half = x.shape[-1] // 2
    theta = 10000.0 ** (-torch.arange(0, half, 2, device=x.device, dtype=torch.float64) / half)
    ang = pos.double()[..., None] * theta
    cs, sn = torch.cos(ang), torch.sin(ang)
    a, b = x[..., 0:half:2], x[..., 1:half:2]
    turned = torch.stack((a * cs - b * sn, a * sn + b * cs), -1).flatten(-2)
    return torch.cat((turned, x[..., half:]), -1)


def exact(case, seed):
    """The layer in 64 bits with plain torch, one head at a time."""
    c, st = case, prepare(case, seed)
    if c["op"] == "topk":
        s = st["scores"].double()
        I = _topk_indices(s, c["k"], False)
        return {"I": I.int(), "r_sel": s.gather(1, I)}
    B, T, d, H, hp, k = (c[n] for n in ("B", "T", "d", "H", "hp", "k"))
    train = c["op"] == "train"
    X = st["X"].double()
    Wr, Wq, Wk, Wv, Wo = (w.double() for w in st["W"])
    D = [w.double() for w in st["D"]]
    dY = st["dY"].double()
    r = torch.sigmoid(X @ Wr).transpose(1, 2)                          # [B,H,T]
    I = _topk_indices(r, k, c["first"])
    Y = torch.zeros_like(X)
    got = {"Y": Y, "I": I.int(), "r_sel": r.gather(2, I)}
    if train:
        got["dX"] = torch.zeros_like(X)
        names = ["dW_r", "dW_q", "dW_k", "dW_v", "dW_o"] + ["dD_q", "dD_k", "dD_v", "dD_o"] * bool(D)
        for n, w in zip(names, [Wr, Wq, Wk, Wv, Wo] + D):
            got[n] = torch.zeros_like(w)

    def head(xs, dys, pos, wr, wq, wk, wv, wo):
        """One head on its tokens xs [n, tokens, d]: output and, in training, gradients."""
        leaves = [t.detach().requires_grad_(train) for t in (xs, wq, wk, wv, wo)]
        xs, wq, wk, wv, wo = leaves
        q, key, v = xs @ wq, xs @ wk, xs @ wv
        if c["rope"]:
            q, key = _turn(q, pos), _turn(key, pos)
        m = xs.shape[1]
        p = (q @ key.transpose(1, 2)) / math.sqrt(hp)
        p = p.masked_fill(torch.ones(m, m, device=p.device, dtype=torch.bool).triu(1), -math.inf)
        o = torch.softmax(p, -1) @ v
        if wr is not None:
            wr = wr.detach().requires_grad_(train)
            leaves.append(wr)
            o = o * torch.sigmoid(xs @ wr)[..., None]
        o = o @ wo
        g = torch.autograd.grad((o * dys).sum(), leaves) if train else None
        return o.detach(), g

    rows = torch.arange(B, device="cuda")[:, None]
    flat = lambda t: t.reshape(B * T, d)  # noqa: E731
    for h in range(H):
        idx = I[:, h]                                                  # [B,k]
        at = (rows * T + idx).reshape(-1)
        o, g = head(X[rows, idx], dY[rows, idx], idx, Wr[:, h], Wq[h], Wk[h], Wv[h], Wo[h])
        flat(Y).index_add_(0, at, o.reshape(-1, d))
        if train:
            flat(got["dX"]).index_add_(0, at, g[0].reshape(-1, d))
            for n, v in zip(("dW_q", "dW_k", "dW_v", "dW_o"), g[1:5]):
                got[n][h] = v
            got["dW_r"][:, h] = g[5]
    w = c["window"] or T
    for h in range(c["dense"]):
        blocks = lambda t: t.reshape(B * T // w, w, d)  # noqa: E731
        o, g = head(blocks(X), blocks(dY), torch.arange(w, device="cuda"), None,
                    *(m[h] for m in D))
        Y += o.reshape(B, T, d)
        if train:
            got["dX"] += g[0].reshape(B, T, d)
            for n, v in zip(("dD_q", "dD_k", "dD_v", "dD_o"), g[1:5]):
                got[n][h] = v
    return got
