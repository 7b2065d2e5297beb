"""Paths that a call takes by the addresses of its tensors or by its size."""
import numpy as np
import pytest
import torch

import oracle
import paper_2505_00315_gb300 as mosa
from paper_2505_00315_gb300 import workloads as W
from _gpu import assert_close, run_layer, to_dev

pytestmark = pytest.mark.gpu

GRADS = ("dX", "dW_r", "dW_q", "dW_k", "dW_v", "dW_o")


def shifted(t):
    """A contiguous copy of t that starts one element past a 256-byte boundary."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    out = buf[1:].view(t.shape)
    out.copy_(t)
    assert out.is_contiguous() and out.data_ptr() % 16 != 0
    return out


# Every tensor of a layer at an address that is not 16-byte aligned, alone and all at once:
# the products and the router that cannot load it in 16-byte pieces run on the CUDA cores,
# beside others of the same call that can.
@pytest.mark.parametrize("cfg", [
    W.MosaConfig("f32", B=2, T=100, d=136, H=5, hp=32, k=40, dtype="f32", seed=101, rope=True),
    W.MosaConfig("bf16_hp128", B=2, T=100, d=72, H=3, hp=128, k=30, dtype="bf16", seed=102),
], ids=lambda c: c.name)
@pytest.mark.parametrize("which", ["X", "W_r", "W_q", "W_k", "W_v", "W_o", "dY", "Y", "dX", "dW_r",
                                   "dW_q", "dW_k", "dW_v", "dW_o", "all"])
def test_tensors_at_unaligned_addresses(cfg, which):
    x = W.make_inputs(cfg)
    names = {"X": "X", "W_r": "Wr", "W_q": "Wq", "W_k": "Wk", "W_v": "Wv", "W_o": "Wo", "dY": "dY"}
    t = {n: to_dev(x[s], cfg.dtype) for n, s in names.items()}
    out = {"Y": torch.empty(t["X"].shape, device="cuda")}
    grads = {"d" + n: torch.empty(t[n].shape, device="cuda") for n in names if n != "dY"}
    for group in (t, out, grads):
        for n in group:
            if which in (n, "all"):
                group[n] = shifted(group[n])
    w = [t[n] for n in ("X", "W_r", "W_q", "W_k", "W_v", "W_o")]
    Y, I, rs, _, ws = mosa.mosa_forward(*w, cfg.k, out=out, rope=cfg.rope)
    g = mosa.mosa_backward(*w, I, rs, t["dY"], ws, out=grads, rope=cfg.rope)
    assert mosa.mosa_check_status(mosa.make_shape(w[0], w[2], cfg.k), ws) == 0
    ow = [x[s] for s in ("Wr", "Wq", "Wk", "Wv", "Wo")]
    Yr, Ir, _, _ = oracle.forward(x["X"], *ow, k=cfg.k, rope=cfg.rope)
    np.testing.assert_array_equal(I.cpu().numpy(), Ir)
    assert_close("Y", Y.cpu().numpy(), Yr, cfg.dtype)
    ref = oracle.backward(x["X"], *ow, I=Ir, dY=x["dY"], rope=cfg.rope)
    for n in GRADS:
        assert_close(n, g[n].cpu().numpy(), ref["dX" if n == "dX" else n[:2] + n[3:]], cfg.dtype)


# CUDA-core attention in tiles of 64 rows on both sides (at least 152 of them), ragged
WIDE = [
    W.MosaConfig("f32_hp32", B=4, T=160, d=72, H=20, hp=32, k=77, dtype="f32", seed=103),
    W.MosaConfig("f32_hp64", B=4, T=160, d=80, H=16, hp=64, k=130, dtype="f32", seed=104),
    W.MosaConfig("bf16_hp16", B=4, T=150, d=96, H=24, hp=16, k=65, dtype="bf16", seed=105),
    W.MosaConfig("bf16_hp128", B=4, T=160, d=96, H=20, hp=128, k=100, dtype="bf16", seed=106),
]


@pytest.mark.parametrize("cfg", WIDE, ids=lambda c: c.name)
def test_attention_in_64_row_tiles_parity(cfg):
    x = W.make_inputs(cfg)
    w = [x[s] for s in ("Wr", "Wq", "Wk", "Wv", "Wo")]
    g = run_layer(cfg, x, backward=True)
    Yr, Ir, _, _ = oracle.forward(x["X"], *w, k=cfg.k)
    np.testing.assert_array_equal(g["I"], Ir)
    assert_close("Y", g["Y"], Yr, cfg.dtype)
    ref = oracle.backward(x["X"], *w, I=Ir, dY=x["dY"])
    for n in GRADS:
        assert_close(n, g[n], ref["dX" if n == "dX" else n[:2] + n[3:]], cfg.dtype)


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("cfg", WIDE, ids=lambda c: c.name)
def test_non_finite_token_stays_behind_the_mask(cfg, value):
    # a non-finite token changes no output of the tokens before it, and a non-finite dY row no
    # gradient of the tokens after it (token sets given, so that they do not depend on it)
    x = W.make_inputs(cfg)
    X, Wr, Wq, Wk, Wv, Wo, dY = (to_dev(x[n], cfg.dtype)
                                 for n in ("X", "Wr", "Wq", "Wk", "Wv", "Wo", "dY"))
    _, I, rs, _, _ = mosa.mosa_forward(X, Wr, Wq, Wk, Wv, Wo, cfg.k)
    at = cfg.T // 2

    def step(X, dY):
        Y, ws = mosa.mosa_forward_with_indices(X, Wq, Wk, Wv, Wo, I, rs)
        g = mosa.mosa_backward(X, Wr, Wq, Wk, Wv, Wo, I, rs, dY, ws)
        return Y.cpu().numpy(), g["dX"].cpu().numpy()

    Y, dX = step(X, dY)
    Xb, dYb = X.clone(), dY.clone()
    Xb[1, at, 3] = value
    dYb[1, at, 3] = value
    Yb, _ = step(Xb, dY)
    _, dXb = step(X, dYb)
    others = [0, 2, 3]
    tol = dict(rtol=1e-4, atol=1e-4)
    assert not np.isfinite(Yb[1, at:]).all() and not np.isfinite(dXb[1, :at + 1]).all()
    np.testing.assert_allclose(Yb[others], Y[others], **tol)
    np.testing.assert_allclose(Yb[1, :at], Y[1, :at], **tol)
    np.testing.assert_allclose(dXb[others], dX[others], **tol)
    np.testing.assert_allclose(dXb[1, at + 1:], dX[1, at + 1:], **tol)


# Router on CUDA cores: tiles of 16, 32 and 64 heads and more than one of them, ragged tokens,
# one chunk of d and several, X at an unaligned address.  A score is one multiply-add
# chain: at most d roundings of 2^-24 of the sum of |x w|, which sigmoid' = 1/4 at most scales,
# and the sigmoid's own few.
@pytest.mark.parametrize("dtype,hp", [("f32", 16), ("bf16", 128)])
@pytest.mark.parametrize("T,d,H", [(37, 8, 1), (100, 72, 16), (33, 264, 17), (257, 136, 33),
                                   (64, 520, 65), (95, 104, 130)])
@pytest.mark.parametrize("unaligned", [False, True])
def test_router_on_cuda_cores(T, d, H, dtype, hp, unaligned):
    cfg = W.MosaConfig("router", B=2, T=T, d=d, H=H, hp=hp, k=2, dtype=dtype, seed=107)
    x = W.make_inputs(cfg, plant=False)
    X, *w = (to_dev(x[n], dtype) for n in ("X", "Wr", "Wq", "Wk", "Wv", "Wo"))
    if unaligned:
        X = shifted(X)
    _, I, rs, rf, _ = mosa.mosa_forward(X, *w, cfg.k, want_r_full=True)
    ref = oracle.router(x["X"], x["Wr"])
    mag = np.einsum("btd,dh->bht", np.abs(x["X"]).astype(np.float64), np.abs(x["Wr"]).astype(np.float64))
    got = rf.cpu().numpy().astype(np.float64)
    assert (np.abs(got - ref) <= 2.0 ** -24 * (d * mag / 4 + 8)).all()
    order = np.argsort(-rf.cpu().numpy(), axis=2, kind="stable")[..., :cfg.k]
    np.testing.assert_array_equal(I.cpu().numpy(), np.sort(order, axis=2))
    np.testing.assert_array_equal(rs.cpu().numpy(), np.take_along_axis(rf.cpu().numpy(), np.sort(order, axis=2), axis=2))


# bf16 layers with heads of 64 move their tensors in 16-byte pieces only: such a tensor at another
# address is refused before anything is launched; W_r, dW_r and the scores may lie anywhere
@pytest.mark.parametrize("hybrid", [False, True])
@pytest.mark.parametrize("k", [32, 160])
def test_unaligned_tensors_of_tensor_core_layers_are_refused(k, hybrid):
    cfg = W.MosaConfig("refused", B=2, T=320, d=72, H=8, hp=64, k=k, dtype="bf16", seed=108)
    x = W.make_inputs(cfg)
    t = {n: to_dev(x[s], "bf16") for n, s in
         {"X": "X", "W_r": "Wr", "W_q": "Wq", "W_k": "Wk", "W_v": "Wv", "W_o": "Wo", "dY": "dY"}.items()}
    names = ["X", "W_r", "W_q", "W_k", "W_v", "W_o"]
    kw = {}
    if hybrid:
        for n, a in W.make_dense_weights(cfg, 2).items():
            t["D_" + n[1]] = to_dev(a, "bf16")
        names += ["D_q", "D_k", "D_v", "D_o"]
        kw = {"window": 160}
    forward = mosa.mosa_hybrid_forward if hybrid else mosa.mosa_forward
    backward = mosa.mosa_hybrid_backward if hybrid else mosa.mosa_backward

    def fresh():
        return ({"Y": torch.empty(t["X"].shape, device="cuda"),
                 "I": torch.empty((cfg.B, cfg.H, k), dtype=torch.int32, device="cuda"),
                 "r_sel": torch.empty((cfg.B, cfg.H, k), device="cuda")},
                {"d" + n: torch.empty(t[n].shape, device="cuda") for n in names})

    out, grads = fresh()
    got = forward(*(t[n] for n in names), k, out=out, **kw)
    ws, I, rs = got[-1], got[1], got[2]
    ref = {n: g.clone() for n, g in backward(*(t[n] for n in names), I, rs, t["dY"], ws, out=grads, **kw).items()}
    ref["Y"] = out["Y"].clone()
    torch.cuda.synchronize()

    anywhere = ("W_r", "dW_r", "I", "r_sel")
    for n in names + ["Y", "I", "r_sel"]:
        a, (o, _) = dict(t), fresh()
        group = o if n in o else a
        group[n] = shifted(group[n])
        before = mosa.mosa_kernel_launches()
        if n in anywhere:
            y = forward(*(a[m] for m in names), k, workspace=ws, out=o, **kw)[0]
            torch.testing.assert_close(y, ref["Y"], rtol=1e-4, atol=1e-4)
            continue
        with pytest.raises(RuntimeError, match="INVALID_ARG"):
            forward(*(a[m] for m in names), k, workspace=ws, out=o, **kw)
        assert mosa.mosa_kernel_launches() == before, n
    forward(*(t[n] for n in names), k, workspace=ws, out=out, **kw)
    for n in names + ["dY"] + ["d" + m for m in names]:
        if n == "W_r":
            continue
        a, (_, g) = dict(t), fresh()
        group = g if n in g else a
        group[n] = shifted(group[n])
        before = mosa.mosa_kernel_launches()
        if n in anywhere:
            got = backward(*(a[m] for m in names), I, rs, a["dY"], ws, out=g, **kw)
            torch.testing.assert_close(got[n], ref[n], rtol=1e-3, atol=1e-4)
            continue
        with pytest.raises(RuntimeError, match="INVALID_ARG"):
            backward(*(a[m] for m in names), I, rs, a["dY"], ws, out=g, **kw)
        assert mosa.mosa_kernel_launches() == before, n
    assert mosa.mosa_check_status(mosa.make_shape(t["X"], t["W_q"], k), ws) == 0
