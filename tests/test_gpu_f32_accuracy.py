"""fp32 layers against 64-bit values: the products on the tensor cores (through bf16 planes) are
no further from them than fp32 multiply-add chains, the same layer on the CUDA cores."""
import numpy as np
import pytest
import torch

import oracle
import paper_2505_00315_gb300 as mosa
from paper_2505_00315_gb300 import workloads as W
from _gpu import assert_close, run_layer, to_dev
from _util import rel_l2

pytestmark = pytest.mark.gpu

OPERANDS = ("X", "Wq", "Wk", "Wv", "Wo", "dY")


def shaped(kind, v):
    """Gaussian values, or ones with other low 16 significand bits: those for which what a cut into
    three 8-bit parts leaves out is largest, and of one sign, if it truncates (all ones, below
    any top bits or below zeros) or if it rounds (0x7FBF)."""
    u = v.view(np.uint32)
    low = {"gauss": None, "ones": 0xFFFF, "ones_only": 0xFFFF, "halves": 0x7FBF}[kind]
    if low is not None:
        u = (u & np.uint32(0xFF800000 if kind == "ones_only" else 0xFFFF0000)) | np.uint32(low)
    return u.view(np.float32)


# The rounding of the two paths is of the same size and independent, and a norm
# over at least 3 x 64 x 32 results varies by about 1%, so 1.25 times the chains' error (and
# 1e-8 for what both have in common, the stored results' own rounding) holds for products that
# lose nothing but rounding; parts cut by truncation are at 1.5 to 4 times it.
@pytest.mark.parametrize("kind", ["gauss", "ones", "ones_only", "halves"])
@pytest.mark.parametrize("cfg", [
    W.MosaConfig("f32_d128", B=2, T=96, d=128, H=3, hp=32, k=48, dtype="f32", seed=81),
    W.MosaConfig("f32_d520", B=3, T=200, d=520, H=4, hp=64, k=90, dtype="f32", seed=82),
    W.MosaConfig("f32_hp128", B=2, T=150, d=264, H=3, hp=128, k=66, dtype="f32", seed=83),
], ids=lambda c: c.name)
def test_f32_layer_as_close_to_64_bits_as_multiply_add_chains(cfg, kind, monkeypatch):
    x = W.make_inputs(cfg)
    for n in OPERANDS:
        x[n] = shaped(kind, x[n])
    planes = run_layer(cfg, x, backward=True)
    monkeypatch.setenv("MOSA_FORCE_SIMT", "1")
    chains = run_layer(cfg, x, backward=True)
    np.testing.assert_array_equal(planes["I"], chains["I"])
    I = planes["I"]
    w = (x["Wr"], x["Wq"], x["Wk"], x["Wv"], x["Wo"])
    ref = {"Y": oracle.forward_indices(x["X"], *w, I=I)}
    for n, g in oracle.backward(x["X"], *w, I=I, dY=x["dY"]).items():
        ref["dX" if n == "dX" else n[:2] + "_" + n[2:].lower()] = g
    errors = {n: (rel_l2(planes[n], r), rel_l2(chains[n], r)) for n, r in ref.items()}
    print(cfg.name, kind, {n: f"{p:.2e}/{c:.2e}" for n, (p, c) in errors.items()})
    for n, (p, c) in errors.items():
        assert p <= 1.25 * c + 1e-8, f"{n}: {p:.3e} against {c:.3e} of the multiply-add chains"


# Infinities beside weights so large that the parts' products pass the fp32 range with both
# signs, and finite products that do: infinite (of the same sign) or NaN where multiply-adds
# are.  (Not compared: dX, dW_q and dW_k, which take up dP - D; between values of this size
# its last bits decide which results overflow, and chains on inputs one bit away differ too.)
@pytest.mark.parametrize("cfg", [
    W.MosaConfig("overflow_d72", B=2, T=120, d=72, H=3, hp=32, k=40, dtype="f32", seed=84),
    W.MosaConfig("overflow_d200", B=4, T=300, d=200, H=2, hp=64, k=70, dtype="f32", seed=85),
], ids=lambda c: c.name)
def test_overflow_of_f32_products_as_with_multiply_adds(cfg, monkeypatch):
    rng = np.random.default_rng(cfg.seed)
    x = W.make_inputs(cfg)
    x["X"][0, 7, 3] = np.inf
    x["X"][1, 9, 5] = -np.inf
    x["X"][0, 31, 8] = 3e25
    x["X"][1, 33, 9] = -2e25
    x["Wv"][1, 3, ::3] *= 1e8
    x["Wq"][0, 5] *= 1e9
    x["Wv"][2 % cfg.H, 8] *= 1e20
    x["Wo"][0, 4] *= 1e30
    x["dY"][1, 20:60, ::7] *= 1e12 * rng.random((40, len(range(0, cfg.d, 7))), dtype=np.float32)
    x["dY"][0, 11, 6] = np.inf
    a = run_layer(cfg, x, backward=True)
    monkeypatch.setenv("MOSA_FORCE_SIMT", "1")
    b = run_layer(cfg, x, backward=True)
    np.testing.assert_array_equal(a["I"], b["I"])
    for n in ("Y", "dW_v", "dW_o", "dW_r"):
        fin = np.isfinite(b[n])
        np.testing.assert_array_equal(np.isfinite(a[n]), fin, err_msg=n)
        np.testing.assert_array_equal(a[n][~fin], b[n][~fin], err_msg=n)   # NaN equal to NaN


def test_one_nan_does_not_slow_an_f32_layer():
    # a diverged step takes about as long as any other: its NaNs are final
    cfg = W.MosaConfig("nan_time", B=4, T=2048, d=768, H=12, hp=64, k=512, dtype="f32", seed=86)
    g = torch.Generator(device="cuda").manual_seed(cfg.seed)
    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda") / cfg.d ** 0.5
    X, dY = (normal(cfg.B, cfg.T, cfg.d) for _ in range(2))
    Wr = normal(cfg.d, cfg.H)
    Wq, Wk, Wv = (normal(cfg.H, cfg.d, cfg.hp) for _ in range(3))
    Wo = normal(cfg.H, cfg.hp, cfg.d)

    def step_us():
        shape = mosa.make_shape(X, Wq, cfg.k)
        ws = mosa.alloc_workspace(shape)
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            Y, I, rs, _, _ = mosa.mosa_forward(X, Wr, Wq, Wk, Wv, Wo, cfg.k, workspace=ws, out=out)
            out.update(Y=Y, I=I, r_sel=rs)
            got = mosa.mosa_backward(X, Wr, Wq, Wk, Wv, Wo, I, rs, dY, ws, out=grads)
            grads.update(got)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 1e3)
        assert mosa.mosa_check_status(shape, ws) == 0
        return sorted(times)[1], got

    out, grads = {}, {}
    plain, _ = step_us()
    X[1, cfg.T - 1, 5] = float("nan")   # kept by every head: a NaN score ranks first
    nan, got = step_us()
    print(f"step {plain:.0f} us, with NaNs {nan:.0f} us")
    assert all(torch.isnan(got[n]).any() for n in ("dX", "dW_q", "dW_o"))
    # (not once: the CUDA-core attention has a slower branch for tiles with non-finite values)
    assert nan < 2.0 * plain, (nan, plain)


def test_weight_gradients_do_not_hang_on_the_workspace_contents():
    # bf16 with heads of 128: dlogit's two columns of the dW product lie beside unused ones
    cfg = W.MosaConfig("stale_workspace", B=2, T=150, d=264, H=20, hp=128, k=66, dtype="bf16", seed=87)
    x = W.make_inputs(cfg)
    X, Wr, Wq, Wk, Wv, Wo, dY = (to_dev(x[n], "bf16")
                                 for n in ("X", "Wr", "Wq", "Wk", "Wv", "Wo", "dY"))
    got = []
    for fill in (0, 255):
        ws = mosa.alloc_workspace(mosa.make_shape(X, Wq, cfg.k)).fill_(fill)
        _, I, rs, _, ws = mosa.mosa_forward(X, Wr, Wq, Wk, Wv, Wo, cfg.k, workspace=ws)
        got.append(mosa.mosa_backward(X, Wr, Wq, Wk, Wv, Wo, I, rs, dY, ws))
    torch.cuda.synchronize()
    for n in ("dW_r", "dW_q", "dW_k", "dW_v", "dW_o"):
        assert torch.equal(got[0][n], got[1][n]), n


# dW_o, dW_q|dW_k|dW_v and dW_r in four and more reduction splits (the second: of unequal
# length): the same bits from call to call
@pytest.mark.parametrize("cfg", [
    W.MosaConfig("splits_f32", B=3, T=700, d=72, H=2, hp=32, k=345, dtype="f32", seed=88),
    W.MosaConfig("splits_f32_uneven", B=4, T=1600, d=136, H=3, hp=64, k=520, dtype="f32", seed=89),
    W.MosaConfig("splits_bf16", B=8, T=600, d=96, H=2, hp=32, k=300, dtype="bf16", seed=90),
], ids=lambda c: c.name)
def test_weight_gradients_repeat_bit_for_bit(cfg):
    x = W.make_inputs(cfg)
    X, Wr, Wq, Wk, Wv, Wo, dY = (to_dev(x[n], cfg.dtype)
                                 for n in ("X", "Wr", "Wq", "Wk", "Wv", "Wo", "dY"))
    _, I, rs, _, ws = mosa.mosa_forward(X, Wr, Wq, Wk, Wv, Wo, cfg.k)
    first = None
    for _ in range(25):
        g = mosa.mosa_backward(X, Wr, Wq, Wk, Wv, Wo, I, rs, dY, ws)
        if first is None:
            first = g
        for n in ("dW_r", "dW_q", "dW_k", "dW_v", "dW_o"):
            assert torch.equal(first[n], g[n]), n
    ref = oracle.backward(x["X"], *(x[n] for n in ("Wr", "Wq", "Wk", "Wv", "Wo")),
                          I=I.cpu().numpy(), dY=x["dY"])
    for n in ("dW_r", "dW_q", "dW_k", "dW_v", "dW_o"):
        assert_close(n, first[n].cpu().numpy(), ref[n[:2] + n[3:]], cfg.dtype)
