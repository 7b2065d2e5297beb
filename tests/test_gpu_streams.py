"""Layer calls and the caller's streams: launch priorities, calls on several streams, the path
without cached graphs."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2505_00315_gb300 as mosa
from paper_2505_00315_gb300 import workloads as W
from _gpu import to_dev

pytestmark = pytest.mark.gpu

KERNEL_NODE = 0            # CU_GRAPH_NODE_TYPE_KERNEL
ATTRIBUTE_PRIORITY = 8     # CU_LAUNCH_ATTRIBUTE_PRIORITY


def kernel_priorities(stream, call):
    """Priorities of the kernels that ``call`` launches, captured from ``stream``."""
    cu = ctypes.CDLL("libcuda.so.1")

    def ok(rc):
        assert rc == 0, f"CUDA driver error {rc}"

    graph = ctypes.c_void_p()
    ok(cu.cuStreamBeginCapture_v2(ctypes.c_void_p(stream.cuda_stream), 1))
    try:
        call()
    finally:
        ok(cu.cuStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(graph)))
    n = ctypes.c_size_t()
    ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (ctypes.c_void_p * n.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    found = []
    for node in nodes:
        kind, value = ctypes.c_int(), (ctypes.c_int * 16)()
        ok(cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)))
        if kind.value == KERNEL_NODE:
            ok(cu.cuGraphKernelNodeGetAttribute(ctypes.c_void_p(node), ATTRIBUTE_PRIORITY, value))
            found.append(value[0])
    ok(cu.cuGraphDestroy(graph))
    return found


@pytest.mark.parametrize("priority", [0, -1])
@pytest.mark.parametrize("what", ["topk", "layer", "hybrid"])
def test_kernels_run_at_the_priority_of_the_callers_stream(what, priority, monkeypatch):
    monkeypatch.setenv("MOSA_GRAPHS", "0")
    cfg = W.MosaConfig("priority", B=2, T=128, d=64, H=8, hp=64, k=32, dtype="bf16", seed=91)
    x = W.make_inputs(cfg)
    X, *w = (to_dev(x[n], "bf16") for n in ("X", "Wr", "Wq", "Wk", "Wv", "Wo"))
    D = [to_dev(a, "bf16") for a in W.make_dense_weights(cfg, 2).values()]
    stream = torch.cuda.Stream(priority=priority)
    assert stream.priority == priority
    out = {"Y": torch.empty(X.shape, device="cuda"),
           "I": torch.empty((cfg.B, cfg.H, cfg.k), dtype=torch.int32, device="cuda"),
           "r_sel": torch.empty((cfg.B, cfg.H, cfg.k), device="cuda")}
    scores = torch.rand((3, 300), device="cuda")
    top = {"I": torch.empty((3, 9), dtype=torch.int32, device="cuda"),
           "r_sel": torch.empty((3, 9), device="cuda")}
    ws = mosa.alloc_workspace(mosa.make_shape(X, w[1], cfg.k))
    hws = mosa.alloc_hybrid_workspace(mosa.make_hybrid_shape(X, w[1], cfg.k, 2, 64))

    def call():
        if what == "topk":
            mosa.mosa_topk(scores, 9, out=top, stream=stream)
        elif what == "layer":
            mosa.mosa_forward(X, *w, cfg.k, workspace=ws, out=out, stream=stream)
        else:
            mosa.mosa_hybrid_forward(X, *w, *D, cfg.k, window=64, workspace=hws, out=out, stream=stream)

    torch.cuda.synchronize()
    call()   # loads the kernels
    torch.cuda.synchronize()
    found = kernel_priorities(stream, call)
    assert len(found) >= (1 if what == "topk" else 3)
    assert set(found) == {priority}, found


HYBRIDS = [
    (W.MosaConfig("dense_bf16", B=2, T=256, d=128, H=4, hp=64, k=64, dtype="bf16", seed=92), 2, 0),
    (W.MosaConfig("local_large_k", B=2, T=512, d=136, H=5, hp=64, k=160, dtype="bf16", seed=93,
                  rope=True), 3, 256),
    (W.MosaConfig("dense_f32", B=2, T=96, d=48, H=3, hp=32, k=24, dtype="f32", seed=94), 2, 0),
]


class HybridStep:
    """One caller's hybrid layer: tensors, buffers and a forward and backward on its stream."""

    def __init__(self, case, seed):
        self.cfg, self.n, self.window = case
        cfg = self.cfg
        x = W.make_inputs(cfg, seed=seed)
        self.X, *self.w = (to_dev(x[n], cfg.dtype) for n in ("X", "Wr", "Wq", "Wk", "Wv", "Wo"))
        self.D = [to_dev(a, cfg.dtype) for a in W.make_dense_weights(cfg, self.n, seed=seed + 1).values()]
        self.dY = to_dev(x["dY"], cfg.dtype)
        shape = mosa.make_hybrid_shape(self.X, self.w[1], cfg.k, self.n, self.window, rope=cfg.rope)
        self.ws = mosa.alloc_hybrid_workspace(shape)
        self.out, self.grads = {}, {}
        torch.cuda.synchronize()

    def run(self, stream=None):
        cfg = self.cfg
        Y, I, rs, _ = mosa.mosa_hybrid_forward(self.X, *self.w, *self.D, cfg.k, window=self.window,
                                               workspace=self.ws, out=self.out, stream=stream,
                                               rope=cfg.rope)
        self.out.update(Y=Y, I=I, r_sel=rs)
        self.grads.update(mosa.mosa_hybrid_backward(
            self.X, *self.w, *self.D, I, rs, self.dY, self.ws, window=self.window, out=self.grads,
            stream=stream, rope=cfg.rope))

    def results(self):
        torch.cuda.synchronize()
        assert mosa.mosa_check_status(mosa.make_shape(self.X, self.w[1], self.cfg.k), self.ws) == 0
        return {n: t.cpu().numpy().astype(np.float64) for n, t in {**self.out, **self.grads}.items()}


def assert_same(got, ref):
    # the same kernels; the order of the scatter's fp32 additions varies
    for n, r in ref.items():
        assert np.abs(got[n] - r).max() <= 1e-5 * max(1.0, np.abs(r).max()), n


@pytest.mark.parametrize("graphs", ["0", "1"])
@pytest.mark.parametrize("case", HYBRIDS, ids=lambda c: c[0].name)
def test_hybrid_callers_on_two_streams_share_the_internal_ones(case, graphs, monkeypatch):
    refs = []
    for seed in (7, 8):
        step = HybridStep(case, seed)
        step.run()
        refs.append(step.results())
    monkeypatch.setenv("MOSA_GRAPHS", graphs)
    steps = [HybridStep(case, seed) for seed in (7, 8)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream(priority=-1)]
    for _ in range(4):   # without a wait between them
        for step, stream in zip(steps, streams):
            step.run(stream)
    for step, ref in zip(steps, refs):
        assert_same(step.results(), ref)


def test_hybrid_callers_in_two_threads(monkeypatch):
    import threading
    case = HYBRIDS[1]
    refs, steps = [], [HybridStep(case, seed) for seed in (7, 8)]
    for seed in (7, 8):
        step = HybridStep(case, seed)
        step.run()
        refs.append(step.results())
    monkeypatch.setenv("MOSA_GRAPHS", "0")
    failed = []

    def work(step):
        try:
            stream = torch.cuda.Stream()
            for _ in range(6):
                step.run(stream)
        except Exception as e:   # reported by the test's own thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in steps]
    for t in threads:
        t.start()
    for t in threads:
        t.join(60)
    assert not failed, failed
    for step, ref in zip(steps, refs):
        assert_same(step.results(), ref)
