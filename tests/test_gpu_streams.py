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
