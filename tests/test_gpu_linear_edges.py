"""The linear layer's GEMM at the edges of its stages and splits: k-blocks that do not fill a
three-block stage, whole tiles per CTA and tiles split over many, row counts around the 16-row
chunks; against float64."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2609_26100_gb300 import native, synth

pytestmark = pytest.mark.gpu


# (k, n): relative 2-norm error allowed, about twice the largest of 12 measured (m as below, three seeds: 0.48,
# 0.57, 0.71, 1.7 and 4.3 e-7).  The last one's tiles are whole, with four accumulators; with one it is 1.9e-6.
LIMIT = {(64, 128): 1e-7, (128, 384): 1.1e-7, (448, 1280): 1.4e-7, (4160, 256): 3.4e-7, (1920, 12288): 8.5e-7}


@pytest.mark.parametrize("m", [1, 16, 17, 64])
@pytest.mark.parametrize("k,n", list(LIMIT))
def test_linear_static_edges(m, k, n):
    from paper_2609_26100_gb300 import build
    build.build()
    x = synth.normal_bf16((m, k), 11, "edge.x", 1.0).cuda()
    w = synth.normal_bf16((n, k), 11, "edge.w", 0.05).cuda()
    exact = (x.double() @ w.double().T).cpu().numpy()
    got = []
    for _ in range(3):  # (each call finds the arrival counters that the one before left)
        y = torch.full((m, n), float("nan"), dtype=torch.float32, device="cuda")
        native.linear_static(x, w, y)
        assert native.linear_static_status() == native.TSS_OK
        got.append(y.cpu().numpy())
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
    assert np.linalg.norm(got[0] - exact) <= LIMIT[k, n] * np.linalg.norm(exact)
    # (the largest error over the largest output measured at most 2.1 times the norms' ratio)
    assert np.abs(got[0] - exact).max() <= 4 * LIMIT[k, n] * np.abs(exact).max()


def captured_nodes(call):
    """The kinds of the graph nodes (0 kernel, 2 memset), sorted, that call(stream) enqueues."""
    rt = ctypes.CDLL("libcudart.so.13")
    stream = torch.cuda.Stream()
    s, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(s, 1) == 0  # (thread-local)
    try:
        call(stream.cuda_stream)
    finally:
        assert rt.cudaStreamEndCapture(s, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes, kinds = (ctypes.c_void_p * n.value)(), []
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    for node in nodes:
        kind = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    assert rt.cudaGraphDestroy(graph) == 0
    return sorted(kinds)


@pytest.mark.parametrize("k,n,kinds", [(4160, 256, [0, 2]), (1920, 12288, [0])])
def test_static_counters_are_cleared_by_every_call_that_uses_them(k, n, kinds):
    """What an earlier call left in the arrival counters (overlapping calls may leave anything) does not
    reach a later one: shared tiles' counters are cleared in stream order, whole tiles use none."""
    x = torch.ones((4, k), dtype=torch.bfloat16, device="cuda")
    w = torch.ones((n, k), dtype=torch.bfloat16, device="cuda")
    y = torch.empty((4, n), dtype=torch.float32, device="cuda")
    native.linear_static(x, w, y)  # (the first call on a device sets it up)
    assert native.linear_static_status() == native.TSS_OK
    assert captured_nodes(lambda s: native.linear_static(x, w, y, s)) == kinds
