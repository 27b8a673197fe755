"""The linear layer's GEMM at the edges of its stages and splits: k-blocks that do not fill a
three-block stage, whole tiles per CTA and tiles split over many, row counts around the 16-row
chunks; against float64 and, for the context's entry point, the same values."""
import numpy as np
import pytest
import torch

from paper_2609_26100_gb300 import native, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 16, 17, 64])
@pytest.mark.parametrize("k,n", [(64, 128), (128, 384), (448, 1280), (4160, 256), (1920, 12288)])
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
    # fp32 sums of k products of bf16 values: relative to the largest output
    assert np.abs(got[0] - exact).max() <= 2 ** -24 * k * np.abs(exact).max()
