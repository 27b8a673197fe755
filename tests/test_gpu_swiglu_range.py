"""GPU parity of SwiGLU where 1 + exp(-gate) lies between 2^126 and the end of the fp32 range: a decoder
whose first MLP has a few features with gates of -87.5 to -88.5, large up and down weights that bring
their products back to order one, and a second layer whose V projection is the identity, so that the
cache's V rows show the first layer's output."""
import os

import numpy as np
import pytest
import torch

from oracle import tss_oracle as O
from paper_2609_26100_gb300 import native, synth
from tests.conftest import oracle_weights
from tests.parity_util import to_device_weights

pytestmark = pytest.mark.gpu

ARCH = synth.Arch(n_layers=2, d_model=256, n_heads=2, head_dim=128, d_mlp=704, vocab=512)
# (MLP feature, gate / 4, log2 up, log2 down, output dimension): gates of -87.5, -88, -88.5, and ordinary ones
FEATURES = [(3, -21.875, 100, 20, 10), (70, -22.0, 100, 20, 77), (513, -22.125, 100, 20, 200), (64, 0.75, -1, -1, 140),
            (700, -2.0, 4, 4, 255)]


@pytest.fixture(scope="module")
def weights():
    from paper_2609_26100_gb300 import build
    build.build()
    d, f, V = ARCH.d_model, ARCH.d_mlp, ARCH.vocab
    embed = torch.ones((V, d), dtype=torch.bfloat16)
    embed[:, 128:] = synth.uniform_ints(V * 128, 2, 5, "swiglu.sign").view(V, 128).to(torch.bfloat16) * 2 - 1
    layers = []
    for _ in range(2):
        w = {k: torch.zeros(s, dtype=torch.bfloat16) for k, s in synth.layer_shapes(ARCH).items()}
        w["attn_norm"].fill_(1)
        w["mlp_norm"].fill_(1)
        layers.append(w)
    for feat, quarter, up, down, dim in FEATURES:
        layers[0]["w_gate"][feat, :4] = quarter  # (embeddings are 1 there)
        layers[0]["w_up"][feat, 4] = 2.0 ** up
        layers[0]["w_down"][dim, feat] = 2.0 ** down
    layers[1]["wv"] = torch.eye(d, dtype=torch.bfloat16)
    w = {"embed": embed, "lm_head": synth.normal_bf16((V, d), 5, "swiglu.head", 0.05),
         "final_norm": torch.ones(d, dtype=torch.bfloat16), "layers": layers}
    return oracle_weights(w), to_device_weights(w)


@pytest.mark.parametrize("path,n", [("prefill", 37), ("persistent", 5), ("persistent", 21), ("multi", 5)])
def test_gates_near_the_end_of_the_exponential(weights, path, n):
    from paper_2609_26100_gb300.runner import TssRunner
    wo, wg = weights
    os.environ["TSS_PATH"] = "multi" if path == "multi" else "persistent"
    try:
        run = TssRunner(ARCH, wg, n_slots=1, kv_cap=128, max_batch=1, max_nodes=32)
    finally:
        os.environ.pop("TSS_PATH")
    toks = synth.uniform_ints(n, ARCH.vocab, 5, "swiglu.tok").tolist()
    if path == "prefill":
        run.prefill([toks], [0], [0])
    else:
        res = run.alloc_results(1, n)
        run.verify(run.batch([synth.Request(0, synth.chain_parents(n - 1), toks, 0)]), res)
    assert run.sync_status() == native.TSS_OK
    ref = O.prefill(wo, ARCH, frozenset(), toks)[1][1]  # V of layer 1: [head, token, dim]
    moved = sorted(dim for *_, dim in FEATURES)
    flat = np.transpose(ref, (1, 0, 2)).reshape(n, -1)
    assert np.abs(flat[:, moved] / flat[:, [0]] - 1).min() > 0.2  # (every feature shows)
    got = run.kv[1][0, 1, :, :n].float().cpu().numpy()
    np.testing.assert_allclose(got, ref, rtol=2 ** -6, atol=2 ** -8)
    run.close()
