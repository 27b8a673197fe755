"""The sums of a projection's tile keep what parts of one 64-column block each, added in fp32, keep: on a
small decoder (every tile split by its k-blocks), value weights of 2^20 and -2^20 in the first and the
last block and, between them, terms that are each below half an ulp of 2^20 but whose sum over a block is
not.  One accumulator over the whole tile loses them all."""
import numpy as np
import pytest
import torch

from paper_2609_26100_gb300 import native, synth

pytestmark = pytest.mark.gpu

SMALL = 0.44921875 / 8  # 0.45 ulp (2^-3) of 2^20, one term per 16 columns
CASES = {"64": (4, 64), "128": (2, 128)}  # heads, head_dim


@pytest.mark.parametrize("n", [1, 8, 9, 40])
@pytest.mark.parametrize("shape", sorted(CASES))
def test_tile_keeps_terms_below_an_ulp(shape, n):
    from paper_2609_26100_gb300 import build
    from paper_2609_26100_gb300.runner import TssRunner
    build.build()
    H, D = CASES[shape]
    a = synth.Arch(n_layers=1, d_model=256, n_heads=H, head_dim=D, d_mlp=704, vocab=512)
    w = {"embed": torch.ones((a.vocab, a.d_model)), "lm_head": torch.zeros((a.vocab, a.d_model)),
         "final_norm": torch.ones(a.d_model), "layers": [{k: torch.zeros(s) for k, s in synth.layer_shapes(a).items()}]}
    w["layers"][0]["attn_norm"].fill_(1)
    w["layers"][0]["mlp_norm"].fill_(1)
    wv = w["layers"][0]["wv"]
    wv[:, 0], wv[:, 255], wv[:, 64:192:16] = 2.0 ** 20, -(2.0 ** 20), SMALL
    w["layers"] = [{k: t.to(torch.bfloat16).cuda() for k, t in w["layers"][0].items()}]
    w.update({k: w[k].to(torch.bfloat16).cuda() for k in ("embed", "lm_head", "final_norm")})
    run = TssRunner(a, w, n_slots=1, kv_cap=64, max_batch=1)
    res = run.alloc_results(1, n)
    run.verify(run.batch([synth.Request(0, synth.chain_parents(n - 1), [3] * n, 0)]), res)
    assert run.sync_status() == native.TSS_OK
    got = run.kv[0][0, 1, :, :n].float().cpu().numpy()
    # exact: 8 terms = 3.6 ulp of 2^20; each 64-column part of 1.8 ulp is rounded to 2 when it is added
    np.testing.assert_allclose(got, 8 * SMALL, rtol=0.15)
    run.close()
