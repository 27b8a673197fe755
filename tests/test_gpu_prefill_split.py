"""GPU parity of the prefill GEMMs where their work items are split between CTAs: a decoder of
d 2048 and MLP 2880 (45 gate/up tiles, so the last pair holds one) with prompts from one token tile
(few items, each shared by many CTAs) to a full pass (whole waves after the split items)."""
import numpy as np
import pytest
import torch

from oracle import tss_oracle as O
from paper_2609_26100_gb300 import native, synth
from tests.conftest import oracle_weights
from tests.parity_util import to_device_weights

pytestmark = pytest.mark.gpu

SEED = synth.DEFAULT_SEED
ARCH = synth.Arch(n_layers=2, d_model=2048, n_heads=16, head_dim=128, d_mlp=2880, vocab=512)


@pytest.fixture(scope="module")
def weights():
    from paper_2609_26100_gb300 import build
    build.build()
    w = synth.make_weights(ARCH, device="cuda")
    return oracle_weights(to_device_weights(w, "cpu")), w


@pytest.mark.parametrize("lengths", [[1], [128], [129, 70], [700], [1900, 1500, 300]])
def test_split_prefill_matches_oracle(weights, lengths):
    """K and V rows of both layers (the second layer's depend on every projection of the first),
    twice into the same cache with the same bits."""
    from paper_2609_26100_gb300.runner import TssRunner
    wo, wg = weights
    run = TssRunner(ARCH, wg, n_slots=len(lengths), kv_cap=2048, max_batch=len(lengths))
    prompts = [synth.uniform_ints(n, ARCH.vocab, SEED, f"split.{b}").tolist() for b, n in enumerate(lengths)]
    got = []
    for _ in range(2):
        run.prefill(prompts, [0] * len(lengths), [0] * len(lengths))
        assert run.sync_status() == native.TSS_OK
        got.append([t.clone() for t in run.kv])
    for l in range(ARCH.n_layers):
        assert torch.equal(got[0][l], got[1][l])
    for b, n in enumerate(lengths):
        ref = O.prefill(wo, ARCH, frozenset(), prompts[b])
        for l in range(ARCH.n_layers):
            for kind in range(2):
                g = got[0][l][b, kind, :, :n].float().cpu().numpy()
                np.testing.assert_allclose(g, ref[l][kind], atol=5e-2, rtol=3e-2, err_msg=f"request {b} layer {l}")
                assert float(np.abs(g - ref[l][kind]).mean()) < 4e-3
    run.close()


@pytest.mark.parametrize("context,lengths", [(900, [1]), (900, [70]), (1023, [130]), (640, [3, 128, 61]), (1921, [128])])
def test_split_attention_matches_oracle(weights, context, lengths):
    """Short prompts appended to a context: the keys of each (head, query tile) split between CTAs, with
    splits that some rows of a tile do not see, and a last split of a few keys."""
    from paper_2609_26100_gb300.runner import TssRunner
    wo, wg = weights
    run = TssRunner(ARCH, wg, n_slots=len(lengths), kv_cap=2080, max_batch=len(lengths))
    prompts = [synth.uniform_ints(context + n, ARCH.vocab, SEED, f"attn.{b}").tolist() for b, n in enumerate(lengths)]
    run.prefill([p[:context] for p in prompts], [0] * len(lengths), [0] * len(lengths))
    got = []
    for _ in range(2):
        run.prefill([p[context:] for p in prompts], [context] * len(lengths), [0] * len(lengths))
        assert run.sync_status() == native.TSS_OK
        got.append([t.clone() for t in run.kv])
    for l in range(ARCH.n_layers):
        assert torch.equal(got[0][l], got[1][l])
    for b, n in enumerate(lengths):
        ref = O.prefill(wo, ARCH, frozenset(), prompts[b])
        for l in range(ARCH.n_layers):
            for kind in range(2):
                g = got[0][l][b, kind, :, context:context + n].float().cpu().numpy()
                r = ref[l][kind][:, context:]
                np.testing.assert_allclose(g, r, atol=5e-2, rtol=3e-2, err_msg=f"request {b} layer {l}")
                assert float(np.abs(g - r).mean()) < 4e-3
    run.close()


def test_wait_for_parts_times_out_and_recovers(weights):
    """Failure injection without a GPU fault: CTA 0 of the first GEMM, whose items are split over all CTAs,
    issues no MMA (tss_inject_timeout); the CTAs that share its item wait for its part until their bound
    (2 s), the call ends with TSS_ERR_TIMEOUT, and the next ones give the bits of a context without it."""
    from paper_2609_26100_gb300.runner import TssRunner
    _, wg = weights
    prompt = synth.uniform_ints(300, ARCH.vocab, SEED, "split.to").tolist()
    out = []
    for fail in (False, True):
        run = TssRunner(ARCH, wg, n_slots=1, kv_cap=512, max_batch=1)
        if fail:
            run.v.inject_timeout(1)
            run.prefill([prompt], [0], [0])
            assert run.sync_status() == native.TSS_ERR_TIMEOUT
        for _ in range(2):
            for t in run.kv:
                t.zero_()
            run.prefill([prompt], [0], [0])
            assert run.sync_status() == native.TSS_OK
            out.append([t.clone() for t in run.kv])
        run.close()
    for o in out[1:]:
        assert all(torch.equal(x, y) for x, y in zip(out[0], o))
