"""GPU parity of the persistent kernel's epilogues over the row counts of a step, on a decoder wide
enough that every projection's tiles are split between CTAs (3 layers, d 2048, MLP 2816) and a
vocabulary whose rows are not a multiple of 16 bytes: the two ways a split tile is finished (last
arriver up to 8 rows, every contributor beyond), the edges of its row groups, the tiny decoder's
tiles of a few k-blocks, and batches whose requests skip different layers (rows that join or leave between
two layers)."""
import numpy as np
import pytest
import torch

from oracle import tss_oracle as O
from paper_2609_26100_gb300 import native, synth
from tests.conftest import oracle_weights
from tests.parity_util import assert_logits, to_device_weights

pytestmark = pytest.mark.gpu

SEED = synth.DEFAULT_SEED
ARCHS = {
    "wide64": synth.Arch(n_layers=3, d_model=2048, n_heads=32, head_dim=64, d_mlp=2816, vocab=2001),
    "wide128": synth.Arch(n_layers=3, d_model=2048, n_heads=16, head_dim=128, d_mlp=2816, vocab=2001),
    "tiny": synth.TINY,
}
# block sizes of the requests: 8 and 9 rows (the edge between the two ways), 16 / 17 (a second
# 16-row chunk), 61 in one block, 85 (more (request, head) items than SMs, most of small blocks: the
# warp-level attention at either head size), 129 (two operand blocks per k-block) and the most rows of a step
BLOCKS = {1: [1], 8: [3, 5], 9: [4, 2, 3], 16: [16], 17: [9, 8], 61: [61], 85: [40] + [5] * 9, 129: [9] * 13 + [12], 256: [16] * 16}
PHI = {0: 0b010, 1: 0b101, 2: 0}


@pytest.fixture(scope="module")
def weights():
    from paper_2609_26100_gb300 import build
    build.build()
    made = {}

    def get(name):
        if name not in made:
            made.clear()
            w = synth.make_weights(ARCHS[name], device="cuda")
            made[name] = (oracle_weights(to_device_weights(w, "cpu")), w)
        return made[name]

    return get


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("rows", sorted(BLOCKS))
@pytest.mark.parametrize("name", sorted(ARCHS))
def test_rows_match_oracle(weights, name, rows, mixed):
    from paper_2609_26100_gb300.runner import TssRunner
    a = ARCHS[name]
    wo, wg = weights(name)
    blocks = BLOCKS[rows]
    reqs = []
    for b, n in enumerate(blocks):
        parents = synth.chain_parents(n - 1)
        reqs.append(synth.Request(20 + 7 * b, parents, synth.draft_tokens(parents, a.vocab, SEED, f"rows.{b}"),
                                  b % 3 if mixed else 2))
    run = TssRunner(a, wg, n_slots=len(reqs), kv_cap=220, max_batch=len(reqs))
    run.set_phi(PHI)
    skips = [O.mask_to_set(PHI[r.domain]) for r in reqs]
    kv = {}
    for b, r in enumerate(reqs):
        for l in range(a.n_layers):
            if l not in skips[b]:
                blk = synth.kv_block(a, l, b, r.ctx_len, SEED, device="cuda")
                run.kv[l][b, :, :, :r.ctx_len] = blk
                f = blk.float().cpu().numpy()
                kv[(b, l)] = (f[0], f[1])
    got = []
    for _ in range(2):
        res = run.alloc_results(len(reqs), rows)
        run.verify(run.batch(reqs), res)
        assert run.sync_status() == native.TSS_OK
        got.append(res["logits"].cpu().numpy())
    assert np.array_equal(got[0], got[1])  # sums are added in a fixed order
    refs = O.verify_requests(wo, a, skips, [(r.tokens, r.parents, r.ctx_len) for r in reqs], lambda b, l: kv[(b, l)])
    assert_logits(got[0], np.concatenate([ref for ref, _ in refs]), f"{name} rows {rows} mixed {mixed}")
    run.close()
    torch.cuda.empty_cache()


@pytest.mark.parametrize("rows", [9, 129])
def test_wait_for_parts_times_out_and_recovers(weights, rows, monkeypatch):
    """Failure injection without a GPU fault: one part of a tile that several CTAs finish together is not
    counted (tss_inject_timeout), so their waits for it run out; the step ends with TSS_ERR_TIMEOUT, and
    the next steps match one of a context without the failure."""
    from paper_2609_26100_gb300.runner import TssRunner
    a = ARCHS["wide128"]
    _, wg = weights("wide128")
    blocks = BLOCKS[rows]
    reqs = []
    for b, n in enumerate(blocks):
        parents = synth.chain_parents(n - 1)
        reqs.append(synth.Request(20 + 7 * b, parents, synth.draft_tokens(parents, a.vocab, SEED, f"rows.{b}"), 2))
    monkeypatch.setenv("TSS_WAIT_LIMIT_MS", "200")
    out = []
    for fail in (False, True):
        run = TssRunner(a, wg, n_slots=len(reqs), kv_cap=220, max_batch=len(reqs))
        for b, r in enumerate(reqs):
            for l in range(a.n_layers):
                run.kv[l][b, :, :, :r.ctx_len] = synth.kv_block(a, l, b, r.ctx_len, SEED, device="cuda")
        res = run.alloc_results(len(reqs), rows)
        if fail:
            run.v.inject_timeout(1)
            run.verify(run.batch(reqs), res)
            assert run.sync_status() == native.TSS_ERR_TIMEOUT
        for _ in range(2):
            run.verify(run.batch(reqs), res)
            assert run.sync_status() == native.TSS_OK
            out.append(res["logits"].cpu().numpy())
        run.close()
    for o in out[1:]:
        assert np.array_equal(out[0], o)
