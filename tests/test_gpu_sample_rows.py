"""GPU parity of the speculative-sampling acceptance over block sizes: the rows' statistics are
computed by one block each and the walk by the block that finishes a request's last row, for blocks
of one to 128 rows, also very different ones in one step, rejected at the first, a middle and no draft, alone and as
a group of a split batch (results and inputs at the caller's places)."""
import numpy as np
import pytest
import torch

from oracle import tss_oracle as O
from paper_2609_26100_gb300 import native, synth
from tests.conftest import oracle_weights
from tests.parity_util import assert_logits, check_sample, to_device_weights

pytestmark = pytest.mark.gpu

ARCH = synth.TINY
SEED = synth.DEFAULT_SEED


@pytest.mark.parametrize("sizes", [[1, 64, 2, 33], [1, 128, 2, 16]])
@pytest.mark.parametrize("grouped", [False, True])
@pytest.mark.parametrize("stop", ["first", "middle", "none"])
def test_sampling_block_sizes(grouped, stop, sizes):
    from paper_2609_26100_gb300 import build
    from paper_2609_26100_gb300.runner import TssRunner
    build.build()
    w = synth.make_weights(ARCH)
    wo = oracle_weights(w)
    run = TssRunner(ARCH, to_device_weights(w), n_slots=4, kv_cap=256, max_batch=4, max_nodes=128)
    phi = {0: 0b0010, 1: 0}
    run.set_phi(phi)
    reqs, skips, q, unif = [], [], [], np.zeros((4, 2 * 127 + 1), dtype=np.float32)
    for b, n in enumerate(sizes):
        parents = synth.chain_parents(n - 1)
        toks = synth.uniform_ints(n, ARCH.vocab, SEED, f"rows.tok{b}").tolist()
        reqs.append(synth.Request(8 + b, parents, toks, b % 2))
        skips.append(O.mask_to_set(phi[b % 2]))
        # flat drafts with small uniforms are accepted (p V is near one); a one-hot draft is rejected
        qb = np.full((n, ARCH.vocab), 1.0 / ARCH.vocab, dtype=np.float32)
        unif[b] = synth.uniform01(unif.shape[1], SEED, f"rows.u{b}").numpy().astype(np.float32)
        unif[b, :n - 1] *= 0.01
        at = {"first": 1, "middle": n // 2, "none": 0}[stop]
        if 0 < at < n:
            qb[at] = 0.0
            qb[at, toks[at]] = 1.0
            unif[b, at - 1] = 0.9
        q.append(qb)
    kv = {}
    for b, r in enumerate(reqs):
        for l in range(ARCH.n_layers):
            if l not in skips[b]:
                blk = synth.kv_block(ARCH, l, b, r.ctx_len, SEED, device="cuda")
                run.kv[l][b, :, :, :r.ctx_len] = blk
                f = blk.float().cpu().numpy()
                kv[(b, l)] = (f[0], f[1])
    res = run.alloc_results(4, sum(sizes), path_stride=128)
    batch = run.batch(reqs, mode=native.TSS_MODE_SAMPLE, temperature=1.0, uniforms=torch.from_numpy(unif).cuda(),
                      draft_probs=torch.from_numpy(np.concatenate(q)).cuda())
    for _ in range(2):  # (the second pass finds the arrival counters reset)
        (run.verify_grouped if grouped else run.verify)(batch, res)
    assert run.sync_status() == native.TSS_OK
    refs = O.verify_requests(wo, ARCH, skips, [(r.tokens, r.parents, r.ctx_len) for r in reqs], lambda b, l: kv[(b, l)])
    gl, row = res["logits"].cpu().numpy(), 0
    for b, (r, (ref, _)) in enumerate(zip(reqs, refs)):
        n = len(r.parents)
        assert_logits(gl[row:row + n], ref, f"rows request {b}")
        ga, gb = int(res["accept_len"][b]), int(res["bonus"][b])
        check_sample(ref, gl[row:row + n], r.tokens, q[b], unif[b].astype(np.float64), 1.0, ga, gb, f"rows request {b}")
        assert res["path"][b, :ga + 1].tolist() == list(range(ga + 1)) and int(res["new_ctx_len"][b]) == r.ctx_len + 1 + ga
        row += n
    run.close()
