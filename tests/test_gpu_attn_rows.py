"""GPU parity of the tcgen05 attention for blocks of more than 16 rows (head_dim 128, separate
attention launches): blocks of 17 rows to the largest, ends of blocks and contexts on tile
boundaries, one split and many (merged partials), requests of very different size in one step and
ones that skip a layer, NaN cache rows past the keys; and against the warp-level kernel."""
import os
import time

import numpy as np
import pytest
import torch

from paper_2609_26100_gb300 import native, synth
from tests.test_gpu_tc_attention import ARCH, SEED, Case, chain, weights  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def runner(wg, n_slots, splits=0, tc=True):
    from paper_2609_26100_gb300.runner import TssRunner
    env = {"TSS_ATTN": "external", "TSS_ATTN_SPLITS": str(splits), "TSS_ATTN_TC": "1" if tc else "0"}
    os.environ.update(env)
    try:
        return TssRunner(ARCH, wg, n_slots=n_slots, kv_cap=1300, max_batch=4, max_nodes=128)
    finally:
        for k in env:
            os.environ.pop(k, None)


def tree(ctx, n, tag, domain=0):
    parents = synth.eagle_tree(n - 1, (8, 4, 3, 2, 2, 1, 1, 1))
    return synth.Request(ctx, parents, synth.draft_tokens(parents, ARCH.vocab, SEED, tag), domain)


CASES = {
    "one": lambda: [tree(1000, 61, "ar.0")],
    "edges": lambda: [tree(64, 64, "ar.1"), tree(63, 17, "ar.2", 1), tree(1, 65, "ar.3"), tree(127, 33, "ar.4", 1)],
    "largest": lambda: [tree(777, 128, "ar.5"), tree(1152, 128, "ar.6", 1)],
    "mixed": lambda: [chain(300, 0, "ar.7"), tree(1100, 100, "ar.8", 1), chain(5, 3, "ar.9"), chain(640, 23, "ar.10")],
}


@pytest.mark.parametrize("splits", [0, 1, 5])
@pytest.mark.parametrize("name", sorted(CASES))
def test_rows_attention_matches_oracle(weights, name, splits):  # noqa: F811
    wo, wg = weights
    reqs = CASES[name]()
    run = runner(wg, len(reqs), splits)
    case = Case(run, reqs, {0: 0, 1: 0b010})
    res = case.step()
    assert run.v.attention_kernel() == (2 if max(len(r.parents) for r in reqs) > 64 else 0)
    first = res["logits"].clone()
    case.check(wo, res, f"rows attention {name} splits {splits}")
    res = case.step()
    assert torch.equal(first, res["logits"])  # partials are added in split order
    run.close()


def test_rows_attention_close_to_warp_kernel(weights):  # noqa: F811
    wo, wg = weights
    out = []
    for tc in (True, False):
        run = runner(wg, 2, tc=tc)
        out.append(Case(run, CASES["largest"](), {0: 0, 1: 0b010}).step()["logits"].cpu().numpy())
        run.close()
    assert np.abs(out[0] - out[1]).max() < 2e-2


@pytest.mark.parametrize("splits", [1, 5])
def test_rows_attention_bounded_wait_times_out_and_recovers(weights, splits, monkeypatch):  # noqa: F811
    """Failure injection without a GPU fault: one CTA of the step's first attention launch issues no MMA
    (tss_inject_timeout), so the kernel's waits run out after their 2 s (the persistent kernel's would
    after 200 ms), the step ends with TSS_ERR_TIMEOUT and the next ones match the oracle."""
    wo, wg = weights
    monkeypatch.setenv("TSS_WAIT_LIMIT_MS", "200")
    run = runner(wg, 2, splits)
    case = Case(run, CASES["largest"](), {0: 0, 1: 0b010})
    case.step()
    run.v.inject_timeout(1)
    res = run.alloc_results(2, 256, path_stride=129)
    t0 = time.monotonic()
    run.verify(run.batch(case.reqs), res)
    assert run.sync_status() == native.TSS_ERR_TIMEOUT
    assert 1.9 < time.monotonic() - t0 < 6.0
    assert run.sync_status() == native.TSS_OK  # reported once, then cleared
    for _ in range(2):
        for l in range(ARCH.n_layers):  # the failed step's appends are discarded
            for b, r in enumerate(case.reqs):
                run.kv[l][b, :, :, r.ctx_len:].fill_(float("nan"))
        case.check(wo, case.step(), f"after a timeout, splits {splits}")
    run.close()
