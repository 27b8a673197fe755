"""GPU parity of the tcgen05 attention's work split, whose ranges weigh an item's fixed cost as well as
its tiles: one-tile items beside long ones, a step with fewer units than CTAs, and requests that
skip the layer between others."""
import pytest

from tests.test_gpu_tc_attention import TC, Case, chain, make_runner, weights  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctxs", [[1], [120, 3], [5, 3000, 122, 123, 1, 700, 60, 2500], [2000] * 8])
def test_ranges_match_oracle(weights, ctxs):  # noqa: F811
    wo, wg = weights
    run = make_runner(wg, n_slots=8, cap=3072, path="hybrid")
    reqs = [chain(c, 5 if b % 3 else 0, f"ranges.{b}", domain=b % 2) for b, c in enumerate(ctxs)]
    case = Case(run, reqs, {0: 0, 1: 0b010})
    res = case.step()
    assert run.v.attention_kernel() == TC
    case.check(wo, res, f"ranges {ctxs}")
    run.close()
