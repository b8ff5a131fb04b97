"""ENCODE of small plans on both sides of the lines of the rule (lq_small_rule.h): blocks of a CTA and clusters that run at once, with
all that test_gpu_small_plans.py compares with the oracle, and which kernels ran."""
import pytest
import torch

from test_gpu_small_plans import test_small_plan as compare_small_plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small, sizes, bits, K, q", [
    # clusters of 16: 13 blocks a CTA, in plans of more than 1024 blocks 12
    (True, [208 * 1024, 100], [8, 3], 2, 2), (False, [208 * 1024 + 1, 100], [4, 3], 2, 2), (True, [207 * 1024 + 1, 0, 9 * 1024], [8, 2, 5], 1, 0),
    (True, [192 * 1024 - 3] * 2, [5, 1], 3, 2), (False, [192 * 1024 + 1] * 2, [5, 1], 3, 2),
    # clusters of 8, 48 at once, 13 blocks a CTA
    (True, [96 * 1024, 95 * 1024 + 700], [8, 1], 24, 2), (False, [96 * 1024, 700], [8, 1], 25, 2),
    (True, [104 * 1024 - 1] * 19, 8, 1, 2), (False, [104 * 1024 + 1] * 19, 5, 1, 2),
    # of 4, 104 at once, and of 2, 222 at once
    (True, [32 * 1024] * 26, 1, 4, 1), (False, [32 * 1024] * 35, 3, 3, 2), (True, [16 * 1024 - 1] * 37, 5, 6, 2), (False, [16 * 1024] * 223, 2, 1, 2),
    (True, [8 * 1024] * 300, 8, 2, 2)])
@pytest.mark.parametrize("hist", [False, True])
def test_small_plan_lines(orc, small, sizes, bits, K, q, hist):
    import paper_2505_14371_b200 as lqm
    compare_small_plan(orc, sizes, bits, K, q, hist)
    plan = lqm.Plan(sizes, bits, q, K, 31)
    plan.lq_profile_enable(True)
    plan.lq_quantize_pack(torch.ones((K, plan.padded_elems), device="cuda"), 1, plan.empty_packed(), plan.empty_norms(),
                          hist=plan.zero_hist() if hist else None)
    ran = {k for k, (_, n) in plan.lq_profile_read().items() if n}
    assert "quantize_pack" in ran and ("norm_partial" in ran) == (not small)
