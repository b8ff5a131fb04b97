"""ENCODE of a plan with layers of several code widths and many waves of CTAs, which take the tiles width by width.
Messages, norms and flags against the oracle bit by bit, the statistic within the tolerance of its summation order."""
import numpy as np
import pytest
import torch

from helpers import compare_messages, oracle_model, to_unpadded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [[1, 2, 3, 4, 5, 6, 7, 8], [8, 3]])
def test_layers_of_several_widths(orc, widths):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    rng = np.random.default_rng(len(widths))
    L, K = 620, 8                                        # 4960 CTAs at least: every layer is a tile or more
    sizes = [int(x) for x in rng.choice([1, 31, 1023, 1024, 1025, 1500, 2049, 9000], L)]
    bits = [widths[i % len(widths)] for i in range(L)]
    plan = lqm.Plan(sizes, bits, 2, K, 17)
    model = oracle_model(orc, plan)
    g = torch.Generator(device="cuda").manual_seed(2)
    pk, nm = [plan.empty_packed(), plan.empty_packed()], [plan.empty_norms(), plan.empty_norms()]
    sum_tol = max(1e-12, 2.0 * K * max(sizes) * 2.0 ** -53)       # fp64 sums of a layer's terms in two different orders
    for t in (1, 2):
        grads = torch.randn((K, plan.padded_elems), generator=g, device="cuda")
        grads[1, 5000:40000] = 0.0
        c, p = t % 2, (t + 1) % 2
        plan.lq_quantize_pack(grads, t, pk[c], nm[c], prev_packed=pk[p] if t > 1 else None, prev_norms=nm[p] if t > 1 else None)
        ref = model.quantize(to_unpadded(plan, grads), t)
        assert compare_messages(orc, plan, pk[c], ref) == (0, 0)
        assert np.array_equal(nm[c].cpu().numpy(), ref["norms"])
        sq, flags = plan.lq_get_statistics()
        assert np.array_equal(flags.numpy(), ref["status"])
        want = np.asarray(ref["sq_diff"], np.float64)
        assert np.max(np.abs(sq.numpy() - want)) <= sum_tol * max(np.max(np.abs(want)), 1e-300)
        model.prev_decoded = model.cur_decoded
