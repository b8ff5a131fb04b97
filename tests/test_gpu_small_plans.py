"""ENCODE of plans whose layers are all small (one cluster per layer and worker): sizes around a cluster's capacity, CTAs of
a cluster that have no block, empty layers, worker ranges; messages, norms, flags and masks against the oracle bit by bit, the
statistic within the tolerance of its summation order."""
import numpy as np
import pytest
import torch

from helpers import compare_messages, oracle_model, to_unpadded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes, bits, K, q", [
    ([256 * 1024, 100], [4, 3], 2, 2), ([256 * 1024 + 1, 100], [4, 3], 2, 2), ([255 * 1024 + 1, 0, 9 * 1024], [8, 2, 5], 1, 0),
    ([8 * 1024], [4], 8, 1), ([8 * 1024 + 1, 17 * 1024 - 3], [3, 6], 3, 3), ([1, 0, 31], [1, 4, 8], 9, 2)])
@pytest.mark.parametrize("hist", [False, True])
def test_small_plan(orc, sizes, bits, K, q, hist):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    plan = lqm.Plan(sizes, bits, q, K, 31)
    model = oracle_model(orc, plan)
    g = torch.Generator(device="cuda").manual_seed(5)
    X1 = torch.randn(plan.padded_elems, generator=g, device="cuda")
    Y, Xh = torch.empty_like(X1), torch.empty_like(X1)
    plan.qoda_init(X1, Y, Xh); model.qoda_init(to_unpadded(plan, X1))
    pk, nm = [plan.empty_packed(), plan.empty_packed()], [plan.empty_norms(), plan.empty_norms()]
    # fp64 sums of D * K non-negative terms in two different orders
    sum_tol = max(1e-12, 2.0 * K * sum(sizes) * 2.0 ** -53)
    for t in (1, 2, 3):
        grads = torch.randn((K, plan.padded_elems), generator=g, device="cuda")
        grads[K - 1, 512: 9000] = 0.0
        if t == 3 and sizes[0] > 2000:
            grads[0, sizes[0] - 1] = float("inf")               # the last CTA of the cluster sees it, all send zeros
        c, p = t % 2, (t + 1) % 2
        h = plan.zero_hist() if hist else None
        plan.lq_quantize_pack(grads, t, pk[c], nm[c], hist=h, prev_packed=pk[p] if t > 1 else None,
                              prev_norms=nm[p] if t > 1 else None)
        ref = model.quantize(to_unpadded(plan, grads), t, want_hist=hist)
        assert compare_messages(orc, plan, pk[c], ref) == (0, 0)
        assert np.array_equal(nm[c].cpu().numpy(), ref["norms"])
        sq, flags = plan.lq_get_statistics()
        assert np.array_equal(flags.numpy(), ref["status"])
        want = np.asarray(ref["sq_diff"], np.float64)
        assert np.max(np.abs(sq.numpy() - want)) <= sum_tol * max(np.max(np.abs(want)), 1e-300)
        if hist:
            assert np.array_equal(h.cpu().numpy().view(np.uint32), ref["hist"])
        plan.qoda_step(pk[c], nm[c], X1, Y, Xh); model.qoda_step()
        assert np.max(np.abs(to_unpadded(plan, Y) - model.Y)) <= 1e-6 * np.max(np.abs(model.Y))
