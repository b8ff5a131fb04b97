"""ENCODE of plans whose layers are all small (one cluster per layer and worker): sizes around a cluster's capacity, CTAs of
a cluster that have no block, empty layers, worker ranges; messages, norms and flags against the oracle bit by bit (the zero-row
masks through the updates and statistics that leave rows out by them), the statistic within the tolerance of its summation
order."""
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


def test_worker_range_keeps_the_order_of_the_sums():
    """A plan whose clusters for all 8 workers are more than the small path takes, while those of one worker alone would not
    be: a process of one worker emits the messages, norms and statistic of the process of all, to the last bit."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    sizes, K = [33 * 1024 + 5] * 20, 8
    whole, part = lqm.Plan(sizes, 3, 2, K, 7), lqm.Plan(sizes, 3, 2, K, 7)
    part.lq_set_worker_range(5, 1)
    g = torch.Generator(device="cuda").manual_seed(3)
    pk = [[p.empty_packed(), p.empty_packed()] for p in (whole, part)]
    nm = [[p.empty_norms(), p.empty_norms()] for p in (whole, part)]
    for t in (1, 2, 3):
        grads = torch.randn((K, whole.padded_elems), generator=g, device="cuda")
        c, p = t % 2, (t + 1) % 2
        for i, (plan, rows) in enumerate(((whole, grads), (part, grads[5:6].contiguous()))):
            plan.lq_quantize_pack(rows, t, pk[i][c], nm[i][c], prev_packed=pk[i][p] if t > 1 else None,
                                  prev_norms=nm[i][p] if t > 1 else None)
        assert torch.equal(pk[0][c][5], pk[1][c][5]) and torch.equal(nm[0][c][5], nm[1][c][5])
        a, b = (plan.lq_get_statistics()[0][5] for plan in (whole, part))
        assert torch.equal(a, b)


def test_layer_norms_are_the_norms_of_the_message():
    """A sum that lies half way between two floats up to terms that a large partial sum swallows and a small one keeps: the
    order of the additions decides the norm, so both calls have to use the same."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    plan = lqm.Plan([196 * 1024, 5], 3, 1, 2, 7)
    grads = torch.zeros((2, plan.padded_elems), device="cuda")
    grads[:, 0], grads[:, 1] = 2.0 ** 24, 1.0                   # 2^24 + 1: between 2^24 and 2^24 + 2
    for blk, worker in ((8, 0), (16, 0), (24, 1), (100, 1)):
        grads[worker, blk * 1024: blk * 1024 + 4] = 2.0 ** -30  # lost one by one beside 2^24, not 4 of them together
    alone, sent = plan.empty_norms(), plan.empty_norms()
    plan.lq_layer_norms(grads, alone)
    plan.lq_quantize_pack(grads, 1, plan.empty_packed(), sent)
    assert torch.equal(alone, sent)
