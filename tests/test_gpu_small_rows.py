"""ENCODE of small plans, a row of 128 coordinates a warp: layers that end inside a row, inside a lane's four coordinates and on
the edges of rows and blocks, rows without values now or before, many (layer, worker) pairs of one CTA each, clusters of every
size up to 16, every code width, and layers sent as zeros; against the oracle.  The same plan encoded for one worker of a range.
The last, partial blocks of large layers are encoded by the same rows, behind the whole blocks of the general encoder."""
import numpy as np
import pytest
import torch

from helpers import compare_messages, oracle_model, to_unpadded

pytestmark = pytest.mark.gpu
ENDS = [1, 3, 4, 127, 128, 129, 255, 511, 513, 900, 1023, 1024, 1025, 1151, 2047, 3000]


@pytest.mark.parametrize("sizes, bits, K, q", [
    (ENDS, 3, 5, 2), (ENDS * 4, 5, 7, 2), ([8 * 1024 - 1] + ENDS, 8, 2, 0), ([9 * 1024, 5, 129], 1, 2, 1),
    ([5 * 1024 + 385], 6, 1, 2), ([17 * 1024 + 2], 7, 2, 3), ([16 * 1024 - 130, 77], 2, 3, 2), ([40 * 1024 + 1, 600], 4, 16, 2),
    (ENDS[:8] + [30 * 1024], [1, 2, 3, 4, 5, 6, 7, 8, 8], 4, 2),
    ([257 * 1024 + 3, 129], 3, 2, 2), ([258 * 1024 + 900, 1023, 2048], 8, 2, 0), ([257 * 1024 + 385, 511], 5, 1, 1),
    ([257 * 1024 + 129] + ENDS[:8], [7, 1, 2, 3, 4, 5, 6, 7, 8], 2, 2)])
@pytest.mark.parametrize("hist", [False, True])
def test_rows_of_small_plans(orc, sizes, bits, K, q, hist):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    plan, part = (lqm.Plan(sizes, bits, q, K, 41) for _ in range(2))
    part.lq_set_worker_range(K - 1, 1)
    model = oracle_model(orc, plan)
    g = torch.Generator(device="cuda").manual_seed(len(sizes) + K)
    X1 = torch.randn(plan.padded_elems, generator=g, device="cuda")
    Y, Xh = torch.empty_like(X1), torch.empty_like(X1)
    plan.qoda_init(X1, Y, Xh); model.qoda_init(to_unpadded(plan, X1))
    pk, nm = [[p.empty_packed(), p.empty_packed()] for p in (plan, part)], [[p.empty_norms(), p.empty_norms()] for p in (plan, part)]
    sum_tol = max(1e-12, 2.0 * K * sum(sizes) * 2.0 ** -53)      # fp64 sums of non-negative terms in two orders
    for t in (1, 2, 3):
        grads = torch.randn((K, plan.padded_elems), generator=g, device="cuda") ** 3
        dead = torch.rand((K, plan.padded_elems // 32), generator=g, device="cuda") < 0.4
        grads.view(K, -1, 32)[dead] = 0.0
        for k in range(K):                                       # whole rows, other ones each time
            for o, n in zip(plan.elem_offsets, sizes):
                for row in range(0, n, 128):
                    if (row // 128 + k + t) % 3 == 0:
                        grads[k, o + row: o + min(row + 128, n)] = 0.0
        if t == 2:
            grads[0, plan.elem_offsets[-1] + sizes[-1] - 1] = float("nan")
        c, p = t % 2, (t + 1) % 2
        h = plan.zero_hist() if hist else None
        plan.lq_quantize_pack(grads, t, pk[0][c], nm[0][c], hist=h, prev_packed=pk[0][p] if t > 1 else None, prev_norms=nm[0][p] if t > 1 else None)
        part.lq_quantize_pack(grads[K - 1:].contiguous(), t, pk[1][c], nm[1][c], prev_packed=pk[1][p] if t > 1 else None,
                              prev_norms=nm[1][p] if t > 1 else None)
        ref = model.quantize(to_unpadded(plan, grads), t, want_hist=hist)
        assert compare_messages(orc, plan, pk[0][c], ref) == (0, 0)
        assert np.array_equal(nm[0][c].cpu().numpy(), ref["norms"])
        assert torch.equal(pk[0][c][K - 1], pk[1][c][K - 1]) and torch.equal(nm[0][c][K - 1], nm[1][c][K - 1])
        sq, flags = plan.lq_get_statistics()
        assert np.array_equal(flags.numpy(), ref["status"])
        want = np.asarray(ref["sq_diff"], np.float64)
        assert np.max(np.abs(sq.numpy() - want)) <= sum_tol * max(np.max(np.abs(want)), 1e-300)
        assert torch.equal(sq[K - 1], part.lq_get_statistics()[0][K - 1])
        if hist:
            assert np.array_equal(h.cpu().numpy().view(np.uint32), ref["hist"])
        plan.qoda_step(pk[0][c], nm[0][c], X1, Y, Xh); model.qoda_step()
        assert np.max(np.abs(to_unpadded(plan, Y) - model.Y)) <= 1e-6 * np.max(np.abs(model.Y))
