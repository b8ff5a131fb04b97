"""The decoder where its pieces meet: plans on both sides of the line between warps that share a block and warps with a
block each, worker counts around a unit and around what the value tables hold at once (16 workers at 8 bits), messages
that do not start on a 16-byte boundary.  Sums are in a fixed order: every comparison is exact."""
import numpy as np
import pytest
import torch

from helpers import oracle_model, to_unpadded

pytestmark = pytest.mark.gpu


def _shifted(t):
    """The same values in a contiguous tensor that starts 4 bytes behind a 16-byte boundary."""
    buf = torch.empty(t.numel() + 4, dtype=t.dtype, device=t.device)
    out = buf[1: 1 + t.numel()].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 == 4
    return out


@pytest.mark.parametrize("scope", ["layer", "bucket"])
@pytest.mark.parametrize("sizes, bits, K", [
    ([1025, 5, 4096], [8, 1, 3], 17), ([1025, 5, 4096], [5, 8, 2], 16),
    ([600 * 1024 + 9, 130, 1024], [8, 2, 4], 17), ([600 * 1024 + 9, 33, 2500], [4, 8, 7], 5),
    ([700 * 1024 - 3], [1], 11), ([700 * 1024 - 1000], [6], 3), ([592 * 1024], [2], 7)])
def test_mean_of_messages(orc, scope, sizes, bits, K):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    plan = lqm.Plan(sizes, bits, 2, K, 99)
    plan.lq_set_norm_scope(scope)
    g = torch.Generator(device="cuda").manual_seed(K)
    grads = torch.randn((K, plan.padded_elems), generator=g, device="cuda")
    grads[0, 700:3000] = 0.0
    packed, norms = plan.empty_packed(), plan.empty_norms()
    X1 = torch.randn(plan.padded_elems, generator=g, device="cuda")
    Y, Xh, gbar = torch.empty_like(X1), torch.empty_like(X1), torch.empty_like(X1)
    plan.qoda_init(X1, Y, Xh)
    plan.lq_quantize_pack(grads, 3, packed, norms)
    plan.lq_decode_aggregate(packed, norms, gbar)
    model = oracle_model(orc, plan)
    model.norm_scope = scope
    ref = model.quantize(to_unpadded(plan, grads), 3)
    want = model.mean_decoded(ref["decoded"])
    assert np.array_equal(to_unpadded(plan, gbar), want)
    gbar2 = torch.empty_like(gbar)
    plan.lq_decode_aggregate(_shifted(packed), _shifted(norms), gbar2)
    assert np.array_equal(to_unpadded(plan, gbar2), want)
    gbar3 = torch.empty_like(gbar)
    plan.qoda_step(packed, norms, X1, Y, Xh, None, gbar3)          # the message's own buffer: all-zero blocks are not read
    assert np.array_equal(to_unpadded(plan, gbar3), want)
    assert np.array_equal(to_unpadded(plan, Y), -want)


@pytest.mark.parametrize("layers, size", [(32, 2000), (33, 2000), (64, 2000), (65, 2000), (64, 300000)])
def test_rates_on_both_sides_of_their_rule(layers, size):
    """The step size from 8 x `layers` statistics, formed by the decoder's CTAs or by a kernel before: the sum of what
    lq_get_statistics returns, in another order."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    plan = lqm.Plan([size] * layers, 4, 2, 8, 5)
    g = torch.Generator(device="cuda").manual_seed(layers)
    X1 = torch.randn(plan.padded_elems, generator=g, device="cuda")
    Y, Xh = torch.empty_like(X1), torch.empty_like(X1)
    plan.qoda_init(X1, Y, Xh)
    total = 0.0
    for t in (1, 2):
        packed, norms = plan.empty_packed(), plan.empty_norms()
        plan.lq_quantize_pack(torch.randn((8, plan.padded_elems), generator=g, device="cuda"), t, packed, norms)
        total += float(plan.lq_get_statistics()[0].numpy().sum()) / 64.0
        plan.qoda_step(packed, norms, X1, Y, Xh)
    now, S, eta = plan.qoda_get_scalars()
    assert now == 3 and abs(S - total) <= 8 * layers * 2.0 ** -52 * total and eta == float(np.float32((1.0 + S) ** -0.5))
