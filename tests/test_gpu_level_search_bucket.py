"""The level searches at the values of test_gpu_level_search.py in the bucket scope, and in all three encoders at 7 bits."""
import numpy as np
import pytest

from helpers import compare_messages, oracle_model, to_padded
from test_gpu_level_search import _levels, test_values_on_and_beside_levels as compare_layer_scope

pytestmark = pytest.mark.gpu
KINDS = ["edges", "beside", "next_to_1", "shared"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("size", [3 * 1024, 300 * 1024 + 77])        # the kernel of small plans, and the general one
def test_seven_bits(orc, size, kind):
    compare_layer_scope(orc, size, kind, 7)


@pytest.mark.parametrize("bits", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("kind", KINDS)
def test_values_on_and_beside_levels_by_bucket(orc, kind, bits):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    n, K, size = 1 << bits, 2, 40 * 1024 + 77
    levels = _levels(kind, n)
    plan = lqm.Plan([size], bits, 0, K, 77 + bits)
    plan.lq_set_norm_scope("bucket")
    plan.lq_set_levels(0, [float(x) for x in levels])
    one = np.float32(1.0)
    special = np.concatenate([levels, np.nextafter(levels, one), np.nextafter(levels, np.float32(0)), np.float32([1e-45, 1e-38, 2.0 ** -126, 2.0 ** -64]),
                              np.nextafter(np.float32(2.0) ** -np.arange(0, 30, dtype=np.float32), np.float32(0))]).astype(np.float32)
    special = special[(special >= 0) & (special <= 1)]
    rng = np.random.default_rng(bits)
    v = (rng.choice(special, (K, size)) * rng.choice(np.float32([1.0, -1.0]), (K, size))).astype(np.float32)      # (-0 among them)
    v[:, ::128] = 1.0                                        # every bucket's norm
    v[:, 2048:2304] = -0.0
    grads = to_padded(plan, v)
    model = oracle_model(orc, plan)
    model.norm_scope = "bucket"
    packed, norms = [plan.empty_packed() for _ in range(2)], [plan.empty_norms() for _ in range(2)]
    for t in (1, 2):
        hist = plan.zero_hist()
        plan.lq_quantize_pack(grads, t, packed[t % 2], norms[t % 2], hist=hist if t == 1 else None, prev_packed=packed[1] if t == 2 else None,
                              prev_norms=norms[1] if t == 2 else None)
        ref = model.quantize(v, t, want_hist=t == 1)
        assert compare_messages(orc, plan, packed[t % 2], ref) == (0, 0)
        if t == 1:
            assert np.array_equal(hist.cpu().numpy().view(np.uint32)[:, :1], ref["hist"])
