"""The encoder's level searches at the values where they can go wrong: levels on the lower edges of the search table's bins (of
1/16 octave), one float beside them, so close to 1 that the finest bins are too coarse, and two in a bin; values on the levels
and one float beside them with both signs, both zeros, the smallest floats and 1, in whole blocks and in a partial one.
With the max norm and a largest value of 1 the normalised value is the value itself."""
import numpy as np
import pytest
import torch

from helpers import compare_messages, oracle_model, to_padded

pytestmark = pytest.mark.gpu


def _levels(kind, n):
    edges = np.array([(1 + m / 16) * 2.0 ** -o for o in range(1, 9) for m in range(16)], np.float32)
    rng = np.random.default_rng(n)
    if kind == "edges":
        inner = rng.choice(edges, min(n - 2, edges.size), replace=False)
    elif kind == "beside":
        inner = np.nextafter(rng.choice(edges, min(n - 2, edges.size), replace=False), np.float32(1.0 if n % 3 else 0.0))
    elif kind == "next_to_1":
        inner = 1.0 - 2.0 ** -24 * np.arange(1, n - 1)
    else:                                                    # two and more in some bins, down to the smallest gap allowed
        inner = np.concatenate([2.0 ** -rng.uniform(0.1, 90.0, n), 0.5 + 2.0 ** -20 * np.arange(n)])[: n - 2]
    inner = np.unique(np.float32(inner))
    while inner.size < n - 2:                                # (256 levels: more than there are edges)
        inner = np.unique(np.concatenate([inner, rng.uniform(0.001, 0.999, n - 2 - inner.size).astype(np.float32)]))
    return np.concatenate([[0.0], inner, [1.0]]).astype(np.float32)


@pytest.mark.parametrize("bits", [1, 2, 3, 4, 5, 6, 8])
@pytest.mark.parametrize("kind", ["edges", "beside", "next_to_1", "shared"])
@pytest.mark.parametrize("size", [3 * 1024, 300 * 1024 + 77])        # the kernel of small plans, and the general one
def test_values_on_and_beside_levels(orc, size, kind, bits):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    n, K = 1 << bits, 2
    levels = _levels(kind, n)
    plan = lqm.Plan([size], bits, 0, K, 77 + bits)
    plan.lq_set_levels(0, [float(x) for x in levels])
    one = np.float32(1.0)
    special = np.concatenate([levels, np.nextafter(levels, one), np.nextafter(levels, np.float32(0)), np.float32([1e-45, 1e-38, 2.0 ** -126, 2.0 ** -64]),
                              np.nextafter(np.float32(2.0) ** -np.arange(0, 30, dtype=np.float32), np.float32(0))]).astype(np.float32)
    special = special[(special >= 0) & (special <= 1)]
    rng = np.random.default_rng(bits)
    v = rng.choice(special, (K, size)) * rng.choice(np.float32([1.0, -1.0]), (K, size))      # (-0 among them)
    v[:, 0] = 1.0
    v[:, 2048:2304] = -0.0
    grads = to_padded(plan, v.astype(np.float32))
    model = oracle_model(orc, plan)
    packed, norms = [plan.empty_packed() for _ in range(2)], [plan.empty_norms() for _ in range(2)]
    for t in (1, 2):
        hist = plan.zero_hist()
        plan.lq_quantize_pack(grads, t, packed[t % 2], norms[t % 2], hist=hist if t == 1 else None, prev_packed=packed[1] if t == 2 else None,
                              prev_norms=norms[1] if t == 2 else None)
        ref = model.quantize(v.astype(np.float32), t, want_hist=t == 1)
        assert compare_messages(orc, plan, packed[t % 2], ref) == (0, 0)
        if t == 1:
            assert np.array_equal(hist.cpu().numpy().view(np.uint32)[:, :1], ref["hist"])
