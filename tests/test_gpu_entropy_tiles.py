"""The entropy encoder where its tiles meet: tiles of 8 to 128 blocks, of one block a warp and many; plans of fewer and of more tiles than a tile looks back over at a time, so that a
tile's place in the stream comes from one or several looks; blocks with rows of zeros under codes whose word for level 0 is
one zero bit, several, or not zeros at all.  Every block of every worker against the oracle's encoder, and the way back."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _code(lqm, kind, n):
    if kind == "zero_long":                                  # level 0 has the longest word, all ones
        return lqm.lq_code_build([0.001] + [0.5 ** min(j, 9) for j in range(1, n)])
    return [n.bit_length() - 1] * n if kind == "flat" else lqm.lq_code_build([0.9] + [0.1 / n] * (n - 1))


@pytest.mark.parametrize("bits, kind", [(1, "fitted"), (2, "zero_long"), (3, "flat"), (4, "fitted"), (5, "zero_long"), (6, "fitted"), (7, "zero_long"), (8, "flat")])
@pytest.mark.parametrize("layers", [1, 32, 33, 70])
def test_streams_of_many_tiles(orc, layers, bits, kind):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    K, rng = 3, np.random.default_rng(layers + bits)
    sizes = [int(x) for x in rng.choice([1, 1023, 1024, 1025, 2500, 9 * 1024 + 7], layers)]
    plan = lqm.Plan(sizes, bits, 2, K, 5 + bits)
    gen = torch.Generator(device="cuda").manual_seed(bits)
    grads = torch.randn((K, plan.padded_elems), generator=gen, device="cuda")
    grads.view(K, -1, 32)[:, ::3] = 0.0                      # a third of the rows' quarters
    grads[:, 2048:4096] = 0.0
    packed, norms = plan.empty_packed(), plan.empty_norms()
    plan.lq_quantize_pack(grads, 1, packed, norms)
    lengths = _code(lqm, kind, 1 << bits)
    for m in range(layers):
        plan.lq_code_set(m, lengths)
    stream = torch.full((K, plan.lq_plan_blocks() * 416), -1, dtype=torch.int32, device="cuda")
    offs = torch.zeros((K, plan.lq_plan_blocks() + 1), dtype=torch.int32, device="cuda")
    runs = plan.empty_run_offsets()
    for _ in range(2):                                       # the second encode finds the first one's scratch
        plan.lq_entropy_encode(packed, stream, offs, runs)
    pk, S, O = packed.cpu().numpy().view(np.uint32), stream.cpu().numpy().view(np.uint32), offs.cpu().numpy().astype(np.int64)
    l = np.uint8(lengths)
    c = orc.canonical_codes(l)
    for k in range(K):
        pos = g = 0
        for m, d in enumerate(sizes):
            at = plan.word_offsets[m]
            idx, sg = orc.unpack_layer(pk[k, at: at + orc.packed_words(d, bits)], d, bits)
            for lo in range(0, d, 1024):
                words, _ = orc.entropy_encode_block(idx[lo: lo + 1024], sg[lo: lo + 1024], l, c)
                assert O[k, g] == pos and np.array_equal(S[k, pos: pos + words.size], words), (k, m, lo)
                pos += words.size
                g += 1
        assert O[k, g] == pos and np.all(S[k, pos:] == 0xffffffff)
    back, again = torch.full_like(packed, -1), torch.full_like(stream, -1)
    plan.lq_entropy_decode(stream, offs, back, runs)
    assert plan.lq_entropy_status() == 0
    plan.lq_entropy_encode(back, again, offs, runs)
    assert torch.equal(again, stream)


def test_overlapping_encodes_stay_in_their_buffers():
    """Two encodes of one plan on two streams, which the caller should have ordered: each clears the counter from which the
    other's CTAs take their tiles, so that more numbers are drawn than there are tiles.  What comes out is undefined; nothing
    outside the buffers is written, and an encode after them is right again."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    K = 8
    plan = lqm.Plan([8 * 1024 - 5] * 30, 4, 2, K, 3)         # 240 CTAs: those of both calls run at once
    grads = torch.randn((K, plan.padded_elems), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    packed, norms = plan.empty_packed(), plan.empty_norms()
    plan.lq_quantize_pack(grads, 1, packed, norms)
    cap, blocks = plan.packed_words, plan.lq_plan_blocks()

    def buffers():                                           # a row more than the call is given, as a guard
        return torch.full((K + 1, cap), -1, dtype=torch.int32, device="cuda"), torch.full((K + 1, blocks + 1), -1, dtype=torch.int32, device="cuda")
    want, mine, theirs = buffers(), buffers(), buffers()
    plan.lq_entropy_encode(packed, want[0][:K], want[1][:K])
    torch.cuda.synchronize()
    plan.lq_entropy_wait(1 << 12)                            # (a tile whose word was cleared waits for nothing: not for long)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(50):
        for s, (words, offs) in zip(streams, (mine, theirs)):
            with torch.cuda.stream(s):
                plan.lq_entropy_encode(packed, words[:K], offs[:K])
    torch.cuda.synchronize()
    for words, offs in (mine, theirs):
        assert bool((words[K] == -1).all()) and bool((offs[K] == -1).all())
    plan.lq_entropy_wait()
    plan.lq_entropy_status()
    plan.lq_entropy_encode(packed, mine[0][:K], mine[1][:K])
    assert plan.lq_entropy_status() == 0
    assert torch.equal(mine[1], want[1])
    for k in range(K):
        n = int(want[1][k, blocks])
        assert torch.equal(mine[0][k, :n], want[0][k, :n])


@pytest.mark.parametrize("sizes", [[9 * 1024 + 7] * 40, [1] * 3, [70 * 1024]])
def test_tiles_that_give_up_say_so(sizes):
    """No tile looks for the words before it: all but each worker's first one give up.  They leave offsets that a decode reports
    as broken, and words that are not theirs as they were; the status names the encode, and the next encode is whole again."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    K = 3
    plan = lqm.Plan(sizes, 4, 2, K, 3)
    grads = torch.randn((K, plan.padded_elems), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    packed, norms = plan.empty_packed(), plan.empty_norms()
    plan.lq_quantize_pack(grads, 1, packed, norms)
    blocks = plan.lq_plan_blocks()

    def encoded():
        words, offs, runs = torch.full_like(packed, -1), torch.zeros((K, blocks + 1), dtype=torch.int32, device="cuda"), plan.empty_run_offsets()
        plan.lq_entropy_encode(packed, words, offs, runs)
        return words, offs, runs
    whole = encoded()
    assert plan.lq_entropy_status() == 0
    plan.lq_entropy_wait(0)
    words, offs, runs = encoded()
    assert plan.lq_entropy_status() == lqm.CODE_GAVE_UP and plan.lq_entropy_status() == 0
    first = min(8, -(-sizes[0] // 1024))                     # blocks of the first tile
    n = whole[1][:, first]                                   # and its words
    assert torch.equal(offs[:, :first], whole[1][:, :first]) and bool((offs[:, first:] == -1).all())
    for k in range(K):
        assert torch.equal(words[k, : n[k]], whole[0][k, : n[k]]) and bool((words[k, n[k]:] == -1).all())
    for side in (runs, None):
        plan.lq_entropy_decode(words, offs, torch.empty_like(packed), side)
        assert plan.lq_entropy_status() == lqm.CODE_BROKEN
    plan.lq_entropy_wait()
    again = encoded()
    assert plan.lq_entropy_status() == 0 and all(torch.equal(a, b) for a, b in zip(again, whole))
    with pytest.raises(lqm.LqError):
        plan.lq_entropy_wait(-1)


@pytest.mark.parametrize("by_width, layers, K, widths, runs", [
    (True, 131, 8, [1, 2, 3, 4, 5, 6, 7, 8], 1), (False, 130, 8, [1, 2, 3, 4, 5, 6, 7, 8], 1), (True, 300, 12, [2, 3, 4, 8], 3),
    (False, 300, 12, [2, 3, 4, 8], 20), (False, 360, 12, [7, 6], 1)])
def test_streams_of_plans_of_several_widths(orc, by_width, layers, K, widths, runs):
    """Plans on both sides of the rule's lines; layers of one block and a few, each with a code of its own."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    rng = np.random.default_rng(layers)
    sizes = [int(x) for x in rng.choice([1, 31, 200, 1023], layers)]
    sizes[3] = 19 * 1024 + 5
    bits = [widths[m // runs % len(widths)] for m in range(layers)]
    plan = lqm.Plan(sizes, bits, 2, K, 11)
    gen = torch.Generator(device="cuda").manual_seed(layers)
    grads = torch.randn((K, plan.padded_elems), generator=gen, device="cuda") ** 3
    grads.view(K, -1, 32)[:, ::3] = 0.0
    grads[:, plan.elem_offsets[3] + 2048: plan.elem_offsets[3] + 6144] = 0.0
    packed, norms = plan.empty_packed(), plan.empty_norms()
    plan.lq_quantize_pack(grads, 1, packed, norms)
    codes = []
    for m, b in enumerate(bits):
        codes.append(lqm.lq_code_build([0.3 + 0.7 * (m % 2)] + [0.5 ** min(j, 3 + m % 8) for j in range(1, 1 << b)]))
        plan.lq_code_set(m, codes[m])
    stream = torch.full((K, plan.lq_plan_blocks() * 416), -1, dtype=torch.int32, device="cuda")
    offs, runs_at = torch.zeros((K, plan.lq_plan_blocks() + 1), dtype=torch.int32, device="cuda"), plan.empty_run_offsets()
    plan.lq_entropy_wait(0)                                  # only tiles in stream order wait for others
    plan.lq_entropy_encode(packed, stream, offs, runs_at)
    assert plan.lq_entropy_status() == (0 if by_width else lqm.CODE_GAVE_UP)
    plan.lq_entropy_wait()
    stream.fill_(-1)
    for _ in range(2):
        plan.lq_entropy_encode(packed, stream, offs, runs_at)
    pk, S, O = packed.cpu().numpy().view(np.uint32), stream.cpu().numpy().view(np.uint32), offs.cpu().numpy().astype(np.int64)
    for k in range(K):
        pos = g = 0
        for m, d in enumerate(sizes):
            at, l = plan.word_offsets[m], np.uint8(codes[m])
            idx, sg = orc.unpack_layer(pk[k, at: at + orc.packed_words(d, bits[m])], d, bits[m])
            c = orc.canonical_codes(l)
            for lo in range(0, d, 1024):
                words, _ = orc.entropy_encode_block(idx[lo: lo + 1024], sg[lo: lo + 1024], l, c)
                assert O[k, g] == pos and np.array_equal(S[k, pos: pos + words.size], words), (k, m, lo)
                pos += words.size
                g += 1
        assert O[k, g] == pos and np.all(S[k, pos:] == 0xffffffff)
    back, again = torch.full_like(packed, -1), torch.full_like(stream, -1)
    plan.lq_entropy_decode(stream, offs, back, runs_at)
    assert plan.lq_entropy_status() == 0
    plan.lq_entropy_encode(back, again, offs, runs_at)
    assert torch.equal(again, stream)


def _sampled_blocks_match(orc, plan, packed, stream, offs, runs, codes, rng, count):
    """`count` random blocks of every worker, and the first and last of every layer, against the oracle's encoder; all sizes of
    blocks add up, in the order of the stream."""
    S, O, R = stream.cpu().numpy().view(np.uint32), offs.cpu().numpy().astype(np.int64), runs.cpu().numpy().view(np.uint16)
    blocks = [(m, i) for m, d in enumerate(plan.layer_sizes) for i in range(-(-d // 1024))]
    ends = [g for g, (m, i) in enumerate(blocks) if i == 0 or g + 1 == len(blocks) or blocks[g + 1][0] != m]
    assert np.all(O[:, 0] == 0) and np.all(np.diff(O, axis=1) >= 0)
    for k in range(plan.num_workers):
        pk = packed[k].cpu().numpy().view(np.uint32)
        for g in {*ends, *(int(x) for x in rng.integers(0, len(blocks), count))}:
            m, i = blocks[g]
            b, d = plan.bits[m], min(1024, plan.layer_sizes[m] - 1024 * i)
            at, l = plan.word_offsets[m] + i * 32 * (b + 1), np.uint8(codes[m])
            idx, sg = orc.unpack_layer(pk[at: at + 32 * (b + 1)], d, b)
            words, _ = orc.entropy_encode_block(idx, sg, l, orc.canonical_codes(l))
            assert O[k, g + 1] - O[k, g] == words.size and np.array_equal(S[k, O[k, g]: O[k, g + 1]], words), (k, m, i)
            # a lane's 32 coordinates are one after the other in the stream: where every fourth lane starts
            size = np.where(idx > 0, l[idx].astype(np.int64) + 1, int(l[0]))
            c = np.arange(d)
            lane = (c // 4) % 32
            per_lane = np.bincount(lane, weights=size, minlength=32).astype(np.int64)
            assert np.array_equal(R[k, g], np.concatenate([[0], np.cumsum(per_lane)])[:32:4])
        assert np.all(S[k, O[k, -1]:] == 0xffffffff)


@pytest.mark.parametrize("sizes, bits, K, tile, kind", [
    ([620 * 1024 + 5, 33], 4, 8, 8, "fitted"), ([1300 * 1024 + 1], 6, 8, 16, "zero_long"), ([140 * 1024 - 1] * 40, 7, 2, 16, "fitted"),
    ([4352 * 1024 + 300, 5000], 2, 8, 32, "fitted"), ([3000 * 1024 - 100], 8, 8, 32, "fitted"), ([33000 * 1024 + 700], 3, 8, 64, "flat"),
    ([33000 * 1024 - 100], 4, 16, 128, "fitted")])
def test_tiles_of_many_blocks(orc, sizes, bits, K, tile, kind):
    """Tiles of every length that plans have, more of them than CTAs run at once, with a partial one at the end: each warp takes
    block after block, whole blocks of zeros between others of the same warp (8 blocks on) and two in a row among them."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    plan = lqm.Plan(sizes, bits, 2, K, 5 + bits)
    gen = torch.Generator(device="cuda").manual_seed(bits)
    grads = torch.empty((K, plan.padded_elems), device="cuda")
    for k in range(K):
        grads[k].normal_(generator=gen).pow_(3)
    grads.view(K, -1, 32)[:, ::5] = 0.0
    whole = grads[:, : plan.padded_elems // 8192 * 8192].view(K, -1, 8, 1024)           # [.., warp, coordinate]
    whole[:, 1::4, 2:5] = 0.0                                # a warp's every fourth block
    whole[:, 2::4, 3:6] = 0.0                                # and the next one: two in a row
    packed, norms = plan.empty_packed(), plan.empty_norms()
    plan.lq_quantize_pack(grads, 1, packed, norms)
    del grads, whole
    lengths = _code(lqm, kind, 1 << bits)
    for m in range(len(sizes)):
        plan.lq_code_set(m, lengths)
    blocks = plan.lq_plan_blocks()
    length = 128                                             # the length of the plan's tiles
    while length > 32 and blocks // length * K < 4096:
        length //= 2
    while length > 8 and blocks // length * K < 592:
        length //= 2
    assert length == tile
    words = max(lengths) + 1
    stream = torch.full((K, blocks * 32 * words), -1, dtype=torch.int32, device="cuda")
    offs, runs = torch.zeros((K, blocks + 1), dtype=torch.int32, device="cuda"), plan.empty_run_offsets()
    for _ in range(2):
        plan.lq_entropy_encode(packed, stream, offs, runs)
    assert plan.lq_entropy_status() == 0
    _sampled_blocks_match(orc, plan, packed, stream, offs, runs, [lengths] * len(sizes), np.random.default_rng(bits), 60)
    back, again = torch.full_like(packed, -1), torch.full_like(stream, -1)
    plan.lq_entropy_decode(stream, offs, back, runs)
    assert plan.lq_entropy_status() == 0
    plan.lq_entropy_encode(back, again, offs, runs)
    assert torch.equal(again, stream)
