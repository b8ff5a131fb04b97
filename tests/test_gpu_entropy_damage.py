"""The entropy decoder against a walk of the definition, run by run: whole streams and damaged ones (what a damaged run decodes
to is defined: the walk goes on over the block's remaining words, zeros past its end, and a pattern without a word counts as
one bit of symbol 0), complete, incomplete and long codes on both sides of the two-coordinate tables' width, partial blocks,
and buffers that start on no 16-byte boundary."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
SIZES = [2 * 1024 + 300, 1024, 5, 3 * 1024 + 1020]


def _codes(lqm, kind, n):
    if kind == "short":
        return lqm.lq_code_build([0.6 ** j for j in range(n)])
    if kind == "long":                                       # the frequent small levels have the longest words
        return lqm.lq_code_build([1.4 ** min(j, 40) for j in range(n)])
    short = lqm.lq_code_build([0.9 ** j for j in range(n)])   # Kraft sum below 1: some patterns are no word
    return [min(x + 1, 12) for x in short]


def _words(lengths):
    """(length, word read first bit first) -> level"""
    table, code, prev = {}, 0, 0
    for l in range(1, 13):
        for j, x in enumerate(lengths):
            if x == l:
                code <<= l - prev
                table[(l, code)] = j
                code, prev = code + 1, l
    return table


def _walk(plan, table, S, O, R):
    """The message of the definition, and whether any run (R: the run offsets) or block (None) is broken."""
    out, broken, g = np.zeros((plan.num_workers, plan.packed_words), np.uint32), False, 0
    for m, (d, b) in enumerate(zip(plan.layer_sizes, plan.bits)):
        C = b + 1
        for blk in range((d + 1023) // 1024):
            for k in range(plan.num_workers):
                first, last = int(O[k, g]), min(int(O[k, g + 1]), S.shape[1])
                bits = np.unpackbits(S[k, first:last].view(np.uint8), bitorder="little")
                nbits = bits.size
                bits = np.concatenate([bits, np.zeros(1024 * 13 + 64, np.uint8)]).tolist()
                pos = at = 0
                for lane in range(32):
                    if R is not None and lane % 4 == 0:
                        pos = int(R[k, g, lane // 4])
                    string = 0
                    for p in range(32):
                        if blk * 1024 + 128 * (p // 4) + 4 * lane + p % 4 >= d:
                            continue
                        at, word, sym, l = pos, 0, None, 0
                        while l < 12 and sym is None:
                            word = 2 * word + bits[pos + l]
                            l += 1
                            sym = table.get((l, word))
                        if sym is None:
                            broken, pos = True, pos + 1
                            continue
                        pos += l
                        if sym:
                            sym = 2 * sym + bits[pos]
                            pos += 1
                        string |= sym << (p * C)
                    for i in range(C):
                        out[k, plan.word_offsets[m] + (blk * C + i) * 32 + lane] = (string >> (32 * i)) & 0xffffffff
                    if R is not None and lane % 4 == 3:
                        broken |= pos != int(R[k, g, lane // 4 + 1]) if lane < 31 else pos > nbits
                if R is None:
                    broken |= at // 32 > nbits // 32          # the last coordinate starts past the word behind the end
            g += 1
    return out, broken


@pytest.mark.parametrize("bits", [1, 2, 4, 5, 8])
@pytest.mark.parametrize("kind", ["short", "long", "incomplete"])
def test_damaged_streams_decode_as_defined(bits, kind):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    K, shift = 2, 1 if bits in (2, 8) else 0
    plan = lqm.Plan(SIZES, bits, 2, K, 17 + bits)
    gen = torch.Generator(device="cuda").manual_seed(bits)
    grads = torch.randn((K, plan.padded_elems), generator=gen, device="cuda") ** 3
    grads[:, 1024:1500] = 0.0
    packed, norms = plan.empty_packed(), plan.empty_norms()
    plan.lq_quantize_pack(grads, 1, packed, norms)
    lengths = _codes(lqm, kind, 1 << bits)
    for m in range(plan.num_layers):
        plan.lq_code_set(m, lengths)
    table = _words(lengths)

    def buffer(shape):                                       # `shift` words off a 16-byte boundary
        flat = torch.full((int(np.prod(shape)) + 4,), -1, dtype=torch.int32, device="cuda")
        return flat[shift: shift + int(np.prod(shape))].view(shape)

    stream, back = buffer((K, plan.lq_plan_blocks() * 416)), buffer((K, plan.packed_words))
    offs = torch.zeros((K, plan.lq_plan_blocks() + 1), dtype=torch.int32, device="cuda")
    runs = plan.empty_run_offsets()
    plan.lq_entropy_encode(packed, stream, offs, runs)
    O, R = offs.cpu().numpy().astype(np.int64), runs.cpu().numpy().view(np.uint16)
    rng = np.random.default_rng(bits)
    whole = stream.cpu().numpy().view(np.uint32).copy()
    for flips in (0, 3, 40):
        S = whole.copy()
        for k in range(K):
            at = rng.integers(0, int(O[k, -1]), flips)
            np.bitwise_xor.at(S[k], at, np.uint32(1) << rng.integers(0, 32, flips).astype(np.uint32))
        stream.copy_(torch.from_numpy(S.view(np.int32)))
        for side, data in ((runs, R), (None, None)):
            want, broken = _walk(plan, table, S, O, data)
            assert flips or not broken
            for _ in range(2):
                back.fill_(-1)
                plan.lq_entropy_decode(stream, offs, back, side)
                assert (plan.lq_entropy_status() != 0) == broken
                assert np.array_equal(back.cpu().numpy().view(np.uint32), want)
