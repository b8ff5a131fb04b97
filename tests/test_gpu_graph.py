"""Two iterations recorded into a CUDA graph and replayed (lq_quantize_pack with LQ_STEP_AUTO + qoda_step) against
the same iterations issued call by call with explicit step numbers: bit-identical messages and iterates."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _setup(lqm, scope, first=50000):
    plan = lqm.Plan([first, 300, 4097, 128], [4, 3, 2, 5], 2, 4, 77)
    plan.lq_set_norm_scope(scope)
    g = torch.Generator(device="cuda").manual_seed(3)
    X1 = torch.randn(plan.padded_elems, generator=g, device="cuda") * 0.1
    Y = torch.empty_like(X1); Xh = torch.empty_like(X1)
    plan.qoda_init(X1, Y, Xh)
    pk = [plan.empty_packed(), plan.empty_packed()]; nm = [plan.empty_norms(), plan.empty_norms()]
    return plan, X1, Y, Xh, pk, nm


@pytest.mark.parametrize("scope", ["layer", "bucket"])
def test_graph_replay_equals_call_by_call(scope):
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    T = 8
    g = torch.Generator(device="cuda").manual_seed(11)
    probe = lqm.Plan([50000, 300, 4097, 128], [4, 3, 2, 5], 2, 4, 77)
    grads = [torch.randn((4, probe.padded_elems), generator=g, device="cuda") * (0.9 ** t) for t in range(T)]
    for t in range(T):
        grads[t][1, 1000:9000] = 0.0

    # call by call, explicit step numbers
    plan, X1, Y, Xh, pk, nm = _setup(lqm, scope)
    for t in range(1, T + 1):
        c, p = t % 2, (t + 1) % 2
        plan.lq_quantize_pack(grads[t - 1], t, pk[c], nm[c], prev_packed=pk[p] if t > 1 else None,
                              prev_norms=nm[p] if t > 1 else None)
        plan.qoda_step(pk[c], nm[c], X1, Y, Xh)
    torch.cuda.synchronize()
    want = [x.cpu().numpy().copy() for x in (Y, Xh, pk[0], pk[1], nm[0], nm[1])]
    want_scalars = plan.qoda_get_scalars()

    # two iterations call by call, then iterations 3-4 recorded once and replayed three times
    plan, X1, Y, Xh, pk, nm = _setup(lqm, scope)
    gin = [torch.empty_like(grads[0]), torch.empty_like(grads[0])]
    for t in (1, 2):
        c, p = t % 2, (t + 1) % 2
        plan.lq_quantize_pack(grads[t - 1], lqm.STEP_AUTO, pk[c], nm[c], prev_packed=pk[p] if t > 1 else None,
                              prev_norms=nm[p] if t > 1 else None)
        plan.qoda_step(pk[c], nm[c], X1, Y, Xh)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for i, t in enumerate((3, 4)):
            c, p = t % 2, (t + 1) % 2
            plan.lq_quantize_pack(gin[i], lqm.STEP_AUTO, pk[c], nm[c], prev_packed=pk[p], prev_norms=nm[p])
            plan.qoda_step(pk[c], nm[c], X1, Y, Xh)
    for r in range(3):
        gin[0].copy_(grads[2 + 2 * r]); gin[1].copy_(grads[3 + 2 * r])
        graph.replay()
    torch.cuda.synchronize()
    got = [x.cpu().numpy() for x in (Y, Xh, pk[0], pk[1], nm[0], nm[1])]
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    assert plan.qoda_get_scalars() == want_scalars


def test_refused_launch_leaves_no_error_behind():
    """A call on the legacy default stream while a stream that waits for it is being recorded is refused by the runtime; the
    calls after it are not blamed for it."""
    import paper_2505_14371_b200 as lqm
    L = lqm.load_library()
    plan, X1, Y, Xh, pk, nm = _setup(lqm, "layer")
    grads = torch.zeros((4, plan.padded_elems), device="cuda")
    counts = torch.zeros((4, plan.num_layers, 256), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    with open("/proc/self/maps") as f:
        rt = C.CDLL(next(line.split()[-1] for line in f if "libcudart.so" in line))
    stream, graph = C.c_void_p(), C.c_void_p()
    assert rt.cudaStreamCreate(C.byref(stream)) == 0 and rt.cudaStreamBeginCapture(stream, 0) == 0
    code = L.lq_layer_norms(plan._h, grads.data_ptr(), nm[0].data_ptr(), None)
    rt.cudaStreamEndCapture(stream, C.byref(graph))
    rt.cudaGetLastError()
    rt.cudaStreamDestroy(stream)
    assert code != 0
    plan.lq_symbol_counts(pk[0], counts)
    torch.cuda.synchronize()


def test_recording_behind_memory_operations_and_other_streams():
    """The library's first kernel of a recording behind a memset, a copy and a join of two streams, and kernels of the caller
    between its calls: the replay equals the calls."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    outs = []
    for record in (False, True):
        plan, X1, Y, Xh, pk, nm = _setup(lqm, "layer")
        g = torch.Generator(device="cuda").manual_seed(3)
        src = torch.randn((4, plan.padded_elems), generator=g, device="cuda")
        grads, hist = torch.zeros_like(src), plan.zero_hist()
        probs = torch.zeros((plan.num_layers, 256), dtype=torch.float64, device="cuda")
        plan.lq_quantize_pack(src, 1, pk[1], nm[1], hist=hist)
        plan.lq_fit_levels(hist, nm[1], 4)
        plan.lq_quantize_pack(src, 2, pk[1], nm[1])
        plan.qoda_step(pk[1], nm[1], X1, Y, Xh)
        side = torch.cuda.Stream()
        torch.cuda.synchronize()

        def iteration():
            here = torch.cuda.current_stream()
            hist.zero_()
            side.wait_stream(here)
            with torch.cuda.stream(side):
                grads[:2].copy_(src[:2])
            grads[2:].copy_(src[2:])
            here.wait_stream(side)
            plan.lq_quantize_pack(grads, lqm.STEP_AUTO, pk[0], nm[0], hist=hist, prev_packed=pk[1], prev_norms=nm[1])
            side.wait_stream(here)
            plan.lq_level_probabilities(hist, nm[0], 4, probs)
            with torch.cuda.stream(side):
                src.mul_(0.5)
            here.wait_stream(side)
            plan.qoda_step(pk[0], nm[0], X1, Y, Xh)

        if record:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                iteration()
            graph.replay()
        else:
            iteration()
        torch.cuda.synchronize()
        outs.append([t.clone() for t in (pk[0], nm[0], Y, Xh, hist, probs, src)])
    for a, b in zip(*outs):
        assert torch.equal(a, b)


@pytest.mark.parametrize("scope, first", [("layer", 50000), ("layer", 2000000), ("bucket", 50000)])
def test_level_changes_are_seen_without_waiting(scope, first):
    """Levels refitted between two encodes, kernel behind kernel: what every kernel reads is what it would read had the
    device been waited for after each call."""
    import paper_2505_14371_b200 as lqm
    lqm.load_library()
    outs = []
    for wait in (False, True):
        plan, X1, Y, Xh, pk, nm = _setup(lqm, scope, first)
        g = torch.Generator(device="cuda").manual_seed(4)
        grads = [torch.randn((4, plan.padded_elems), generator=g, device="cuda") ** (1 + 2 * (i % 2)) for i in range(4)]
        hist, kept = [plan.zero_hist() for _ in range(12)], []
        probs = [torch.zeros((plan.num_layers, 256), dtype=torch.float64, device="cuda") for _ in range(12)]
        pause = torch.cuda.synchronize if wait else lambda: None
        torch.cuda.synchronize()
        for t in range(1, 13):
            c, p = t % 2, (t + 1) % 2
            plan.lq_quantize_pack(grads[t % 4], t, pk[c], nm[c], hist=hist[t - 1], prev_packed=pk[p] if t > 1 else None,
                                  prev_norms=nm[p] if t > 1 else None); pause()
            plan.lq_fit_levels(hist[t - 1], nm[c], 4); pause()
            plan.lq_level_probabilities(hist[t - 1], nm[c], 4, probs[t - 1], staged=True); pause()
            plan.qoda_step(pk[c], nm[c], X1, Y, Xh); pause()
            kept += [pk[c].clone(), Xh.clone()]
        outs.append(kept + hist + probs)
    for a, b in zip(*outs):
        assert torch.equal(a, b)
