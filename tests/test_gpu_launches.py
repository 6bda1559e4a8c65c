"""Which calls run as one kernel, whose CTAs all have to be resident at once, and how those get there."""
import pytest
import torch

from paper_2507_08771_b200 import binding as B
from test_gpu_chain import make, reference

pytestmark = pytest.mark.gpu


def launches(layer, call):
    n = layer.launch_count()
    call()
    torch.cuda.synchronize()
    assert layer.last_status() == 0
    return layer.launch_count() - n


@pytest.mark.parametrize("L", [1, 8, 9, 16, 17, 32])
def test_calls_with_and_without_a_promise(L):
    """Scores or a list given: a chunk of more than 8 tokens is one kernel, with a promise or (launched
    when all its CTAs fit) without; with CFG_TWO_KERNELS kernels that follow one another."""
    d, E, d_e = 512, 24, 64
    dw = make(d, E, d_e, 1, 0.0)
    x, scores = torch.randn(L, d, device="cuda").bfloat16(), torch.rand(L, E, device="cuda")
    ids, n = torch.arange(E, device="cuda", dtype=torch.int32), torch.full((1,), E, device="cuda", dtype=torch.int32)
    z = torch.einsum("ejd,td->tej", dw.tensors["U"].double(), x.double())
    ref = torch.einsum("tej,ecj->tc", scores.double()[:, :, None] * z * torch.sigmoid(z), dw.tensors["D"].double())
    for cfg in (0, B.CFG_TWO_KERNELS):
        layer = B.Layer(d, E, d_e, L_max=L, flags=cfg)
        for flags in (0, B.CALL_INDEPENDENT):
            for call in (lambda out: B.blockffn_layer_forward_scores(layer.h, dw.struct, x, scores, L, out, call_flags=flags),
                         lambda out: B.blockffn_expert_ffn(layer.h, dw.struct, x, scores, L, ids, n, out, call_flags=flags)):
                out = torch.zeros(L, d, device="cuda")
                torch.cuda.synchronize()
                assert launches(layer, lambda: call(out)) == (1 if L > 8 and not cfg else 2)
                assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()


@pytest.mark.parametrize("L", [16, 32])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("d,E,d_e,n", [(1024, 32, 64, 40), (2048, 128, 128, 20)])     # the one-kernel form; clusters
def test_calls_without_a_promise_beside_other_streams(d, E, d_e, n, L, graph):
    """Two handles' calls on streams of different priorities beside a stream of large products: every
    call gets its places on the SMs as a whole, none gives up waiting, and the results are those of
    the same calls alone."""
    dws = [make(d, E, d_e, s, 0.0) for s in range(2)]
    layers = [B.Layer(d, E, d_e, L_max=L) for _ in range(2)]
    x = [torch.randn(L, d, device="cuda").bfloat16() for _ in range(2)]
    scores = [torch.rand(L, E, device="cuda") for _ in range(2)]
    outs = [[torch.zeros(L, d, device="cuda") for _ in range(n)] for _ in range(2)]
    a = torch.randn(2048, 2048, device="cuda").bfloat16()

    def calls(k):
        for i in range(n):
            B.blockffn_layer_forward_scores(layers[k].h, dws[k].struct, x[k], scores[k], L, outs[k][i])

    want = []
    for k in range(2):
        calls(k)
        torch.cuda.synchronize()
        want.append(outs[k][0].clone())
        assert all(torch.equal(o, want[k]) for o in outs[k])
        for o in outs[k]:
            o.zero_()
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1)]
    graphs = []
    for k, st in enumerate(streams):
        if graph:
            graphs.append(torch.cuda.CUDAGraph())
            with torch.cuda.graph(graphs[k], stream=st):
                calls(k)
    busy = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(busy):
        for _ in range(30):
            b = a @ a
    for k, st in enumerate(streams):
        with torch.cuda.stream(st):
            graphs[k].replay() if graph else calls(k)
    torch.cuda.synchronize()
    for k in range(2):
        assert layers[k].last_status() == 0
        assert all(torch.equal(o, want[k]) for o in outs[k])
    del b


@pytest.mark.parametrize("d,E,L,want", [
    # clusters (too many experts for the pools of the chain kernel)
    (2048, 544, 32, 1), (1024, 992, 32, 1), (2048, 712, 24, 1), (2048, 952, 17, 1),
    (512, 1024, 16, 1), (512, 1024, 32, 1),          # the chain kernel, clusters
])
@pytest.mark.parametrize("flags", [0, B.CALL_INDEPENDENT])
def test_dependent_router_on_calls_of_many_experts(d, E, L, want, flags):
    """One kernel with the router inside, whatever room the score matrix of a chunk takes."""
    dw, layer = make(d, E, 64, 2, -1.2), B.Layer(d, E, 64, L_max=L)
    g = torch.Generator(device="cuda").manual_seed(L)
    h = torch.randn(L, d, device="cuda", generator=g)
    x = [h.bfloat16(), torch.empty(L, d, dtype=torch.bfloat16, device="cuda")]
    torch.cuda.synchronize()

    before = h.double()
    n = layer.launch_count()
    B.blockffn_layer_forward(layer.h, dw.struct, x[0], L, h, x[1], None, flags | B.CALL_ACCUMULATE)
    torch.cuda.synchronize()
    assert layer.launch_count() - n == want and layer.last_status() == 0
    _, ref = reference(dw.tensors, x[0])
    assert (h.double() - before - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()
    assert torch.equal(x[1], h.bfloat16())

    results = []
    start = h.clone()
    for sync in (True, False):   # three layers one after the other, with and without a pause
        h.copy_(start)
        x[0].copy_(start)
        torch.cuda.synchronize()
        for i in range(3):
            B.blockffn_layer_forward(layer.h, dw.struct, x[i % 2], L, h, x[(i + 1) % 2], None, flags | B.CALL_ACCUMULATE)
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        results.append(h.clone())
    assert torch.equal(*results) and layer.last_status() == 0
