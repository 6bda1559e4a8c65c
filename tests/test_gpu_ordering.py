"""What a call may read before it has waited for the work before it: nothing is synchronised between
the calls of a sequence, and every result has to be the one of the same sequence with a
synchronisation after every call, bit for bit (the same kernels do the same sums)."""
import pytest
import torch

from paper_2507_08771_b200 import binding as B
from test_gpu_chain import make

pytestmark = pytest.mark.gpu

D, E, D_E, N = 1024, 48, 64, 12


def sequence(kind, L, sync, E=E, D_E=D_E, last=None):
    layer, other = B.Layer(D, E, D_E, L_max=L), make(D, E, D_E, 99, -0.5)
    g = torch.Generator(device="cuda").manual_seed(L)
    dws = [make(D, E, D_E, s, -0.5) for s in range(2)]
    xs = [torch.randn(L, D, device="cuda", generator=g).bfloat16() for _ in range(N)]
    scores = [torch.zeros(L, E, device="cuda") for _ in range(N)]
    dummy = torch.zeros(L, E, device="cuda")
    fixed = torch.rand(L, E, device="cuda", generator=g) * (torch.rand(L, E, device="cuda", generator=g) < 0.3)
    ids = [torch.zeros(E, dtype=torch.int32, device="cuda") for _ in range(N)]
    n = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(N)]
    outs = [torch.zeros(L, D, device="cuda") for _ in range(2 * N)]
    step = torch.cuda.synchronize if sync else lambda: None
    torch.cuda.synchronize()
    for i in range(N):
        x, w = xs[i], dws[i % 2].struct
        if kind == "copied scores":        # what the layer call left, copied out, given to another layer
            B.blockffn_layer_forward(layer.h, w, x, L, outs[N + i])
            step()
            B.blockffn_read_routing(layer.h, L, scores[i], None, None, None, None)
            step()
        else:
            B.blockffn_router(layer.h, w, x, L, scores[i])
            step()
        if kind == "two routers":          # the scores of the router call before the last
            B.blockffn_router(layer.h, other.struct, x, L, dummy)
            step()
        if kind == "two promised calls":   # the scores of the router call before a call that may start early itself
            B.blockffn_layer_forward_scores(layer.h, other.struct, x, fixed, L, outs[N + i], call_flags=B.CALL_INDEPENDENT)
            step()
        n0 = layer.launch_count()
        if kind == "union list":
            B.blockffn_chunk_union(layer.h, scores[i], L, None, ids[i], n[i])
            step()
            B.blockffn_expert_ffn(layer.h, w, x, scores[i], L, ids[i], n[i], outs[i], call_flags=B.CALL_INDEPENDENT)
        else:
            B.blockffn_layer_forward_scores(layer.h, w, x, scores[i], L, outs[i], call_flags=B.CALL_INDEPENDENT)
        assert last is None or layer.launch_count() - n0 == last
        step()
    torch.cuda.synchronize()
    assert layer.last_status() == 0
    return outs


@pytest.mark.parametrize("kind", ["copied scores", "two routers", "union list"])
@pytest.mark.parametrize("L", [1, 8, 32])
def test_promised_inputs_from_the_call_before(kind, L):
    want, got = sequence(kind, L, True), sequence(kind, L, False)
    assert all(bool(w.any()) for w in want[:N])
    for i, (w, o) in enumerate(zip(want, got)):
        assert torch.equal(w, o), i


@pytest.mark.parametrize("L", [1, 8, 32])
def test_scores_of_a_router_call_before_a_promised_call(L):
    test_promised_inputs_from_the_call_before("two promised calls", L)


@pytest.mark.parametrize("kind", ["copied scores", "two routers", "two promised calls"])
@pytest.mark.parametrize("L", [1, 8, 13, 16])
def test_promised_scores_of_the_dependent_chain_kernel(kind, L):
    """The same where a scores-given call is one kernel for every length, which reads scores, U and D before it waits."""
    want, got = (sequence(kind, L, sync, 64, 128, 1) for sync in (True, False))
    assert all(bool(w.any()) for w in want[:N])
    for i, (w, o) in enumerate(zip(want, got)):
        assert torch.equal(w, o), i
