"""Router-on layer calls of 17 to 32 tokens (and of 9 to 16 with a large union) behind one another: one
kernel on clusters of four CTAs. Edges of its K quarters, row tiles and expert groups; references and
tolerances as in test_gpu_chain."""
import pytest
import torch

from paper_2507_08771_b200 import binding as B
from test_gpu_chain import check, make, reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,E,d_e,L", [
    (256, 8, 64, 32),          # one k block per quarter; fewer blocks of h than quarters
    (448, 20, 64, 17),         # quarters of one and two blocks
    (1984, 40, 512, 25),       # rows in several passes, all columns of a cluster but two
    (2048, 530, 64, 32),       # more groups of 16 experts than clusters, more than 4 mask words
    (512, 1024, 64, 20),       # the most experts
    (2048, 128, 128, 13),      # 9 to 16 tokens
    (1536, 80, 256, 16),
])
def test_edges(d, E, d_e, L):
    layer = B.Layer(d, E, d_e, L_max=32)
    g = torch.Generator(device="cuda").manual_seed(d + E)
    for bias in (-2.4, -1.0, 0.3, 9.0):         # a few, some, most, all of the experts
        dw = make(d, E, d_e, d + E, bias)
        x = torch.randn(L, d, device="cuda", generator=g).bfloat16()
        check(layer, dw, x, B.CALL_INDEPENDENT)
    assert layer.last_status() == 0


@pytest.mark.parametrize("L", [20, 32])
def test_a_token_that_is_not_finite_spoils_only_itself(L):
    d, E, d_e = 512, 24, 64
    layer, dw = B.Layer(d, E, d_e, L_max=L), make(d, E, d_e, 3, -0.5)
    x = torch.randn(L, d, device="cuda").bfloat16()
    _, ref = reference(dw.tensors, x)
    x[18, 5] = float("nan")
    x[3, 400] = float("inf")
    out = layer.forward(dw, x).out
    assert bool(out[18].isnan().all()) and not bool(out[3].isfinite().any())
    keep = [t for t in range(L) if t not in (3, 18)]
    assert (out[keep].double() - ref[keep]).abs().max() <= 2e-2 * ref.square().mean().sqrt()
    assert layer.last_status() == 0


@pytest.mark.parametrize("listed", [False, True])
@pytest.mark.parametrize("flags", [0, B.CALL_INDEPENDENT])
@pytest.mark.parametrize("d,E,d_e,L", [(2048, 64, 128, 17), (1024, 128, 128, 32), (1984, 100, 128, 16), (2048, 48, 256, 9)])
def test_scores_given(d, E, d_e, L, flags, listed):
    """Dependent calls with scores, and with scores and a list: x from the call before, some, all and none of
    the experts, a list with an id out of range, a token that is not finite."""
    layer, dw = B.Layer(d, E, d_e, L_max=32), make(d, E, d_e, 5, 0.0)
    t = dw.tensors
    g = torch.Generator(device="cuda").manual_seed(d + L)
    x = torch.randn(L, d, device="cuda", generator=g).bfloat16()
    for u, nan in ((E * 3 // 10, False), (E, False), (0, False), (E // 4, True)):
        pick = torch.randperm(E, device="cuda", generator=g)[:u].sort().values.int()
        s = torch.zeros(L, E, device="cuda")
        s[:, pick.long()] = (torch.rand(L, u, device="cuda", generator=g) < 0.5) * 0.5 + 0.25
        ids = torch.full((E,), -1, dtype=torch.int32, device="cuda")
        ids[:u] = pick
        xs = x.clone()
        if nan:
            xs[L - 1, 3] = float("nan")
            if listed:
                ids[u // 2] = E + 7                    # skipped and reported
                s[:, pick[u // 2].long()] = 0
        z = torch.einsum("ejd,td->tej", t["U"].double(), xs.double())
        ref = torch.einsum("tej,ecj->tc", s.double()[:, :, None] * z * torch.sigmoid(z), t["D"].double())
        base = torch.randn(L, d, device="cuda", generator=g)
        out, nxt = base.clone(), torch.empty(L, d, dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        if listed:
            n = torch.tensor([u], dtype=torch.int32, device="cuda")
            B.blockffn_expert_ffn(layer.h, dw.struct, xs, s, L, ids, n, out, nxt, flags | B.CALL_ACCUMULATE)
        else:
            r = layer.forward_scores(dw, xs, s, out=out, x_next=nxt, call_flags=flags | B.CALL_ACCUMULATE)
            assert int(r.n_union.item()) == u and torch.equal(r.union_ids[:u], pick)
        assert layer.last_status(clear=True) == (B.DEV_BAD_UNION_ID if listed and nan else 0)
        rows = L - 1 if nan else L
        rms = max(ref[:rows].square().mean().sqrt().item(), 1e-6)
        assert (out[:rows].double() - base[:rows].double() - ref[:rows]).abs().max().item() <= 2e-2 * rms + 1e-6
        assert torch.equal(nxt[:rows], out[:rows].bfloat16())
        if nan:
            assert bool(out[L - 1].isnan().all())
