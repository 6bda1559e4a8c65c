"""Dependent calls of 17 to 32 tokens, and of 9 to 16 with a large union, as one kernel on clusters of four CTAs:
router on, scores given, a list given. Edges of its K quarters, row tiles and expert groups, calls one behind
the other, and calls that give up; references and tolerances as in test_gpu_chain. (That a shape takes this kernel
shows in test_one_cta_that_gives_up: in the others, all CTAs give up or none.)"""
import pytest
import torch

from paper_2507_08771_b200 import binding as B
from test_gpu_chain import chain, check, layers, make, reference

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


@pytest.mark.parametrize("d,E,d_e,L", [(2048, 160, 64, 16), (2048, 64, 64, 32), (256, 8, 64, 17)])
def test_one_expert_router_on(d, E, d_e, L):
    """64 rows of U in fours: half of the clusters have none, but columns of D like the others."""
    layer, dws = B.Layer(d, E, d_e, L_max=L), [make(d, E, d_e, s, -12.0) for s in range(4)]
    g = torch.Generator(device="cuda").manual_seed(E)
    for i, dw in enumerate(dws):
        dw.tensors["bias"][(5 * i) % E] = 12.0
    x = torch.randn(L, d, device="cuda", generator=g).bfloat16()
    for dw in dws:
        check(layer, dw, x, B.CALL_INDEPENDENT)
    out = torch.zeros(L, d, device="cuda")
    torch.cuda.synchronize()
    for i in range(40):
        B.blockffn_layer_forward(layer.h, dws[i % 4].struct, x, L, out, None, None, B.CALL_INDEPENDENT | B.CALL_ACCUMULATE)
    ref = 10 * sum(reference(dw.tensors, x)[1] for dw in dws)
    assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt() and layer.last_status() == 0


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


@pytest.mark.parametrize("flags", [0, B.CALL_INDEPENDENT])
@pytest.mark.parametrize("lengths", [[12], [16], [32], [16, 32, 9, 17, 8, 13]], ids=str)
def test_router_on_one_behind_the_other(lengths, flags):
    """As test_calls_one_behind_the_other of test_gpu_chain, with unions large enough for chunks of 9 to 16
    tokens, whose CTAs are on the SMs two calls at a time."""
    d, E, d_e = 2048, 128, 128
    dws, layer = layers(E, d, d_e), B.Layer(d, E, d_e, L_max=32)
    lengths = (lengths * 20)[:20]
    start = torch.randn(32, d, device="cuda")
    h, x = start.clone(), torch.zeros(2, 32, d, dtype=torch.bfloat16, device="cuda")

    def run(each=lambda i: None):
        h.copy_(start)
        x.copy_(start.expand(2, 32, d))
        chain(layer, dws, lengths, h, x, flags, each)
        return h.clone(), x.clone()
    seen = {"h": start.double(), "x": start.bfloat16()}

    def compare(i):
        L = lengths[i]
        torch.cuda.synchronize()
        _, ref = reference(dws[i % len(dws)].tensors, seen["x"][:L])
        rms = max(ref.square().mean().sqrt().item(), 1e-6)
        assert (h[:L].double() - seen["h"][:L] - ref).abs().max().item() <= 2e-2 * rms + 1e-5
        seen["h"], seen["x"] = h.double(), x[(i + 1) % 2].clone()
    want = run(compare)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        h.copy_(start)
        x.copy_(start.expand(2, 32, d))
        chain(layer, dws, lengths, h, x, flags)
    for _ in range(3):
        graph.replay()
        got = run()
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(h, want[0]) and torch.equal(x, want[1]) and layer.last_status() == 0


@pytest.mark.parametrize("listed", [False, True])
@pytest.mark.parametrize("d,E,d_e,L", [(2048, 128, 128, 12), (2048, 64, 256, 16), (2048, 64, 128, 20), (2048, 128, 128, 32)])
def test_scores_given_one_behind_the_other(d, E, d_e, L, listed):
    """Nothing but such calls on the stream, every x from the call before and U asked for under it: call
    numbers, the two buffers of h, tensor memory of two calls on an SM (up to 16 tokens). The same bits as with
    a pause behind every call, where every layer is compared with float64; eagerly and from a graph."""
    n, u = 12, E * 3 // 10
    g = torch.Generator(device="cuda").manual_seed(L)
    dws = [make(d, E, d_e, s, 0.0) for s in range(3)]
    layer = B.Layer(d, E, d_e, L_max=32)
    scores, ids = [], []
    for i in range(n):
        k = (u, E, 1, u)[i % 4]                        # (most experts, one: rows in several passes, few rows)
        pick = torch.randperm(E, device="cuda", generator=g)[:k].sort().values.int()
        s = torch.zeros(L, E, device="cuda")
        s[:, pick.long()] = (torch.rand(L, k, device="cuda", generator=g) < 0.5) * (0.5 / k) + 0.1 / k
        scores.append(s)
        ids.append(torch.cat([pick, torch.full((E - k,), -1, dtype=torch.int32, device="cuda")]))
    counts = [torch.tensor([(u, E, 1, u)[i % 4]], dtype=torch.int32, device="cuda") for i in range(n)]
    start = torch.randn(L, d, device="cuda", generator=g)
    h, x = start.clone(), torch.zeros(2, L, d, dtype=torch.bfloat16, device="cuda")

    def chain(each=lambda i: None):
        h.copy_(start)
        x.copy_(start.expand(2, L, d))
        for i in range(n):
            w, xi, xn = dws[i % 3].struct, x[i % 2], x[(i + 1) % 2]
            if listed:
                B.blockffn_expert_ffn(layer.h, w, xi, scores[i], L, ids[i], counts[i], h, xn,
                                      B.CALL_ACCUMULATE | B.CALL_INDEPENDENT)
            else:
                B.blockffn_layer_forward_scores(layer.h, w, xi, scores[i], L, h, xn, None,
                                                B.CALL_ACCUMULATE | B.CALL_INDEPENDENT)
            each(i)
    seen = {"h": start.double(), "x": start.bfloat16()}

    def compare(i):
        torch.cuda.synchronize()
        t = dws[i % 3].tensors
        z = torch.einsum("ejd,td->tej", t["U"].double(), seen["x"].double())
        ref = torch.einsum("tej,ecj->tc", scores[i].double()[:, :, None] * z * torch.sigmoid(z), t["D"].double())
        assert (h.double() - seen["h"] - ref).abs().max().item() <= 2e-2 * ref.square().mean().sqrt().item() + 1e-5
        seen["h"], seen["x"] = h.double(), x[(i + 1) % 2].clone()
        assert torch.equal(seen["x"], h.bfloat16())
    torch.cuda.synchronize()
    before = layer.launch_count()
    chain(compare)
    assert layer.launch_count() - before == n          # one kernel each
    want = (h.clone(), x.clone())
    for _ in range(3):
        chain()
    torch.cuda.synchronize()
    assert torch.equal(h, want[0]) and torch.equal(x, want[1])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain()
    for _ in range(5):
        graph.replay()
    chain()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(h, want[0]) and torch.equal(x, want[1])
    assert layer.last_status() == 0


@pytest.mark.parametrize("L", [12, 32])
def test_a_call_behind_one_that_gives_up(L):
    """The call before holds the device until its wait has run out. Those of the next one, whose CTAs are
    there already, start behind it."""
    d, E, d_e = 2048, 128, 128
    layer, dw = B.Layer(d, E, d_e, L_max=L), make(d, E, d_e, 1, 0.0)
    cfg = B.Config.from_address(layer.h.value)       # the handle begins with its configuration
    assert (cfg.d, cfg.E, cfg.d_e, cfg.L_max, cfg.flags) == (d, E, d_e, L, 0)
    x = torch.randn(L, d, device="cuda").bfloat16()
    scores = torch.rand(L, E, device="cuda") * (torch.arange(E, device="cuda") % 3 == 0)
    want, held, out = (torch.full((L, d), 7.0, device="cuda") for _ in range(3))

    def call(o, flags):
        cfg.flags = flags
        B.blockffn_layer_forward_scores(layer.h, dw.struct, x, scores, L, o, call_flags=B.CALL_INDEPENDENT)
        cfg.flags = 0
    torch.cuda.synchronize()
    call(want, 0)
    for _ in range(3):
        out.fill_(7.0)
        torch.cuda.synchronize()
        call(held, B.CFG_TEST_EXPIRE_WAIT)
        call(out, 0)
        assert layer.last_status(clear=True) == B.DEV_WAIT_EXPIRED
        assert bool((held == 7.0).all()) and torch.equal(out, want)


@pytest.mark.parametrize("kind", ["logits", "h, router on", "scores", "list"])
@pytest.mark.parametrize("flags", [0, B.CALL_INDEPENDENT])
@pytest.mark.parametrize("L", [12, 32])
def test_all_ctas_that_give_up(L, flags, kind):
    """The bounded waits, for logits and for the intermediate, in every form of the kernel: out stays as it was."""
    d, E, d_e = 2048, 128, 128
    held = B.Layer(d, E, d_e, L_max=L, flags=B.CFG_TEST_EXPIRE_WAIT | (B.CFG_NO_SPLIT if kind == "h, router on" else 0))
    dw, x = make(d, E, d_e, 2, -0.5), torch.randn(L, d, device="cuda").bfloat16()
    scores = torch.rand(L, E, device="cuda") * (torch.arange(E, device="cuda") % 3 == 0)
    ids = torch.arange(E, dtype=torch.int32, device="cuda") * 3 % E
    n = torch.tensor([E // 3], dtype=torch.int32, device="cuda")
    out = torch.full((L, d), 7.0, device="cuda")
    torch.cuda.synchronize()
    for _ in range(3):
        if kind in ("logits", "h, router on"):
            B.blockffn_layer_forward(held.h, dw.struct, x, L, out, call_flags=flags)
        elif kind == "scores":
            B.blockffn_layer_forward_scores(held.h, dw.struct, x, scores, L, out, call_flags=flags)
        else:
            B.blockffn_expert_ffn(held.h, dw.struct, x, scores, L, ids, n, out, call_flags=flags)
        assert held.last_status(clear=True) == B.DEV_WAIT_EXPIRED
        assert bool((out == 7.0).all())


@pytest.mark.parametrize("kind", ["masks", "h, router on", "h, scores", "h, list"])
@pytest.mark.parametrize("L", [12, 32])
def test_one_cta_that_gives_up(L, kind):
    """One CTA of the first cluster runs out of time alone, rows of U being in several passes. With the union not
    known to it, the intermediate stays incomplete and nobody writes out; with h missing, its cluster's columns
    are not written and the others are as always. All come to their end, and the next calls are right."""
    d, E, d_e = 2048, 128, 128
    layer, dw = B.Layer(d, E, d_e, L_max=32), make(d, E, d_e, 4, 9.0)
    cfg = B.Config.from_address(layer.h.value)
    assert (cfg.d, cfg.E, cfg.d_e, cfg.L_max, cfg.flags) == (d, E, d_e, 32, 0)
    x = torch.randn(L, d, device="cuda").bfloat16()
    scores = torch.rand(L, E, device="cuda") + 0.1
    ids, n = torch.arange(E, dtype=torch.int32, device="cuda"), torch.tensor([E], dtype=torch.int32, device="cuda")
    flags = B.CFG_TEST_EXPIRE_WAIT | B.CFG_NO_CHAINING | (B.CFG_NO_SPLIT if kind == "h, router on" else 0)

    def call(o):
        if kind in ("masks", "h, router on"):
            B.blockffn_layer_forward(layer.h, dw.struct, x, L, o)
        elif kind == "h, scores":
            B.blockffn_layer_forward_scores(layer.h, dw.struct, x, scores, L, o)
        else:
            B.blockffn_expert_ffn(layer.h, dw.struct, x, scores, L, ids, n, o)
    want, out = (torch.full((L, d), 7.0, device="cuda") for _ in range(2))
    call(want)
    assert layer.last_status() == 0 and not bool((want == 7.0).all(0).any())
    for _ in range(3):
        out.fill_(7.0)
        cfg.flags = flags
        call(out)
        cfg.flags = 0
        assert layer.last_status(clear=True) == B.DEV_WAIT_EXPIRED
        untouched = (out == 7.0).all(0)
        if kind == "masks":
            assert bool(untouched.all())
        else:
            c = int(untouched.sum())
            assert 1 < c <= 64 and bool(untouched[:c].all()) and torch.equal(out[:, c:], want[:, c:])
        out.fill_(7.0)
        call(out)
        assert torch.equal(out, want) and layer.last_status() == 0
