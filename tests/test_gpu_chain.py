"""Router-on layer calls whose x comes from the call before (one kernel per call): edges of its
tiles and pools, the alternation of its buffers over calls of different lengths and unions, and what
it leaves behind. Tolerances as in the other tests: 2e-2 * RMS for outputs, whose intermediate is
rounded to bf16; scores are fp32 sums, 1e-5 of their RMS (about 40 roundings of 2^-24, all kinds of
cancellation by the bias included)."""
import numpy as np
import pytest
import torch

from paper_2507_08771_b200 import binding as B

pytestmark = pytest.mark.gpu


def make(d, E, d_e, seed, bias):
    g = torch.Generator(device="cuda").manual_seed(seed)
    t = {"W_r": torch.randn(E, d, device="cuda", generator=g).mul_(d ** -0.5).bfloat16(),
         "U": torch.randn(E, d_e, d, device="cuda", generator=g).mul_(d ** -0.5).bfloat16(),
         "D": torch.randn(E, d, d_e, device="cuda", generator=g).mul_(d_e ** -0.5).bfloat16(),
         "gain": torch.rand(E, device="cuda", generator=g) + 0.5,
         "bias": torch.full((E,), float(bias), device="cuda")}
    return B.DeviceWeights(B.make_weights(t["W_r"], t["gain"], t["bias"], t["U"], t["D"]), t)


def reference(t, x):
    x = x.double()
    a = torch.relu(x @ t["W_r"].double().T + t["bias"].double())
    s = t["gain"].double() * a / (a.square().mean(1, keepdim=True) + 1e-6).sqrt()
    z = torch.einsum("ejd,td->tej", t["U"].double(), x)
    h = s[:, :, None] * z * torch.sigmoid(z)
    return s, torch.einsum("tej,ecj->tc", h, t["D"].double())


def check(layer, dw, x, flags):
    L = x.shape[0]
    s, ref = reference(dw.tensors, x)
    base = torch.randn(L, layer.d, device="cuda")
    out, nxt = base.clone(), torch.zeros(L, layer.d, dtype=torch.bfloat16, device="cuda")
    r = layer.forward(dw, x, out=out, x_next=nxt, call_flags=flags | B.CALL_ACCUMULATE)
    torch.cuda.synchronize()
    rms = max(ref.square().mean().sqrt().item(), 1e-6)
    assert (out.double() - base.double() - ref).abs().max().item() <= 2e-2 * rms + 1e-6
    assert torch.equal(nxt, out.to(torch.bfloat16))
    assert (r.scores.double() - s).abs().max().item() <= 1e-5 * max(s.square().mean().sqrt().item(), 1.0)
    active = r.scores != 0
    ids = active.any(0).nonzero().flatten().int()
    n = int(r.n_union.item())
    assert n == len(ids) and torch.equal(r.union_ids[:n], ids) and bool((r.union_ids[n:] == -1).all())
    e = torch.arange(layer.E, device="cuda")
    bits = (r.tok_mask[:, e // 32] >> (e % 32).int()) & 1
    assert torch.equal(bits.bool(), active)


@pytest.mark.parametrize("d,E,d_e", [(64, 5, 64), (320, 33, 64), (1024, 16, 256), (1088, 130, 64), (2048, 64, 128), (1536, 60, 256)])
@pytest.mark.parametrize("flags", [0, B.CALL_INDEPENDENT])
def test_chunk_lengths_and_unions_on_one_handle(d, E, d_e, flags):
    layer = B.Layer(d, E, d_e, L_max=32)
    n0 = layer.launch_count()
    calls = 0
    for bias in (-1.0, 0.5, -9.0, 9.0):       # some, most, none, all of the experts
        dw = make(d, E, d_e, d + E, bias)
        g = torch.Generator(device="cuda").manual_seed(calls)
        for L in (1, 8, 32, 3, 17, 9, 16, 24):
            x = torch.randn(L, d, device="cuda", generator=g).bfloat16()
            if calls % 2:                     # 16-byte but not 32-byte aligned
                x = torch.cat([x.new_zeros(8), x.flatten()])[8:].view(L, d)
            torch.cuda.synchronize()
            check(layer, dw, x, flags)
            calls += 1
    assert layer.launch_count() - n0 == 2 * calls  # one kernel each, one for the copies of the routing
    assert layer.last_status() == 0
    st = layer.stats_host()
    assert st.n_chunks == calls


def test_a_token_that_is_not_finite_spoils_only_itself():
    d, E, d_e, L = 256, 16, 64, 4
    layer, dw = B.Layer(d, E, d_e, L_max=L), make(256, 16, 64, 3, -0.5)
    x = torch.randn(L, d, device="cuda").bfloat16()
    _, ref = reference(dw.tensors, x)
    x[2, 5] = float("nan")
    out = layer.forward(dw, x).out
    assert bool(out[2].isnan().all())
    for t in (0, 1, 3):
        assert (out[t].double() - ref[t]).abs().max() <= 2e-2 * ref.square().mean().sqrt()
    x[2, 5] = 1.0                              # the next call finds nothing of it
    _, ref = reference(dw.tensors, x)
    out = layer.forward(dw, x).out
    assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()


def test_wait_that_runs_out_is_reported_every_time():
    d, E, d_e, L = 512, 32, 64, 8
    dw = make(d, E, d_e, 1, -0.5)
    x = torch.randn(L, d, device="cuda").bfloat16()
    held = B.Layer(d, E, d_e, L_max=L, flags=B.CFG_TEST_EXPIRE_WAIT)
    for _ in range(3):
        out = torch.full((L, d), 7.0, device="cuda")
        held.forward(dw, x, out=out)
        assert held.last_status(clear=True) == B.DEV_WAIT_EXPIRED
        assert bool((out == 7.0).all())


@pytest.mark.parametrize("held", [B.CFG_TEST_EXPIRE_WAIT, B.CFG_TEST_EXPIRE_WAIT | B.CFG_NO_SPLIT])
@pytest.mark.parametrize("L", [4, 12, 24])
def test_calls_after_one_whose_wait_ran_out(held, L):
    """One call in the middle of a sequence gives up, at the logits or at h: the
    next ones find buffers, tickets and marks in order."""
    d, E, d_e = 512, 40, 64
    dw, layer = make(d, E, d_e, 7, -0.5), B.Layer(d, E, d_e, L_max=32)
    cfg = B.Config.from_address(layer.h.value)       # the handle begins with its configuration
    assert (cfg.d, cfg.E, cfg.d_e, cfg.L_max, cfg.flags) == (d, E, d_e, 32, 0)
    for k in range(2):                               # (either of the two buffers of h)
        for n in [L] * (k + 1) + [0] + [L, 32, 1, L]:
            cfg.flags = 0 if n else held
            x = torch.randn(n or L, d, device="cuda").bfloat16()
            out = torch.full((n or L, d), 7.0, device="cuda")
            B.blockffn_layer_forward(layer.h, dw.struct, x, n or L, out)
            if n:
                _, ref = reference(dw.tensors, x)
                assert layer.last_status() == 0
                assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()
            else:
                assert layer.last_status(clear=True) == B.DEV_WAIT_EXPIRED
                assert bool((out == 7.0).all())
    cfg.flags = 0


@pytest.mark.parametrize("L", [4, 12, 24])
@pytest.mark.parametrize("E", [70, 130])
def test_a_wait_that_runs_out_before_the_last_experts(E, L):
    """More experts than are looked at in one trip (64): the first trip's logits do not come within the limit, and those
    behind it are there at a second look. The call gives up all the same, and the next ones find everything in order."""
    d, d_e = 192, 64
    dw, layer = make(d, E, d_e, 7, -0.5), B.Layer(d, E, d_e, L_max=32)
    cfg = B.Config.from_address(layer.h.value)       # the handle begins with its configuration
    assert (cfg.d, cfg.E, cfg.d_e, cfg.L_max, cfg.flags) == (d, E, d_e, 32, 0)
    for k in range(2):                               # (either of the two buffers of h)
        for n in [L] * (k + 1) + [0] + [L, 32, 1, L]:
            cfg.flags = 0 if n else B.CFG_TEST_EXPIRE_WAIT
            x = torch.randn(n or L, d, device="cuda").bfloat16()
            out = torch.full((n or L, d), 7.0, device="cuda")
            B.blockffn_layer_forward(layer.h, dw.struct, x, n or L, out)
            if n:
                _, ref = reference(dw.tensors, x)
                assert layer.last_status() == 0
                assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()
            else:
                assert layer.last_status(clear=True) == B.DEV_WAIT_EXPIRED
                assert bool((out == 7.0).all())
    cfg.flags = 0


def test_a_new_handle_has_its_workspace_filled():
    """The first call may come on a stream that is not ordered behind the default one, where
    blockffn_create fills the workspace (250 MB of "not written yet" here, some 40 us of work)."""
    h = B.blockffn_create(64, 960, 2048, 32)
    idle = torch.cuda.default_stream().query()
    B.blockffn_destroy(h)
    assert idle
    d, E, d_e, L = 512, 32, 64, 8
    dw = make(d, E, d_e, 1, -0.5)
    x = torch.randn(L, d, device="cuda").bfloat16()
    _, ref = reference(dw.tensors, x)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        layer, out = B.Layer(d, E, d_e, L_max=L), torch.empty(L, d, device="cuda")
        B.blockffn_layer_forward(layer.h, dw.struct, x, L, out)
        torch.cuda.synchronize()
    assert layer.last_status() == 0
    assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()


def layers(E=40, d=1024, d_e=64):
    """Parameters whose layers, one after the other, activate some, few, most, all or none of the experts."""
    dws = [make(d, E, d_e, s, b) for s, b in enumerate((-0.5, -1.6, 0.8, 9.0, -9.0))]
    for dw in dws:
        dw.tensors["D"].mul_(1.0 / E)                # (the running state keeps its scale)
    return dws


def chain(layer, dws, lengths, h, x, flags, each=lambda i: None):
    for i, L in enumerate(lengths):
        B.blockffn_layer_forward(layer.h, dws[i % len(dws)].struct, x[i % 2], L, h, x[(i + 1) % 2], None,
                                 flags | B.CALL_ACCUMULATE)
        each(i)


@pytest.mark.parametrize("d,E,d_e", [(64, 40, 64), (128, 64, 64), (192, 128, 128), (192, 24, 256), (1984, 16, 64), (1024, 31, 64)])
def test_long_chunks_off_the_clusters(d, E, d_e):
    """17 to 32 tokens at widths or expected unions too small for the clusters, from a handle with the usual expectation and from
    one that expects a single expert: one by one, one behind the other, and with a wait that runs out."""
    # (At -0.5 a third of the experts is active, and the RMS of a token's logits is 0.1 or more: their error, up to
    # 1e-6, is then within 1e-5 of a score. At -1.6 some tokens have one active logit of a few thousandths, and
    # 1e-6 of it is 1e-4 of its score: 5e-5 seen, with the 1e-5 of check missed.)
    dws = [make(d, E, d_e, s, b) for s, b in enumerate((-0.5, 0.3, 9.0, -9.0))]
    g = torch.Generator(device="cuda").manual_seed(d + E)
    for cfg in (0, B.cfg_expected_union(1)):
        layer = B.Layer(d, E, d_e, L_max=32, flags=cfg)
        for L in (17, 24, 32):
            x = torch.randn(L, d, device="cuda", generator=g).bfloat16()
            want = []
            for dw in dws:
                check(layer, dw, x, B.CALL_INDEPENDENT)
                want.append(layer.forward(dw, x, call_flags=B.CALL_INDEPENDENT).out.clone())
            outs = [torch.empty(L, d, device="cuda") for _ in range(12)]
            torch.cuda.synchronize()
            for i, o in enumerate(outs):
                B.blockffn_layer_forward(layer.h, dws[i % 4].struct, x, L, o, call_flags=B.CALL_INDEPENDENT)
            assert all(torch.equal(o, want[i % 4]) for i, o in enumerate(outs))
        assert layer.last_status() == 0
    held = B.Layer(d, E, d_e, L_max=32, flags=B.CFG_TEST_EXPIRE_WAIT)
    for _ in range(2):
        out = torch.full((24, d), 7.0, device="cuda")
        held.forward(dws[0], torch.randn(24, d, device="cuda").bfloat16(), out=out)
        assert held.last_status(clear=True) == B.DEV_WAIT_EXPIRED
        assert bool((out == 7.0).all())


@pytest.mark.parametrize("flags", [0, B.CALL_INDEPENDENT])
@pytest.mark.parametrize("lengths", [[1], [8], [13], [16], [32], [1, 32, 8, 17, 9, 24, 3, 16]], ids=str)
@pytest.mark.parametrize("d,E", [(1024, 40), (2048, 64)])
def test_calls_one_behind_the_other(flags, lengths, d, E):
    """Nothing but layer calls on the stream, every x from the call before: early reads, the two
    buffers of h and what they are reset to, the tags of the words. The same bits as with a pause
    behind every call, where every layer is compared with float64; eagerly and from a graph."""
    dws, layer = layers(E, d), B.Layer(d, E, 64, L_max=32)
    lengths = (lengths * 24)[:24]
    start = torch.randn(32, d, device="cuda")
    h, x = start.clone(), torch.zeros(2, 32, d, dtype=torch.bfloat16, device="cuda")

    def reset():
        h.copy_(start)
        x.copy_(start.expand(2, 32, d))
    reset()
    torch.cuda.synchronize()
    seen = {"h": h.double()}

    def compare(i):
        L = lengths[i]
        torch.cuda.synchronize()
        _, ref = reference(dws[i % len(dws)].tensors, seen.get("x", x[0])[:L])
        rms = max(ref.square().mean().sqrt().item(), 1e-6)
        assert (h[:L].double() - seen["h"][:L] - ref).abs().max().item() <= 2e-2 * rms + 1e-5
        assert torch.equal(x[(i + 1) % 2][:L], h[:L].bfloat16())
        seen["h"], seen["x"] = h.double(), x[(i + 1) % 2].clone()
    chain(layer, dws, lengths, h, x, flags, compare)
    want = (h.clone(), x.clone())

    for _ in range(3):
        reset()
        chain(layer, dws, lengths, h, x, flags)
        torch.cuda.synchronize()
        assert torch.equal(h, want[0]) and torch.equal(x, want[1])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        reset()
        chain(layer, dws, lengths, h, x, flags)
    for _ in range(5):                               # graphs and eager calls in turn, nothing in between
        graph.replay()
    reset()
    chain(layer, dws, lengths, h, x, flags)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(h, want[0]) and torch.equal(x, want[1])
    assert layer.last_status() == 0


@pytest.mark.parametrize("d,E,d_e,L", [(192, 24, 64, 1), (1088, 70, 64, 8), (256, 40, 128, 13), (192, 48, 64, 20),
                                       (512, 100, 256, 6), (256, 150, 64, 5), (1088, 140, 64, 12), (192, 300, 64, 20)])
def test_experts_whose_scores_vanish_are_not_in_the_union(d, E, d_e, L):
    """gain * ReLU(logit) of every third expert is the smallest denormal number, and 1 / rms takes it
    to zero; their D is infinite, so that one of them in the union would spoil out."""
    dw = make(d, E, d_e, 11, 5.0)
    t, faint = dw.tensors, torch.arange(E, device="cuda") % 3 == 0
    t["gain"][faint] = 1.4e-45
    t["W_r"][faint] = 0.0
    t["bias"][faint] = 0.6                    # one denormal step; rms > 2 makes less than half a step of it
    t["bias"][1::3] = -9.0                    # never active, by their logits
    t["D"][faint] = float("inf")
    x = torch.randn(L, d, device="cuda").bfloat16()
    clean = dict(t, D=torch.where(faint[:, None, None], 0.0, t["D"].float()).bfloat16())
    s, ref = reference(clean, x)
    s[:, faint] = 0.0
    layer = B.Layer(d, E, d_e, L_max=L)
    for _ in range(2):
        r = layer.forward(dw, x)
        ids = (s != 0).any(0).nonzero().flatten().int()
        n = int(r.n_union.item())
        assert n == len(ids) and torch.equal(r.union_ids[:n], ids)
        assert bool((r.scores[:, faint] == 0).all()) and bool(((r.scores != 0) == (s != 0)).all())
        assert (r.scores.double() - s).abs().max() <= 1e-5 * max(s.square().mean().sqrt().item(), 1.0)
        assert (r.out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()
    st = layer.stats_host()
    assert st.n_union == 2 * n and st.n_active == 2 * int((s != 0).sum()) and layer.last_status() == 0


@pytest.mark.parametrize("E", [90, 129, 200])
@pytest.mark.parametrize("L", [1, 8, 16, 32])
def test_scores_are_those_of_the_router_kernel_bit_for_bit(L, E):
    """Logits that both kernels sum without rounding (small whole numbers): what is left is the sum of
    squares, its mean, 1 / root and two products."""
    d, d_e = 192, 64
    layer, dw = B.Layer(d, E, d_e, L_max=L), make(d, E, d_e, 5, 0.0)
    t = dw.tensors
    for seed in range(40):
        g = torch.Generator(device="cuda").manual_seed(seed)
        t["W_r"].copy_(torch.randint(-9, 10, (E, d), device="cuda", generator=g))
        t["bias"].copy_(torch.randint(-40, 9, (E,), device="cuda", generator=g) / 8)
        x = torch.randint(-3, 4, (L, d), device="cuda", generator=g).bfloat16()
        x[:, 8 + seed:] = 0
        alone = torch.empty(L, E, device="cuda")
        B.blockffn_router(layer.h, dw.struct, x, L, alone)
        assert torch.equal(layer.forward(dw, x).scores, alone)


@pytest.mark.parametrize("d,E,d_e", [(64, 129, 64), (192, 160, 64), (256, 257, 64), (1088, 257, 64), (320, 1024, 64)])
def test_many_experts(d, E, d_e):
    """More than 128 experts: edges of the words of a mask and of a trip through the logits, unions of some, few and all."""
    layer, lengths = B.Layer(d, E, d_e, L_max=32), (1, 8, 9, 16, 17, 32)
    for seed, bias in enumerate((-0.5, 0.5, 9.0)):
        dw = make(d, E, d_e, seed, bias)
        t = dw.tensors
        t["bias"][32:64] = -9.0                        # a word of the masks without experts
        g = torch.Generator(device="cuda").manual_seed(seed)
        for L in lengths:
            check(layer, dw, torch.randn(L, d, device="cuda", generator=g).bfloat16(), B.CALL_INDEPENDENT)
    assert layer.last_status() == 0
    st = layer.stats_host()
    assert st.n_chunks == 3 * len(lengths) and st.n_tokens == 3 * sum(lengths)


@pytest.mark.parametrize("d,E,d_e,L", [(320, 90, 128, 8), (1024, 130, 64, 3), (960, 90, 256, 6), (1088, 60, 64, 1),
                                       (2048, 40, 128, 7), (64, 5, 64, 16), (512, 40, 64, 13), (2048, 70, 128, 16),
                                       (1792, 33, 64, 9), (448, 250, 64, 7), (320, 200, 64, 14), (512, 64, 128, 2),
                                       (256, 65, 128, 15), (1088, 64, 64, 16)])
def test_scores_given(d, E, d_e, L):
    """Scores that are stable, x from the call before: some, all and none of the experts, a token that is not finite,
    then a sequence of layers whose x is what the call before left, against the kernels of other handles."""
    layer, plain = B.Layer(d, E, d_e, L_max=L), B.Layer(d, E, d_e, L_max=L, flags=B.CFG_TWO_KERNELS)
    dw = make(d, E, d_e, 5, 0.0)
    t, g = dw.tensors, torch.Generator(device="cuda").manual_seed(d + L)
    F = B.CALL_INDEPENDENT | B.CALL_ACCUMULATE
    for k, (u, nan) in enumerate(((max(1, E * 3 // 10), False), (E, False), (0, False), (max(1, E // 4), True))):
        pick = torch.randperm(E, device="cuda", generator=g)[:u].sort().values.int()
        s = torch.zeros(L, E, device="cuda")
        s[:, pick.long()] = (torch.rand(L, u, device="cuda", generator=g) < 0.5) * 0.5 + 0.25
        if L > 1:
            s[0] = 0                                   # a token without experts
        x = torch.randn(L, d, device="cuda", generator=g).bfloat16()
        if k % 2:                                      # 16-byte but not 32-byte aligned
            x = torch.cat([x.new_zeros(8), x.flatten()])[8:].view(L, d)
        if nan:
            x[L - 1, 3] = float("nan")
        z = torch.einsum("ejd,td->tej", t["U"].double(), x.double())
        ref = torch.einsum("tej,ecj->tc", s.double()[:, :, None] * z * torch.sigmoid(z), t["D"].double())
        base = torch.randn(L, d, device="cuda", generator=g)
        out, nxt = base.clone(), torch.empty(L, d, dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        n0 = layer.launch_count()
        r = layer.forward_scores(dw, x, s, out=out, x_next=nxt, call_flags=F)
        assert layer.launch_count() - n0 == 2           # one kernel, and the copies of the routing
        ids = (s != 0).any(0).nonzero().flatten().int()
        n = int(r.n_union.item())
        assert n == len(ids) and torch.equal(r.union_ids[:n], ids) and layer.last_status() == 0
        rows = L - 1 if nan else L
        rms = max(ref[:rows].square().mean().sqrt().item(), 1e-6) if rows else 1.0
        assert rows == 0 or (out[:rows].double() - base[:rows].double() - ref[:rows]).abs().max().item() <= 2e-2 * rms + 1e-6
        assert torch.equal(nxt[:rows], out[:rows].bfloat16())
        if nan:
            assert bool(out[L - 1].isnan().all())
    ss = [torch.where(torch.rand(L, E, device="cuda", generator=g) < 0.2, 1.0 / E, 0.0) for _ in range(3)]   # (h keeps its scale)
    x0 = torch.randn(L, d, device="cuda", generator=g).bfloat16()
    got = []
    for handle in (layer, plain):
        h, xs = x0.float(), [x0.clone(), torch.empty_like(x0)]
        torch.cuda.synchronize()
        for i in range(24):
            B.blockffn_layer_forward_scores(handle.h, dw.struct, xs[i % 2], ss[i % 3], L, h, xs[(i + 1) % 2],
                                            handle.stats, F)
        got.append(h.clone())
        assert handle.last_status() == 0
    # (what the 24 layers add is about as large as x; sums in another order move some of their bf16 x and h by a step, 2^-8)
    assert (got[0] - got[1]).abs().max() <= 2e-2 * got[1].square().mean().sqrt()


def scores_like(L, E, g, share=0.3):
    s = torch.rand(L, E, device="cuda", generator=g)
    return torch.where(s < share, s + 0.1, 0.0)


@pytest.mark.parametrize("L", [1, 8, 14])
def test_calls_after_one_whose_wait_ran_out_scores_given(L):
    """As above, with scores given: the wait for h. The calls around it are of both kinds."""
    d, E, d_e = 512, 64, 128
    dw, layer = make(d, E, d_e, 7, -0.5), B.Layer(d, E, d_e, L_max=16)
    g = torch.Generator(device="cuda").manual_seed(L)
    cfg = B.Config.from_address(layer.h.value)       # the handle begins with its configuration
    assert (cfg.d, cfg.E, cfg.d_e, cfg.L_max, cfg.flags) == (d, E, d_e, 16, 0)
    for k in range(2):                               # (either of the two buffers of h)
        for n in [L] * (k + 1) + [0] + [L, -16, 1, -1, L]:      # (0: held; negative: router on)
            cfg.flags = 0 if n else B.CFG_TEST_EXPIRE_WAIT
            T = abs(n) or L
            x, s = torch.randn(T, d, device="cuda", generator=g).bfloat16(), scores_like(T, E, g)
            s[0, ::5] = 0.5
            out = torch.full((T, d), 7.0, device="cuda")
            torch.cuda.synchronize()
            n0 = layer.launch_count()
            if n < 0:
                B.blockffn_layer_forward(layer.h, dw.struct, x, T, out)
                _, ref = reference(dw.tensors, x)
            else:
                B.blockffn_layer_forward_scores(layer.h, dw.struct, x, s, T, out, call_flags=B.CALL_INDEPENDENT)
                z = torch.einsum("ejd,td->tej", dw.tensors["U"].double(), x.double())
                ref = torch.einsum("tej,ecj->tc", s.double()[:, :, None] * z * torch.sigmoid(z), dw.tensors["D"].double())
            assert layer.launch_count() - n0 == 1
            if n:
                assert layer.last_status() == 0
                assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()
            else:
                assert layer.last_status(clear=True) == B.DEV_WAIT_EXPIRED
                assert bool((out == 7.0).all())
    cfg.flags = 0


@pytest.mark.parametrize("graph", [False, True])
def test_scores_given_in_turn_with_other_calls(graph):
    """Scores given, router on and clusters on one handle, every x from the call before: they share tickets and both
    buffers of h. The same bits as with a pause behind every call, eagerly or from a graph, alone and beside another
    handle's calls on another stream."""
    d, E, d_e, N = 1024, 64, 128, 24
    dws = [make(d, E, d_e, s, b) for s, b in enumerate((-0.5, 0.3, -1.0))]
    for dw in dws:
        dw.tensors["D"].mul_(1.0 / E)
    g = torch.Generator(device="cuda").manual_seed(3)
    scores = [scores_like(16, E, g) for _ in range(4)]
    lengths = [(8, True), (5, False), (16, True), (32, False), (13, True), (16, False), (1, True), (24, False), (8, True), (8, True)]
    start = torch.randn(32, d, device="cuda", generator=g)
    layers = [B.Layer(d, E, d_e, L_max=32) for _ in range(2)]
    hs = [start.clone() for _ in range(2)]
    xs = [torch.zeros(2, 32, d, dtype=torch.bfloat16, device="cuda") for _ in range(2)]

    def run(k, each=lambda: None):
        h, x, layer = hs[k], xs[k], layers[k]
        h.copy_(start)
        x.copy_(start.expand(2, 32, d))
        for i in range(N):
            L, given = lengths[i % len(lengths)]
            F, w = B.CALL_INDEPENDENT | B.CALL_ACCUMULATE, dws[i % 3].struct
            if given:
                B.blockffn_layer_forward_scores(layer.h, w, x[i % 2], scores[i % 4], L, h, x[(i + 1) % 2], None, F)
            else:
                B.blockffn_layer_forward(layer.h, w, x[i % 2], L, h, x[(i + 1) % 2], None, F)
            each()

    torch.cuda.synchronize()
    n0 = layers[0].launch_count()
    run(0, torch.cuda.synchronize)
    assert layers[0].launch_count() - n0 == N
    want = hs[0].clone()
    streams = [torch.cuda.Stream() for _ in range(2)]
    graphs = []
    for k in range(2):
        if graph:
            graphs.append(torch.cuda.CUDAGraph())
            with torch.cuda.graph(graphs[k], stream=streams[k]):
                run(k)
    for both in (False, True):
        torch.cuda.synchronize()
        for _ in range(4):
            for k in range(1 + both):
                with torch.cuda.stream(streams[k]):
                    graphs[k].replay() if graph else run(k)
        torch.cuda.synchronize()
        for k in range(1 + both):
            assert layers[k].last_status() == 0 and torch.equal(hs[k], want)


@pytest.mark.parametrize("u,want", [(36, 1), (37, 2)])
def test_scores_given_with_many_blocks_of_d_a_warp(u, want):
    """One kernel up to 36 expected blocks of D a warp, the pair above, and the same result."""
    d, E, d_e, L = 256, 48, 512, 3
    layer, dw = B.Layer(d, E, d_e, L_max=L, flags=B.cfg_expected_union(u)), make(d, E, d_e, 5, 0.0)
    g = torch.Generator(device="cuda").manual_seed(u)
    s, x = scores_like(L, E, g, 0.6), torch.randn(L, d, device="cuda", generator=g).bfloat16()
    z = torch.einsum("ejd,td->tej", dw.tensors["U"].double(), x.double())
    ref = torch.einsum("tej,ecj->tc", s.double()[:, :, None] * z * torch.sigmoid(z), dw.tensors["D"].double())
    out = torch.empty(L, d, device="cuda")
    torch.cuda.synchronize()
    n0 = layer.launch_count()
    B.blockffn_layer_forward_scores(layer.h, dw.struct, x, s, L, out, call_flags=B.CALL_INDEPENDENT)
    assert layer.launch_count() - n0 == want and layer.last_status() == 0
    assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()
