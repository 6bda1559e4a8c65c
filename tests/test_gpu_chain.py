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


@pytest.mark.parametrize("d,E,d_e", [(64, 5, 64), (320, 33, 64), (1024, 16, 256), (1088, 130, 64), (2048, 64, 128)])
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


def test_wait_that_runs_out_leaves_the_handle_usable():
    d, E, d_e, L = 512, 32, 64, 8
    dw = make(d, E, d_e, 1, -0.5)
    x = torch.randn(L, d, device="cuda").bfloat16()
    held = B.Layer(d, E, d_e, L_max=L, flags=B.CFG_TEST_EXPIRE_WAIT)
    for _ in range(3):
        out = torch.full((L, d), 7.0, device="cuda")
        held.forward(dw, x, out=out)
        assert held.last_status(clear=True) == B.DEV_WAIT_EXPIRED
        assert bool((out == 7.0).all())


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
