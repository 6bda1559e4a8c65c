"""The expert stage for any shape (32-bit intermediate), at the edges of its tiles: 16 rows or
columns per tile, 32 k per step, 8 tokens per group, steps dealt out to 8 warps.

Tolerance: the intermediate and all sums are fp32. An output is a sum of at most 2000 terms here,
added in chains of at most 64 plus a tree; with independent roundings of 2^-24 that is below
sqrt(64) 2^-24 = 5e-7 of the RMS and five times that over the largest of some 10^4 outputs, and the
tensor cores cut sums of 32 products off rather than round them. 2e-5 * RMS leaves a factor of 8.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_08771_b200 import binding as B
from paper_2507_08771_b200 import inputs as I

pytestmark = pytest.mark.gpu

TOL = 2e-5


def scores_of(rng, L, E, p):
    s = (np.abs(rng.standard_normal((L, E))) + 0.05).astype(np.float32)
    s[rng.random((L, E)) >= p] = 0.0
    return s


def reference(x, s, w, ids):
    return oracle.expert_ffn(x, s.astype(np.float64), w["U"], w["D"], expert_ids=ids)


@pytest.mark.parametrize("d,E,d_e,L", [
    (8, 3, 8, 1), (24, 5, 40, 7), (264, 9, 56, 8), (1000, 7, 24, 9), (512, 33, 64, 16),
    (72, 40, 104, 17), (328, 12, 168, 32), (4104, 2, 8, 3),
])
@pytest.mark.parametrize("flags", [0, B.CALL_INDEPENDENT, B.CALL_INDEPENDENT_X])
def test_edges_of_tiles(d, E, d_e, L, flags):
    w = I.make_layer(I.Shape("t", d=d, E=E, d_e=d_e, L=L, union_frac=0.3), 77)
    layer = B.Layer(d, E, d_e, L_max=L, variant=B.VARIANT_SIMT)
    dw = layer.upload_weights(w)
    rng = np.random.default_rng(d + E)
    for p in (0.4, 1.0, 0.0):
        x, s = I.make_x(d, L, 77), scores_of(rng, L, E, p)
        ids = np.flatnonzero(s.any(0)).astype(np.int32)
        ref = reference(x, s, w, ids)
        rms = float(np.sqrt(np.mean(ref ** 2)))
        xd, sd = B.to_device_bf16(x), torch.from_numpy(s).cuda()
        base = torch.randn(L, d, device="cuda")
        torch.cuda.synchronize()
        out = base.clone()
        nxt = torch.zeros(L, d, dtype=torch.bfloat16, device="cuda")
        torch.cuda.synchronize()
        r = layer.forward_scores(dw, xd, sd, out=out, x_next=nxt, call_flags=flags | B.CALL_ACCUMULATE)
        assert int(r.n_union.item()) == len(ids)
        want = base.double().cpu().numpy() + ref
        got = out.double().cpu().numpy()
        assert np.abs(got - want).max() <= TOL * (rms + 1.0)
        assert torch.equal(nxt, out.to(torch.bfloat16))
        # the same call with the list given, where there is room an entry out of range in its middle
        bad = len(ids) < E
        lst = np.full(E, -1, np.int32)
        counted = np.insert(ids, len(ids) // 2, E) if bad else ids
        lst[:len(counted)] = counted
        idd = torch.from_numpy(lst).cuda()
        nd = torch.tensor([len(counted)], dtype=torch.int32, device="cuda")
        out2 = torch.full((L, d), float("nan"), device="cuda")
        torch.cuda.synchronize()
        B.blockffn_expert_ffn(layer.h, dw.struct, xd, sd, L, idd, nd, out2, call_flags=flags)
        torch.cuda.synchronize()
        assert np.abs(out2.double().cpu().numpy() - ref).max() <= TOL * max(rms, 1e-30)
        assert layer.last_status(clear=True) == (B.DEV_BAD_UNION_ID if bad else 0)


def test_ends_of_the_float_range():
    """The intermediate is split into three bf16: nothing may overflow on the way, a NaN stays one."""
    d, E, d_e, L = 72, 4, 24, 5
    w = I.make_layer(I.Shape("t", d=d, E=E, d_e=d_e, L=L, union_frac=0.3), 5)
    layer = B.Layer(d, E, d_e, L_max=L, variant=B.VARIANT_SIMT)
    dw = layer.upload_weights(w)
    x = I.make_x(d, L, 5)
    s = np.abs(np.random.default_rng(5).standard_normal((L, E))).astype(np.float32) + 0.1
    s[1] *= np.float32(1e37)
    s[2] *= np.float32(1e-30)
    clean = reference(x, s, w, np.arange(E, dtype=np.int32))
    s[3, 2] = np.nan
    out = layer.forward_scores(dw, B.to_device_bf16(x), torch.from_numpy(s).cuda()).out
    got = out.double().cpu().numpy()
    assert np.isnan(got[3]).all()
    for t in (0, 1, 2, 4):
        assert np.abs(got[t] - clean[t]).max() <= TOL * np.sqrt(np.mean(clean[t] ** 2))


def test_sums_up_to_the_largest_float():
    """The scaled planes of the intermediate may not overflow in sums that do not. Three neurons give
    h = 2^126 (1 + 2^-7 - 2^-23), whose second plane is as large as it gets next to the first; the
    output is their sum, exact to two roundings."""
    d, E, d_e = 8, 1, 8
    U, D = torch.zeros(E, d_e, d), torch.zeros(E, d, d_e)
    U[0, :3, 0], D[0, :, :3] = 32.0, 1.0                   # swish(32) is 32
    t = {"U": U.bfloat16().cuda(), "D": D.bfloat16().cuda()}
    h = 2.0 ** 126 * (1 + 2.0 ** -7 - 2.0 ** -23)
    for L in (1, 9, 17):
        layer = B.Layer(d, E, d_e, L_max=L, variant=B.VARIANT_SIMT)
        x = torch.zeros(L, d, dtype=torch.bfloat16, device="cuda")
        x[:, 0] = 1.0
        s = torch.full((L, E), h / 32, device="cuda")
        out = layer.forward_scores(B.DeviceWeights(B.make_weights(U=t["U"], D=t["D"]), t), x, s).out
        assert ((out.double() - 3 * h).abs() <= 2.0 ** -22 * 3 * h).all()


def test_infinite_weight():
    """An infinite weight gives an infinity, as one fp32 product does: h = swish(32) = 32 is a bf16, so
    the planes behind the first are zero, and zero times an infinity is no number."""
    d, E, d_e = 8, 1, 8
    U, D = torch.zeros(E, d_e, d), torch.zeros(E, d, d_e)
    U[0, 0, 0] = 32.0
    D[0, :, 0] = torch.tensor([float("inf"), -float("inf")] + 6 * [1.0])
    t = {"U": U.bfloat16().cuda(), "D": D.bfloat16().cuda()}
    for L in (1, 9, 17):
        layer = B.Layer(d, E, d_e, L_max=L, variant=B.VARIANT_SIMT)
        x = torch.zeros(L, d, dtype=torch.bfloat16, device="cuda")
        x[:, 0] = 1.0
        s = torch.ones(L, E, device="cuda")
        out = layer.forward_scores(B.DeviceWeights(B.make_weights(U=t["U"], D=t["D"]), t), x, s).out
        assert torch.equal(out, (32.0 * D[0, :, 0]).cuda().expand(L, d))


@pytest.mark.parametrize("d,E,d_e,L", [(1000, 40, 96, 8), (2048, 64, 128, 8), (1000, 40, 96, 1), (1000, 40, 96, 24)])
def test_precision_of_one_call(d, E, d_e, L):
    """One call against float64, without a stack that would round x in between. Products are exact;
    what rounds in one projection is at most eight sums of 32 products in the tensor core, cut off
    (2^-23 of a partial sum), their addition in fp32 and a tree over eight warps: some 12 errors of up
    to 2^-23 of partial sums that are about half the result in RMS, independent of one another,
    sqrt(12) 2^-24 = 3.5 * 2^-24. Both projections: 5 * 2^-24, with the Swish and the score less than
    8 * 2^-24 in the 2-norm. (Measured 2.0 to 2.45; a stack of such layers shows 1e-5 and more once an
    x falls on the other side of a bf16 boundary.)"""
    g = torch.Generator(device="cuda").manual_seed(d + L)
    t = {"U": torch.randn(E, d_e, d, device="cuda", generator=g).mul_(d ** -0.5).bfloat16(),
         "D": torch.randn(E, d, d_e, device="cuda", generator=g).mul_(d_e ** -0.5).bfloat16()}
    x = torch.randn(L, d, device="cuda", generator=g).bfloat16()
    s = torch.randn(L, E, device="cuda", generator=g).abs() + 0.05
    s *= (torch.rand(1, E, device="cuda", generator=g) < 0.3) * (torch.rand(L, E, device="cuda", generator=g) < 0.7)
    z = torch.einsum("ejd,td->tej", t["U"].double(), x.double())
    ref = torch.einsum("tej,ecj->tc", s.double()[:, :, None] * z * torch.sigmoid(z), t["D"].double())
    layer = B.Layer(d, E, d_e, L_max=L, variant=B.VARIANT_SIMT)
    out = layer.forward_scores(B.DeviceWeights(B.make_weights(U=t["U"], D=t["D"]), t), x, s).out
    assert (out.double() - ref).norm() <= 8 * 2.0 ** -24 * ref.norm()


@pytest.mark.parametrize("d,E,d_e,L", [(1000, 40, 96, 8), (264, 9, 56, 17), (1000, 40, 96, 1)])
@pytest.mark.parametrize("kind", ["router", "scores", "independent", "noalloc"])
def test_calls_one_behind_the_other(d, E, d_e, L, kind):
    """Nothing but these calls on the stream: the weights, scores and (independent) x that a call asks
    for under the call before, the one intermediate that all share. The same bits as with a pause
    behind every call, eagerly and from a graph."""
    n = 12
    g = torch.Generator(device="cuda").manual_seed(d + L)
    dws, scores, ids, nu = [], [], [], []
    for i in range(3):
        t = {"U": torch.randn(E, d_e, d, device="cuda", generator=g).mul_(d ** -0.5).bfloat16(),
             "D": torch.randn(E, d, d_e, device="cuda", generator=g).mul_(d_e ** -0.5 / E).bfloat16(),
             "W_r": torch.randn(E, d, device="cuda", generator=g).mul_(d ** -0.5).bfloat16(),
             "gain": torch.rand(E, device="cuda", generator=g) + 0.5, "bias": torch.full((E,), 0.8 * i - 1, device="cuda")}
        dws.append(B.DeviceWeights(B.make_weights(t["W_r"], t["gain"], t["bias"], t["U"], t["D"]), t))
        s = torch.rand(L, E, device="cuda", generator=g) * (torch.rand(1, E, device="cuda", generator=g) < 0.2 + 0.3 * i)
        e = (s != 0).any(0).nonzero().flatten().int()
        scores.append(s)
        ids.append(torch.cat([e, e.new_full((E - len(e),), -1)]))
        nu.append(torch.full((1,), len(e), dtype=torch.int32, device="cuda"))
    layer, cfg = B.Layer(d, E, d_e, L_max=L, variant=B.VARIANT_SIMT), B.Config(d, E, d_e, L, 1e-6, 0, 0)
    start = torch.randn(L, d, device="cuda", generator=g)
    h, x, outs = start.clone(), torch.zeros(2, L, d, dtype=torch.bfloat16, device="cuda"), torch.zeros(n, L, d, device="cuda")
    xs = torch.randn(n, L, d, device="cuda", generator=g).bfloat16()
    dep = B.CALL_ACCUMULATE | B.CALL_INDEPENDENT

    def run(pause=lambda: None):
        h.copy_(start)
        x[0].copy_(start)
        for i in range(n):
            w, s, a, b = dws[i % 3].struct, scores[i % 3], x[i % 2], x[(i + 1) % 2]
            if kind == "router":
                B.blockffn_layer_forward(layer.h, w, a, L, h, b, None, dep)
            elif kind == "scores":
                B.blockffn_layer_forward_scores(layer.h, w, a, s, L, h, b, None, dep)
            elif kind == "independent":
                B.blockffn_layer_forward_scores(layer.h, w, xs[i], s, L, outs[i], None, None, B.CALL_INDEPENDENT_X)
            else:
                B.blockffn_expert_ffn_noalloc(cfg, w, a, s, L, ids[i % 3], nu[i % 3], h, b, dep if i % 4 else B.CALL_ACCUMULATE)
            pause()
    run(torch.cuda.synchronize)
    want = [b.clone() for b in (h, x, outs)]
    assert all(bool(torch.isfinite(b).all() and b.any()) for b in (want[2:] if kind == "independent" else want[:2]))
    graph = torch.cuda.CUDAGraph()
    for k in range(4):
        outs.zero_()
        if k == 2:
            with torch.cuda.graph(graph):
                run()
        graph.replay() if k >= 2 else run()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip((h, x, outs), want))
    assert layer.last_status() == 0
