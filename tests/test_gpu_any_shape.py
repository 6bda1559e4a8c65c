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
        # the same call with the list given, an entry out of range among its entries
        lst = np.full(E, -1, np.int32)
        lst[:len(ids)] = ids
        idd = torch.from_numpy(lst).cuda()
        nd = torch.tensor([len(ids)], dtype=torch.int32, device="cuda")
        out2 = torch.full((L, d), float("nan"), device="cuda")
        torch.cuda.synchronize()
        B.blockffn_expert_ffn(layer.h, dw.struct, xd, sd, L, idd, nd, out2, call_flags=flags)
        torch.cuda.synchronize()
        assert np.abs(out2.double().cpu().numpy() - ref).max() <= TOL * max(rms, 1e-30)
    assert layer.last_status() == 0


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
