"""The native argument unpacking: what is not plain goes through ctypes, which accepts or refuses."""
import ctypes
import sys
import types

import pytest
import torch

from paper_2507_08771_b200 import binding as B


def test_what_is_not_plain_is_left_to_ctypes():
    fast = B._load_fast()
    h, w, t = ctypes.c_void_p(0), B.make_weights(), torch.zeros(8)
    plain = [h, w, None, 1, None, None, None, 0, None]
    for i, odd in [(0, 0), (0, None), (1, None), (1, h), (2, t), (2, 64), (2, t[::2]), (3, 1.0), (3, True),
                   (3, 1 << 40), (4, torch.nn.Parameter(t)), (7, None), (8, 0)]:
        args = list(plain)
        args[i] = odd
        assert fast.layer_forward(*args) is NotImplemented, (i, odd)
    with pytest.raises(TypeError):
        fast.layer_forward(h)


def test_a_layer_call_that_is_not_plain_is_left_to_its_parts():
    fast = B._load_fast()
    h, w, t = ctypes.c_void_p(0), B.make_weights(), torch.zeros(8)
    plain = [h, w, t, None, None, 0, 8, 4, 1, 1 << 6]      # (a tensor that is not on a GPU, a device that does not exist)
    for i, odd in [(0, None), (1, None), (2, None), (2, 64), (2, t), (3, t), (5, None), (6, 1.0), (9, None)]:
        args = list(plain)
        args[i] = odd
        assert fast.layer_call(*args) is NotImplemented, (i, odd)
    with pytest.raises(TypeError):
        fast.layer_call(h)


def test_buffers_that_cannot_be_allocated_leave_nothing_behind():
    fast = B._load_fast()
    args = (1 << 30, 1 << 30, 1 << 30, 0, 1 << 6)      # a device that does not exist
    for _ in range(3):
        assert fast.routing_buffers(*args) is NotImplemented
    before = sys.getallocatedblocks()
    for _ in range(1000):
        fast.routing_buffers(*args)
    assert sys.getallocatedblocks() - before < 500     # (1000 where each call loses its tuple)


@pytest.mark.parametrize("module", [None, types.SimpleNamespace(TORCH_VERSION="1.0.0")])
def test_without_a_module_for_this_torch_every_call_goes_through_ctypes(monkeypatch, module):
    monkeypatch.setitem(sys.modules, B.__package__ + "._fastcall", module)
    monkeypatch.setattr(B, "_fast", None)
    with pytest.warns(UserWarning, match="ctypes"):
        with pytest.raises(B.BlockFFNError) as e:       # the library's own answer to a NULL handle
            B.blockffn_router(ctypes.c_void_p(0), B.make_weights(), None, 1, None, stream=0)
    assert e.value.code == B.ERR_INVALID_ARG
    for call in (lambda: B.blockffn_chunk_union(None, None, 1, None, None, None, stream=0),
                 lambda: B.blockffn_expert_ffn(None, B.make_weights(), None, None, 1, None, None, None, stream=0),
                 lambda: B.blockffn_expert_ffn_noalloc(B.Config(), B.make_weights(), None, None, 1, None, None, None, stream=0),
                 lambda: B.blockffn_layer_forward(None, B.make_weights(), None, 1, None, stream=0),
                 lambda: B.blockffn_layer_forward_scores(None, B.make_weights(), None, None, 1, None, stream=0),
                 lambda: B.blockffn_read_routing(None, 1, stream=0),
                 lambda: B.blockffn_reuse_ratio(None, None, 1, None, stream=0)):
        with pytest.raises(B.BlockFFNError) as e:
            call()
        assert e.value.code == B.ERR_INVALID_ARG


@pytest.mark.gpu
def test_a_layer_without_the_module(monkeypatch):
    layer, x = B.Layer(256, 40, 64, L_max=5), torch.randn(5, 256, device="cuda").bfloat16()
    t = {"W_r": torch.randn(40, 256, device="cuda").bfloat16(), "gain": torch.ones(40, device="cuda"),
         "U": torch.randn(40, 64, 256, device="cuda").bfloat16(), "D": torch.randn(40, 256, 64, device="cuda").bfloat16()}
    dw = B.DeviceWeights(B.make_weights(t["W_r"], t["gain"], None, t["U"], t["D"]), t)
    want = layer.forward(dw, x)
    monkeypatch.setitem(sys.modules, B.__package__ + "._fastcall", None)
    monkeypatch.setattr(B, "_fast", None)
    with pytest.warns(UserWarning, match="ctypes"):
        got = layer.forward(dw, x)
    assert all(torch.equal(a, b) for a, b in zip(vars(want).values(), vars(got).values()))


@pytest.mark.gpu
def test_both_ways_give_the_same():
    d, E, L = 256, 40, 5
    layer = B.Layer(d, E, 64, L_max=L)
    x = torch.randn(L, d, device="cuda").bfloat16()
    W_r = torch.randn(E, d, device="cuda").bfloat16()
    gain = torch.ones(E, device="cuda")
    w = B.make_weights(W_r, gain)
    want, got = torch.zeros(L, E, device="cuda"), torch.zeros(L, E, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    B.blockffn_router(layer.h, w, x.data_ptr(), L, want.data_ptr(), stream=side)     # ctypes
    side.synchronize()
    with torch.cuda.stream(side):
        B.blockffn_router(layer.h, w, x, L, got)                                     # native, its stream
    side.synchronize()
    assert torch.equal(want, got) and bool((got > 0).any())
    with pytest.raises(AssertionError):
        B.blockffn_router(layer.h, w, x.t(), L, got)
    with pytest.raises(AssertionError):        # a CPU tensor
        B.blockffn_router(layer.h, w, x.cpu(), L, got)
    with pytest.raises(B.BlockFFNError) as e:  # a handle that is NULL
        B.blockffn_router(ctypes.c_void_p(0), w, x, L, got)
    assert e.value.code == B.ERR_INVALID_ARG
    bufs = layer._routing(L, True)
    assert [tuple(b.shape) for b in bufs] == [(L, E), (L, 2), (2,), (E,), (1,)]
    assert [b.dtype for b in bufs] == [torch.float32] + 4 * [torch.int32]
    assert [b is None for b in layer._routing(L, False)] == [True, True, False, False, False]


@pytest.mark.gpu
def test_a_layer_call_at_once_is_the_call_in_its_parts():
    layer = B.Layer(256, 16, 64, L_max=8)
    g = torch.Generator(device="cuda").manual_seed(1)
    t = {"W_r": (256 ** -0.5 * torch.randn(16, 256, device="cuda", generator=g)).bfloat16(), "gain": torch.ones(16, device="cuda"),
         "U": torch.randn(16, 64, 256, device="cuda", generator=g).bfloat16(),
         "D": torch.randn(16, 256, 64, device="cuda", generator=g).bfloat16()}
    dw = B.DeviceWeights(B.make_weights(t["W_r"], t["gain"], None, t["U"], t["D"]), t)
    for L in (1, 5, 8):
        x, nxt = torch.randn(L, 256, device="cuda", generator=g).bfloat16(), [torch.empty(L, 256, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        a = layer.forward(dw, x, x_next=nxt[0])
        b = layer.forward(dw, x, out=torch.empty(L, 256, device="cuda"), x_next=nxt[1])
        for u, v in zip((a.out, a.scores, a.tok_mask, a.union_mask, a.n_union, nxt[0]), (b.out, b.scores, b.tok_mask, b.union_mask, b.n_union, nxt[1])):
            assert u.shape == v.shape and u.dtype == v.dtype and torch.equal(u, v)
        assert torch.equal(a.union_ids, b.union_ids)
    with pytest.raises(B.BlockFFNError) as e:
        layer.forward(dw, torch.zeros(9, 256, dtype=torch.bfloat16, device="cuda"))       # more than L_max
    assert e.value.code == B.ERR_INVALID_ARG and "blockffn_layer_forward" in str(e.value)
