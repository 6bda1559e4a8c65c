"""Which calls run as one kernel, whose CTAs all have to be resident at once, and which do not."""
import pytest
import torch

from paper_2507_08771_b200 import binding as B
from test_gpu_chain import make

pytestmark = pytest.mark.gpu


def launches(layer, call):
    n = layer.launch_count()
    call()
    torch.cuda.synchronize()
    assert layer.last_status() == 0
    return layer.launch_count() - n


@pytest.mark.parametrize("L", [1, 8, 9, 16, 17, 32])
def test_calls_without_a_promise_need_no_resident_grid(L):
    """Scores or a list given and nothing promised: kernels that follow one another. With the promise
    a chunk of more than 8 tokens is one kernel."""
    d, E, d_e = 512, 24, 64
    dw, layer = make(d, E, d_e, 1, 0.0), B.Layer(d, E, d_e, L_max=L)
    x, scores = torch.randn(L, d, device="cuda").bfloat16(), torch.rand(L, E, device="cuda")
    ids, n = torch.arange(E, device="cuda", dtype=torch.int32), torch.full((1,), E, device="cuda", dtype=torch.int32)
    z = torch.einsum("ejd,td->tej", dw.tensors["U"].double(), x.double())
    ref = torch.einsum("tej,ecj->tc", scores.double()[:, :, None] * z * torch.sigmoid(z), dw.tensors["D"].double())
    for flags, want in ((0, 2), (B.CALL_INDEPENDENT, 1 if L > 8 else 2)):
        for call in (lambda out: B.blockffn_layer_forward_scores(layer.h, dw.struct, x, scores, L, out, call_flags=flags),
                     lambda out: B.blockffn_expert_ffn(layer.h, dw.struct, x, scores, L, ids, n, out, call_flags=flags)):
            out = torch.zeros(L, d, device="cuda")
            torch.cuda.synchronize()
            assert launches(layer, lambda: call(out)) == want
            assert (out.double() - ref).abs().max() <= 2e-2 * ref.square().mean().sqrt()
