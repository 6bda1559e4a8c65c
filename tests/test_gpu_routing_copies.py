"""blockffn_read_routing into buffers that are not the handle's device's own: copies, as a kernel may
not be able to reach them (another GPU's memory without peer access; here pinned host memory, which
either way could reach)."""
import pytest
import torch

from paper_2507_08771_b200 import binding as B
from test_gpu_chain import make

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [5, 64, 130])
def test_buffers_elsewhere_are_copied_to(E):
    d, L = 256, 9
    layer, dw = B.Layer(d, E, 64, L_max=L), make(d, E, 64, 4, -0.3)
    x = torch.randn(L, d, device="cuda").bfloat16()
    want = layer.forward(dw, x)
    shapes = [((L, E), torch.float32), ((L, layer.words), torch.int32), ((layer.words,), torch.int32),
              ((E,), torch.int32), ((1,), torch.int32)]
    for where in range(2 ** len(shapes)):      # bit k: buffer k is pinned host memory
        bufs = [torch.zeros(s, dtype=t).pin_memory() if where >> k & 1 else torch.zeros(s, dtype=t, device="cuda")
                for k, (s, t) in enumerate(shapes)]
        torch.cuda.synchronize()
        n = layer.launch_count()
        B.blockffn_read_routing(layer.h, L, *[b.data_ptr() for b in bufs])
        torch.cuda.synchronize()
        assert layer.launch_count() - n == (1 if where == 0 else 0)
        for b, w in zip(bufs, (want.scores, want.tok_mask, want.union_mask, want.union_ids, want.n_union)):
            assert torch.equal(b.cuda(), w)
