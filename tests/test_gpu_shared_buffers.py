"""Gradients written over operands that the backward pass has read by then: the bits are those of separate buffers."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B
from paper_2202_09368_b200 import inputs as IN

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


@pytest.mark.parametrize("dtype,n,d,dff,E,kw", [(BF16, 2048, 256, 512, 8, {}), (BF16, 4096, 768, 3072, 32, {}), (BF16, 600, 200, 600, 10, dict(fuse_gather=True)),
                                                (BF16, 1024, 256, 512, 64, {}), (F32, 2048, 256, 1024, 8, {}), (F32, 300, 36, 100, 3, {})])
def test_gradients_may_take_the_place_of_operands(dtype, n, d, dff, E, kw):
    """Products of one tile and of many, turned ones (32 rows per expert) and the multiply-add kernels."""
    cfg = B.make_config(n, d, dff, E, 2.0, dtype, **kw)
    li = IN.make_layer_inputs(n, d, dff, E, dtype, seed=n)
    X, Wg, W1, W2, dY = (t.cuda() for t in (li.X, li.Wg, li.W1, li.W2, li.dX_out))
    ws = B.alloc_workspace(cfg)
    _, saved = B.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws)
    want = B.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, ws=ws)
    for over_dx_out in (False, True):
        for _ in range(3):
            x, w2, dy = X.clone(), W2.clone(), dY.clone()
            got = B.ec_moe_backward(cfg, x, Wg, W1, w2, dy, saved, (dy if over_dx_out else x, torch.empty_like(Wg), torch.empty_like(W1), w2), ws)
            assert all(torch.equal(a, b) for a, b in zip(got, want))
