"""GeLU and its derivative in the epilogues: values that are not numbers."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


def _layer(n, d, dff, E, dtype, gelu, b1):
    """Forward and backward with the given hidden biases; (Y, saved view, dW1, dW2, db1)."""
    cfg = B.make_config(n, d, dff, E, 1.0, dtype, gelu=gelu)
    gen = torch.Generator(device="cuda").manual_seed(n)

    def normal(scale, *shape):
        return (torch.empty(shape, device="cuda").normal_(generator=gen) * scale).to(dtype)

    X, Wg, W1, W2, dY = normal(1, n, d), normal(d ** -0.5, d, E), normal(d ** -0.5, E, d, dff), normal(dff ** -0.5, E, d, dff), normal(1, n, d)
    b2, ws = torch.zeros(E, d, dtype=dtype, device="cuda"), B.alloc_workspace(cfg)
    Y, saved = B.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws, b1=b1, b2=b2)
    bias_grads = (torch.empty_like(b1), torch.empty_like(b2))
    _, _, dW1, dW2 = B.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, None, ws, bias_grads)
    assert B.ec_read_status(ws) == B.EC_OK
    return Y, B.saved_view(cfg, saved), dW1, dW2, bias_grads[0]


# rows per expert and widths of: multiply-adds, three bf16 pieces, 128-row tiles, tiles of CTA pairs, turned tiles
@pytest.mark.parametrize("dtype,k,d,dff,E", [(torch.float32, 8, 64, 128, 4), (torch.float32, 260, 316, 1028, 8), (torch.bfloat16, 128, 64, 264, 4),
                                             (torch.bfloat16, 520, 256, 1032, 4), (torch.bfloat16, 40, 64, 264, 4)])
@pytest.mark.parametrize("gelu", ["erf", "tanh"])
def test_nan_before_the_gelu_reaches_the_gradients(dtype, k, d, dff, E, gelu):
    """One hidden unit of one expert is NaN: its column of the weight gradients is, and no other hidden unit's."""
    b1 = torch.zeros(E, dff, dtype=dtype, device="cuda")
    b1[1, dff - 3] = float("nan")
    _, _, dW1, dW2, db1 = _layer(k * E, d, dff, E, dtype, gelu, b1)
    want = torch.zeros(E, dff, dtype=torch.bool, device="cuda")
    want[1, dff - 3] = True
    assert torch.equal(torch.isnan(db1), want)
    assert torch.equal(torch.isnan(dW1), want[:, None].expand(E, d, dff))
    assert torch.equal(torch.isnan(dW2), want[:, None].expand(E, d, dff))
