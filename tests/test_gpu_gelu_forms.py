"""GeLU and its derivative in the epilogues: values that are not numbers, and the fp32 forms far from zero."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


def _layer(n, d, dff, E, dtype, gelu, b1):
    """Forward and backward with the given hidden biases: the saved tensors, the backward's intermediates, dW1, dW2, db1, W2."""
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
    return B.saved_view(cfg, saved), B.backward_view(cfg, ws), dW1, dW2, bias_grads[0], W2


# rows per expert and widths of: multiply-adds, three bf16 pieces, 128-row tiles, tiles of CTA pairs, turned tiles
@pytest.mark.parametrize("dtype,k,d,dff,E", [(torch.float32, 8, 64, 128, 4), (torch.float32, 260, 316, 1028, 8), (torch.bfloat16, 128, 64, 264, 4),
                                             (torch.bfloat16, 520, 256, 1032, 4), (torch.bfloat16, 40, 64, 264, 4)])
@pytest.mark.parametrize("gelu", ["erf", "tanh"])
def test_nan_before_the_gelu_reaches_the_gradients(dtype, k, d, dff, E, gelu):
    """One hidden unit of one expert is NaN: its column of the weight gradients is, and no other hidden unit's."""
    b1 = torch.zeros(E, dff, dtype=dtype, device="cuda")
    b1[1, dff - 3] = float("nan")
    _, _, dW1, dW2, db1, _ = _layer(k * E, d, dff, E, dtype, gelu, b1)
    want = torch.zeros(E, dff, dtype=torch.bool, device="cuda")
    want[1, dff - 3] = True
    assert torch.equal(torch.isnan(db1), want)
    assert torch.equal(torch.isnan(dW1), want[:, None].expand(E, d, dff))
    assert torch.equal(torch.isnan(dW2), want[:, None].expand(E, d, dff))


@pytest.mark.parametrize("k,d,dff,E", [(8, 64, 128, 4), (260, 316, 1028, 8)])        # multiply-adds, three bf16 pieces
@pytest.mark.parametrize("gelu", ["erf", "tanh"])
def test_fp32_gelu_far_from_zero(k, d, dff, E, gelu):
    """Pre-activations from -100 to 100, by way of the biases, against 64 bits; where the function has run into its ends they are exact."""
    b1 = torch.linspace(-100, 100, E * dff, device="cuda").reshape(E, dff)
    saved, back, _, _, _, W2 = _layer(k * E, d, dff, E, torch.float32, gelu, b1)
    Z, H = saved["Z"].double().requires_grad_(), saved["H"].double()
    want = torch.nn.functional.gelu(Z, approximate="tanh" if gelu == "tanh" else "none")
    slope = torch.autograd.grad(want.sum(), Z)[0]
    Z, want = Z.detach(), want.detach()
    # erff and tanhf are within 2 units of 2^-24, their argument within three more roundings whose effect on them is below one unit,
    # one rounding of 1 + erf and one of the product: in units of 2^-24, half of (2 + 1 + 2) on the gate and 1 of the result
    assert ((H - want).abs() <= 2.0 ** -24 * (2.5 * Z.abs() + want.abs())).all()
    far = Z.abs() > 9
    assert torch.equal(H[far], Z[far].clamp(min=0))
    acc = back["dX_e"].double() @ W2.double()
    # the derivative adds z times the density to the gate: its exponent z^2 / 2 carries three roundings, z^3 phi(z) / 2 < 0.24 of them.
    # The tanh form's 1 - th^2 carries twice th's five units, times z u'(z) / 2.  The product: 17 + K / 64 units as in
    # test_gpu_f32_tensor, of the sum of its sizes
    gate = 6 + (5 * 0.7979 * Z.abs() * (1 + 3 * 0.044715 * Z ** 2) * ~far if gelu == "tanh" else 0)
    size = back["dX_e"].double().abs() @ W2.double().abs()
    units = 20 + (d + 63) // 64
    assert ((back["dZ"].double() - acc * slope).abs() <= 2.0 ** -24 * (gate * acc.abs() + units * size * slope.abs())).all()
    assert torch.all(back["dZ"].double()[Z < -9].abs() <= 1e-12 * acc[Z < -9].abs() + 1e-30)
