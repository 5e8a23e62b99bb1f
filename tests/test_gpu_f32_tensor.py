"""fp32 products on the tensor cores at the edges of their tiles, against the same arithmetic in 64 bits: orientations, epilogues,
bias terms, rows picked through a list."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


# one short of, at and beyond the 128 rows, the 64 or 128 columns and the 64 of a k-block; several tiles a CTA; a last group of four
@pytest.mark.parametrize("k,d,dff,E", [(127, 256, 508, 8), (129, 260, 516, 8), (128, 192, 384, 16), (260, 316, 1028, 16), (44, 700, 1284, 8),
                                       (512, 128, 4096, 8)])
def test_products_match_64_bits(k, d, dff, E):
    cfg = B.make_config(k * E, d, dff, E, 1.0, torch.float32)
    gen = torch.Generator(device="cuda").manual_seed(k + d)

    def normal(*shape):
        return torch.empty(shape, device="cuda").normal_(generator=gen)

    for kind, A, Bm, terms in ((B.EC_GEMM_XW1, normal(E, k, d), normal(E, d, dff), d), (B.EC_GEMM_HW2T, normal(E, k, dff), normal(E, d, dff), dff),
                               (B.EC_GEMM_ATB, normal(E, k, d), normal(E, k, dff), k)):
        out = torch.full((E, k, dff) if kind == B.EC_GEMM_XW1 else (E, k, d) if kind == B.EC_GEMM_HW2T else (E, d, dff), float("nan"), device="cuda")
        B.ec_expert_gemm(cfg, kind, A, Bm, out=out)
        a = A.double().transpose(1, 2) if kind == B.EC_GEMM_ATB else A.double()
        b = Bm.double().transpose(1, 2) if kind == B.EC_GEMM_HW2T else Bm.double()
        # a k-block of 64: four truncations (2^-23 each, twice: the sum of 16 and the accumulator) of large terms, twenty of terms below
        # 2^-8; one rounding of the running sum per k-block; the three dropped terms 2^-26 each.  In units of 2^-24 of the sum of sizes
        units = 16 + 20 * 4 / 256 + (terms + 63) // 64 + 0.75
        assert ((out.double() - a @ b).abs() <= units * 2.0 ** -24 * (a.abs() @ b.abs())).all(), kind


@pytest.mark.parametrize("gelu", ["erf", "tanh"])
@pytest.mark.parametrize("fuse", [False, True])
def test_layer_matches_64_bits(gelu, fuse):
    """Two groups, biases, ragged sizes; with fuse the rows of X come through I in the products."""
    n, d, dff, E, c, groups = 1000, 196, 708, 6, 2.0, 2
    cfg = B.make_config(n, d, dff, E, c, torch.float32, gelu=gelu, groups=groups, fuse_gather=fuse)
    gen = torch.Generator(device="cuda").manual_seed(7)

    def normal(scale, *shape):
        return torch.empty(shape, device="cuda").normal_(generator=gen) * scale

    X, Wg, W1, W2 = normal(1, n * groups, d), normal(d ** -0.5, d, E), normal(d ** -0.5, E, d, dff), normal(dff ** -0.5, E, d, dff)
    b1, b2, dY = normal(0.5, E, dff), normal(0.5, E, d), normal(1, n * groups, d)
    ws = B.alloc_workspace(cfg)
    Y, saved = B.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws, b1=b1, b2=b2)
    v = {name: t.clone() for name, t in B.saved_view(cfg, saved).items() if t is not None}
    only = B.ec_moe_forward(cfg, X, Wg, W1, W2, forward_only=True, b1=b1, b2=b2)[0]
    bias_grads = (torch.empty_like(b1), torch.empty_like(b2))
    dX, dWg, dW1, dW2 = B.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, None, ws, bias_grads)
    assert B.ec_read_status(ws) == B.EC_OK
    assert torch.equal(only, Y)
    p = [t.double().requires_grad_() for t in (X, W1, W2, b1, b2)]
    x, w1, w2, c1, c2 = p
    rows, G = v["I"].long(), v["G"].double().requires_grad_()
    h = torch.nn.functional.gelu(x[rows] @ w1 + c1[:, None], approximate="tanh" if gelu == "tanh" else "none")
    y = h @ w2.transpose(1, 2) + c2[:, None]
    out = torch.zeros_like(x).index_add(0, rows.flatten(), (G[..., None] * y).flatten(0, 1))
    out.backward(dY.double())
    assert torch.allclose(Y.double(), out.detach(), rtol=0, atol=1e-5 * out.detach().pow(2).mean().sqrt().item())
    for got, want in zip((dW1, dW2, *bias_grads), (w1.grad, w2.grad, c1.grad, c2.grad)):
        # sums of at most 1332 terms in fp32: measured 2e-6 of the root mean square at most
        assert (got.double() - want).abs().max() <= 1e-5 * want.pow(2).mean().sqrt()
