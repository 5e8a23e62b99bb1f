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


def _three_products(cfg, k, d, dff, E, make):
    """The three kinds with operands made by make(kind, which, shape): (result, A as it multiplies, B as it multiplies) in 64 bits."""
    for kind, sa, sb in ((B.EC_GEMM_XW1, (E, k, d), (E, d, dff)), (B.EC_GEMM_HW2T, (E, k, dff), (E, d, dff)), (B.EC_GEMM_ATB, (E, k, d), (E, k, dff))):
        A, Bm = make(kind, 0, sa), make(kind, 1, sb)
        out = B.ec_expert_gemm(cfg, kind, A, Bm)
        yield out.double(), A.double().transpose(1, 2) if kind == B.EC_GEMM_ATB else A.double(), Bm.double().transpose(1, 2) if kind == B.EC_GEMM_HW2T else Bm.double()


# operands of 2^a and 2^b: subnormal numbers, products near both ends of the range and beyond the middle of it
@pytest.mark.parametrize("a,b", [(-120, 10), (10, -120), (-140, 100), (100, -100), (-60, -60), (60, 60), (120, -10)])
def test_products_over_the_range_of_fp32(a, b):
    k, d, dff, E = 260, 316, 1028, 8
    cfg = B.make_config(k * E, d, dff, E, 1.0, torch.float32)
    gen = torch.Generator(device="cuda").manual_seed(a + 1000)
    for out, A, Bm in _three_products(cfg, k, d, dff, E, lambda kind, which, shape: torch.ldexp(torch.empty(shape, device="cuda").normal_(generator=gen),
                                                                                              torch.tensor(b if which else a, device="cuda"))):
        terms = A.shape[2]
        # as above; elements taken by multiply-adds have a rounding per term instead, and results below 2^-126 one of 2^-149 on top
        units = 16 + 20 * 4 / 256 + (terms + 63) // 64 + 0.75 if a + b < 100 else terms
        assert ((out - A @ Bm).abs() <= units * 2.0 ** -24 * (A.abs() @ Bm.abs()) + 2.0 ** -148).all()


def test_infinities_huge_values_and_nan_stay_in_their_rows_and_columns():
    """One infinity, one finite value that bf16 would round to infinity, one overflowing pair and one NaN: what 64 bits say they make
    of their rows and columns, and nothing elsewhere."""
    k, d, dff, E = 260, 316, 1028, 8
    cfg = B.make_config(k * E, d, dff, E, 1.0, torch.float32)
    gen = torch.Generator(device="cuda").manual_seed(3)

    def make(kind, which, shape):
        t = torch.empty(shape, device="cuda").normal_(generator=gen)
        if which == 0:
            t[0, 5, 7], t[1, 131, 3], t[2, 9, 11], t[3, 200, 100] = float("inf"), 3.396e38, 1e30, float("nan")
        else:
            t[4, 17, 19] = -float("inf")
            t[1] *= 1e-6                               # the huge value's products are finite
            t[2, 3:5, 21:25] = 1e30
            if kind != B.EC_GEMM_HW2T:
                t[2, 11 if kind == B.EC_GEMM_XW1 else 9, 30] = 3e30
        return t

    for out, A, Bm in _three_products(cfg, k, d, dff, E, make):
        want = (A @ Bm).float().double()               # rounded to fp32: sums beyond its range are infinite
        assert torch.equal(torch.isnan(out), torch.isnan(want))
        assert torch.equal(torch.isinf(out), torch.isinf(want)) and torch.equal(out[torch.isinf(out)], want[torch.isinf(want)])
        fine = torch.isfinite(want)
        size = A.abs().nan_to_num(0, 0) @ Bm.abs().nan_to_num(0, 0)
        assert ((out - want).abs()[fine] <= A.shape[2] * 2.0 ** -24 * size[fine]).all()
