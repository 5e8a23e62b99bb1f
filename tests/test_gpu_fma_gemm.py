"""The FMA kernels at the edges of their tiles, against the same arithmetic in 64 bits: the fp32 expert products, the gate gradients
and products of very wide layers, the gate."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


# (k, d, d', E): sizes that take the 128 x 128 tile (with and without the shared contraction), the 64 x 64 and the 64 x 32
# tile, one short of, at and beyond whole tiles and k-tiles in every dimension, down to a single row and one k-tile
@pytest.mark.parametrize("k,d,dff,E", [(260, 260, 1028, 16), (256, 508, 2052, 16), (127, 132, 516, 12), (129, 64, 124, 5), (65, 36, 60, 3),
                                       (1, 4, 4, 2), (31, 16, 32, 4), (300, 768, 1100, 2)])
def test_fp32_products_match_64_bits(k, d, dff, E):
    n = k * E                                           # c = 1: k = n / E
    cfg = B.make_config(n, d, dff, E, 1.0, torch.float32)
    assert B.ec_capacity(cfg) == k
    gen = torch.Generator(device="cuda").manual_seed(k + d)

    def normal(*shape):
        return torch.empty(shape, device="cuda").normal_(generator=gen)

    for kind, A, Bm, terms in ((B.EC_GEMM_XW1, normal(E, k, d), normal(E, d, dff), d), (B.EC_GEMM_HW2T, normal(E, k, dff), normal(E, d, dff), dff),
                               (B.EC_GEMM_ATB, normal(E, k, d), normal(E, k, dff), k)):
        C = B.ec_expert_gemm(cfg, kind, A, Bm)
        a = A.double().transpose(1, 2) if kind == B.EC_GEMM_ATB else A.double()
        b = Bm.double().transpose(1, 2) if kind == B.EC_GEMM_HW2T else Bm.double()
        # a chain of `terms` fused multiply-adds in fp32: at most terms * 2^-24 of the sum of the terms' sizes
        bound = (terms + 1) * 2.0 ** -24 * (a.abs() @ b.abs())
        assert ((C.double() - a @ b).abs() <= bound).all(), kind


@pytest.mark.parametrize("dtype,E", [(torch.float32, 2), (torch.float32, 4), (torch.bfloat16, 2)])
def test_rows_wider_than_one_grid_of_column_tiles(dtype, E):
    """d = 2^21 + 8: 65537 column tiles of 32, more than a grid has places for: dX = dL . Wg^T + slot rows takes wider ones, with the
    number of experts a multiple of four (fp32) or not, and so do GEMM-2 and dX_in."""
    n, d, dff = 8, (1 << 21) + 8, 8
    cfg = B.make_config(n, d, dff, E, 1.0, dtype)
    gen = torch.Generator(device="cuda").manual_seed(E)

    def normal(scale, *shape):
        return (torch.empty(shape, device="cuda").normal_(generator=gen) * scale).to(dtype)

    X, Wg, W1, W2, dY = normal(1, n, d), normal(d ** -0.5, d, E), normal(d ** -0.5, E, d, dff), normal(dff ** -0.5, E, d, dff), normal(1, n, d)
    ws = B.alloc_workspace(cfg)
    Y, saved = B.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws)
    v = {name: t.clone() for name, t in B.saved_view(cfg, saved).items()}
    dX = B.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, ws=ws)[0]
    assert B.ec_read_status(ws) == B.EC_OK
    w = B.backward_view(cfg, ws)
    eps = 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -8          # of one rounding to the result's type; the sums are fp32

    def check(got, a, b, rows=None):
        want, size = a.double() @ b.double(), a.double().abs() @ b.double().abs()
        if rows is not None:                            # each token's slot rows, and the sizes of what is added up
            want.index_add_(0, v["I"].flatten().long(), rows.double().flatten(0, 1))
            size.index_add_(0, v["I"].flatten().long(), rows.double().abs().flatten(0, 1))
        bound = (a.shape[-1] + E + 1) * 2.0 ** -24 * size + eps * want.abs() + 1e-30
        assert ((got.double() - want).abs() <= bound).all()

    check(v["X_e"], v["H"], W2.transpose(1, 2))
    check(w["dX_in"], w["dZ"], W1.transpose(1, 2))
    check(dX, w["dL"], Wg.T, w["dX_in"])


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,d,E", [(33, 136, 36), (100, 1000, 60), (65, 72, 33), (31, 264, 70), (200, 520, 100), (64, 8, 130), (40, 640, 132), (97, 200, 253),
                                   (500, 40, 252), (32, 128, 30)])
def test_gate_widths_of_the_fma_kernel(n, d, E, dtype):
    """Expert counts the tensor-core gate does not take (no multiple of eight) from one to eight column groups, in whole groups of
    four and not, tokens and depths that end inside a chunk: against the softmax in 64 bits."""
    cfg = B.make_config(n, d, 8, E, 4.0 * E / n, dtype)
    gen = torch.Generator(device="cuda").manual_seed(n + E)
    X = torch.empty(n, d, device="cuda").normal_(generator=gen).to(dtype)
    Wg = (torch.empty(d, E, device="cuda").normal_(generator=gen) / d ** 0.5).to(dtype)
    r = B.ec_route(cfg, X, Wg)
    want = torch.softmax(X.double() @ Wg.double(), dim=1)
    # a logit is off by at most d * 2^-24 of the sum of its terms' sizes, twice that (with the largest one) in the exponent; expf, the
    # sum and the quotient add at most (E + 8) roundings
    logit = d * 2.0 ** -24 * (X.double().abs() @ Wg.double().abs()).amax(dim=1, keepdim=True)
    assert ((r.S.double() - want).abs() <= (2 * logit + (E + 8) * 2.0 ** -23) * want).all()
    assert B.ec_validate_routing(cfg, r.I, r.row_ptr, r.slots) == 0
