"""The fp32 expert products at the edges of the FMA kernel's tiles, against the same products in 64 bits."""
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
