"""The selection at the edges of its sort and its scans (keys per thread, keys per warp, one key, all tokens, beyond one tile),
with distinct and with heavily tied scores, against a stable sort of the same scores."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [0, 3])
@pytest.mark.parametrize("n,E,k,groups", [(64, 4, 1, 1), (40, 4, 31, 2), (64, 4, 33, 1), (128, 4, 128, 1), (300, 8, 65, 3), (513, 4, 257, 1),
                                          (1000, 8, 129, 1), (2048, 8, 512, 1), (2049, 4, 1025, 1), (4100, 4, 4096, 1), (16384, 4, 2049, 1),
                                          (16384, 8, 4096, 1), (16385, 4, 600, 1), (17000, 4, 4097, 1), (40000, 4, 17000, 1)])
def test_selection_is_a_stable_sort(n, E, k, groups, levels):
    cfg = B.make_config(n, E, 8, E, (k + 0.25) * E / n, torch.float32, groups=groups)
    assert B.ec_capacity(cfg) == k
    gen = torch.Generator(device="cuda").manual_seed(n + k)
    X = torch.empty(groups * n, E, device="cuda").normal_(generator=gen)
    if levels:
        X = (X * levels).round().clamp(-levels, levels) / levels       # few distinct rows: equal scores everywhere
    r = B.ec_route(cfg, X, torch.eye(E, device="cuda"))
    for g in range(groups):
        S = r.S[g * n:(g + 1) * n]
        want = torch.sort(S, dim=0, descending=True, stable=True)[1][:k].T + g * n
        got = r.I[:, g * k:(g + 1) * k].long()
        assert torch.equal(got, want)
        assert torch.equal(r.G[:, g * k:(g + 1) * k], torch.gather(r.S.T, 1, got))


# rows of NaN: fewer than k, more than k, more than the final sort chooses from, all
@pytest.mark.parametrize("n,k,groups,nans", [(2048, 16, 1, 300), (2048, 512, 1, 100), (16384, 40, 1, 16384), (1000, 100, 3, 700), (20000, 300, 1, 100),
                                             (20000, 300, 1, 400), (20000, 300, 2, 9000), (20000, 5000, 1, 20000)])
def test_rows_that_are_not_numbers_leave_the_selection_whole(n, k, groups, nans):
    """A model that has diverged hands in rows of NaN.  They count as the largest scores, so an expert still takes k tokens of its
    group, NaN rows first (the lower tokens of them), then the best of the others."""
    E = 4
    cfg = B.make_config(n, E, 8, E, (k + 0.25) * E / n, torch.float32, groups=groups)
    assert B.ec_capacity(cfg) == k
    gen = torch.Generator(device="cuda").manual_seed(n + k + nans)
    X = torch.empty(groups * n, E, device="cuda").normal_(generator=gen)
    for g in range(groups):
        X[g * n + torch.randperm(n, generator=gen, device="cuda")[:nans]] = float("nan")
    r = B.ec_route(cfg, X, torch.eye(E, device="cuda"))
    assert torch.equal(r.S.isnan().all(dim=1), X.isnan().any(dim=1))
    for g in range(groups):
        S = r.S[g * n:(g + 1) * n]
        want = torch.sort(S.nan_to_num(nan=2.0), dim=0, descending=True, stable=True)[1][:k].T + g * n
        assert torch.equal(r.I[:, g * k:(g + 1) * k].long(), want)
    got = torch.gather(r.S.T, 1, r.I.long())
    assert torch.equal(r.G.view(torch.int32), got.view(torch.int32))
    assert B.ec_validate_routing(cfg, r.I, r.row_ptr, r.slots) == 0


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n,d,E,c", [(130, 8, 4, 2.0), (777, 40, 3, 1.0), (3000, 296, 16, 2.0), (9000, 600, 64, 1.5), (2048, 1032, 8, 2.0)])
def test_shuffle_and_unshuffle_at_odd_widths(n, d, E, c, dtype):
    """Rows of 1 to 258 pieces: the shuffle copies bits, the unshuffle adds at most a few slots' rows per token in fp32."""
    cfg = B.make_config(n, d, 8, E, c, dtype)
    gen = torch.Generator(device="cuda").manual_seed(n + d)
    X = torch.empty(n, d, dtype=dtype, device="cuda").normal_(generator=gen)
    Wg = (torch.empty(d, E, device="cuda").normal_(generator=gen) / d ** 0.5).to(dtype)
    r = B.ec_route(cfg, X, Wg)
    assert torch.equal(B.ec_shuffle(cfg, X, r.I), X[r.I.long()])
    k = B.slots_per_expert(cfg)
    X_e = torch.empty(E, k, d, device="cuda").normal_(generator=gen)
    Y = B.ec_unshuffle(cfg, X_e, r.G, r.row_ptr, r.slots).double()
    terms = r.G.double()[..., None] * X_e.double()
    want = torch.zeros(n, d, dtype=torch.float64, device="cuda").index_add_(0, r.I.flatten().long(), terms.flatten(0, 1))
    size = torch.zeros_like(want).index_add_(0, r.I.flatten().long(), terms.abs().flatten(0, 1))
    # at most E products and sums in fp32, then one rounding to the output's type
    bound = (E + 1) * 2.0 ** -24 * size + (2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -24) * want.abs()
    assert ((Y - want).abs() <= bound + 1e-30).all()
