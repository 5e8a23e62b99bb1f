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
