"""The backward of the combine where all experts take the same block of tokens (many slots a token, most tokens none): the same numbers
as 64 bits give, and no longer than anywhere."""
import ctypes

import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


def _layer(n, d, E, c, dtype, alike):
    """Forward with all tokens alike (ties go to the lowest: every expert takes the same) or not; what the backward needs."""
    cfg = B.make_config(n, d, 16, E, c, dtype)
    gen = torch.Generator(device="cuda").manual_seed(n + E)

    def normal(scale, *shape):
        return (torch.empty(shape, device="cuda").normal_(generator=gen) * scale).to(dtype)

    X, Wg, W1, W2, dY = normal(1, n, d), normal(d ** -0.5, d, E), normal(d ** -0.5, E, d, 16), normal(0.25, E, d, 16), normal(1, n, d)
    if alike:
        X[:] = X[0]
    ws = B.alloc_workspace(cfg)
    _, saved = B.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws)
    return cfg, (X, Wg, W1, W2, dY), saved, ws


# 9 slots a token (one more than a warp takes alone), 40 (more than a warp has lanes), 64; fp32; an expert count without tensor cores
@pytest.mark.parametrize("n,d,E,c,dtype", [(900, 64, 9, 1.0, torch.float32), (4000, 136, 40, 2.0, torch.bfloat16), (9000, 64, 64, 0.5, torch.bfloat16),
                                           (1000, 264, 33, 2.0, torch.bfloat16)])
def test_crowded_tokens_match_64_bits(n, d, E, c, dtype):
    cfg, args, saved, ws = _layer(n, d, E, c, dtype, True)
    v = {k: t.clone() for k, t in B.saved_view(cfg, saved).items() if t is not None}
    assert int((v["row_ptr"][1:] - v["row_ptr"][:-1]).max()) == E
    B.ec_moe_backward(cfg, *args, saved, ws=ws)
    assert B.ec_read_status(ws) == B.EC_OK
    back = B.backward_view(cfg, ws)
    I, G, S, X_e = v["I"].long(), v["G"].double(), v["S"].double(), v["X_e"].double()
    dy = args[4].double()[I]
    eps = 2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -24
    assert ((back["dX_e"].double() - G[..., None] * dy).abs() <= 1.01 * eps * (G[..., None] * dy).abs()).all()
    size = (dy * X_e).abs().sum(2)                     # a sum of d products in fp32
    assert ((back["dG"].double() - (dy * X_e).sum(2)).abs() <= d * 2.0 ** -24 * size).all()
    dS = torch.zeros_like(S)
    dS[I, torch.arange(E, device="cuda")[:, None].expand_as(I)] = back["dG"].double()
    dot, total = (dS * S).sum(1, keepdim=True), (dS * S).abs().sum(1, keepdim=True)
    want = S * (dS - dot)
    bits = 2.0 ** -8 if back["dL"].dtype == torch.bfloat16 else 2.0 ** -23
    assert ((back["dL"].double() - want).abs() <= bits * want.abs() + S * (E + 2) * 2.0 ** -24 * (dS.abs() + total)).all()


@pytest.mark.parametrize("n,d,E", [(16384, 1024, 64), (16384, 4096, 64)])
def test_crowded_tokens_take_no_longer(n, d, E):
    """The first stage of the backward, by the library's own clock: a warp per token takes twice as long with 64 slots a token."""
    took, L = [], B.lib()
    for alike in (False, True):
        cfg, args, saved, ws = _layer(n, d, E, 2.0, torch.bfloat16, alike)
        grads = tuple(torch.empty_like(t) for t in args[:4])
        times = []
        L.ec_profile_enable(1)
        for _ in range(12):
            B.ec_moe_backward(cfg, *args, saved, grads, ws)
            ms, names = (ctypes.c_float * 40)(), (ctypes.c_char_p * 40)()
            stages = [names[i].decode() for i in range(L.ec_profile_read(ms, names, 40))]
            times.append(ms[stages.index("bwd_combine")])
        L.ec_profile_enable(0)
        took.append(sorted(times)[6])
    assert took[1] <= 1.5 * took[0], took
