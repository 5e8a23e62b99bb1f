"""The capped solver at the edges of its resident forms (tokens per warp, experts per lane, groups, the state in registers and in
shared memory), against the same rounds in 64 bits."""
import math

import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu

LAM, ITERS = 1e-2, 30


def _rounds_in_64_bits(S, k, b):
    L = S.double() / LAM
    qb, qc = torch.zeros_like(L), torch.zeros_like(L[:, :1])
    for _ in range(ITERS):
        L = L + math.log(k) - torch.logsumexp(L, dim=0, keepdim=True) + qc
        m = torch.clamp(math.log(b) - torch.logsumexp(L, dim=1, keepdim=True), max=0.0)
        qc = -m
        box = L + m + qb
        L = torch.clamp(box, max=0.0)
        qb = box - L
    return torch.exp(L)


# tokens per warp on 148 SMs of 32 warps: up to 4736 one, 9472 two, 18944 four, 37888 eight (of 32 experts at most)
@pytest.mark.parametrize("n,E,groups", [(33, 8, 1), (4736, 32, 1), (4737, 7, 1), (9473, 20, 1), (18945, 32, 1), (18900, 64, 1), (4737, 33, 1),
                                        (9470, 100, 1), (4730, 256, 1), (130, 200, 1), (1500, 16, 3), (40, 64, 160), (16384, 128, 1),
                                        (20000, 65, 1)])
def test_capped_rounds_match_64_bits(n, E, groups):
    c, b = 2.0, 2
    cfg = B.make_config(n, 8, 8, E, c, torch.bfloat16, groups=groups, cap_b=b, cap_iters=ITERS, cap_lambda=LAM)
    k = B.ec_capacity(cfg)
    gen = torch.Generator(device="cuda").manual_seed(n + E)
    S = torch.softmax(torch.empty(n * groups, E, device="cuda").normal_(generator=gen), dim=1)
    ws = B.alloc_workspace(cfg)
    # log A is at most 1 / LAM = 100 in size and is rounded about four times a round: 4 * 30 * 100 * 2^-24
    bound = 4 * ITERS / LAM * 2.0 ** -24
    for _ in range(2):                                  # the second call finds the first one's words in the workspace
        A = B.ec_capped_assignment(cfg, S, ws=ws)
        assert B.ec_read_status(ws) == B.EC_OK
        for g in range(groups):
            rows = slice(g * n, (g + 1) * n)
            assert (A[rows].double() - _rounds_in_64_bits(S[rows], k, b)).abs().max().item() <= bound
