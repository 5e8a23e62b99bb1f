"""The capped solver in one cluster per group: the limits of eight and sixteen CTAs in tokens, experts and ranks that own none, more
passes than one use of every buffer, and sizes just beyond.  Against the same rounds in 64 bits, the same bits on every call, and in a captured graph."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

from test_gpu_capped_forms import ITERS, LAM, _rounds_in_64_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,E,groups", [(5, 2, 1), (300, 4, 1), (512, 8, 1), (2048, 32, 1), (2049, 31, 1), (1024, 64, 1), (512, 128, 1), (256, 256, 1),
                                        (257, 250, 1), (256, 100, 4), (700, 16, 6), (4096, 16, 1), (4097, 32, 1), (2048, 64, 1), (2049, 60, 1), (512, 256, 1),
                                        (1500, 33, 9)])
def test_clusters_match_64_bits(n, E, groups):
    cfg = B.make_config(n, 8, 8, E, 2.0, torch.bfloat16, groups=groups, cap_b=2, cap_iters=ITERS, cap_lambda=LAM)
    k = B.ec_capacity(cfg)
    gen = torch.Generator(device="cuda").manual_seed(n + E)
    S = torch.softmax(torch.empty(n * groups, E, device="cuda").normal_(generator=gen), dim=1)
    ws = B.alloc_workspace(cfg)
    ws.fill_(0x5A)
    A = B.ec_capped_assignment(cfg, S, ws=ws)
    assert B.ec_read_status(ws) == B.EC_OK
    bound = 4 * ITERS / LAM * 2.0 ** -24                # see test_gpu_capped_forms
    for g in range(groups):
        rows = slice(g * n, (g + 1) * n)
        assert (A[rows].double() - _rounds_in_64_bits(S[rows], k, 2)).abs().max().item() <= bound
    out = torch.empty_like(A)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.ec_capped_assignment(cfg, S, ws=ws, A=out)
    for _ in range(3):
        out.zero_()
        graph.replay()
        assert torch.equal(out, A)
    assert B.ec_read_status(ws) == B.EC_OK
