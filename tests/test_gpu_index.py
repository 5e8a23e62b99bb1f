"""The token -> slot index against a stable sort of I: one CTA's limit (4096 tokens, or what fits its shared memory), the cluster's
(16384 tokens, 2^17 slots), mark words of 1 to 8 per token, the scan beyond them with and without ranks, routing groups, empty slots."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,E,c,groups,router", [
    (256, 4, 2.0, 1, "expert"), (1, 1, 1.0, 1, "expert"), (31, 31, 3.0, 1, "expert"), (2048, 8, 2.0, 1, "expert"), (4096, 32, 2.0, 1, "expert"),
    (4096, 33, 2.0, 1, "expert"), (16384, 64, 2.0, 1, "expert"), (8192, 256, 8.0, 1, "expert"), (16384, 128, 4.0, 1, "expert"),
    (8191, 104, 9.0, 1, "expert"), (16385, 32, 2.0, 1, "expert"), (16385, 40, 2.0, 1, "expert"), (20000, 256, 2.0, 1, "expert"),
    (16384, 4, 2.0, 1, "expert"), (4096, 8, 2.0, 1, "expert"), (4097, 8, 2.0, 1, "expert"), (16384, 32, 8.0, 1, "expert"), (16383, 32, 8.01, 1, "expert"),
    (16384, 64, 8.01, 1, "expert"), (4096, 256, 2.0, 1, "expert"), (512, 256, 2.0, 8, "expert"), (1000, 16, 1.5, 5, "expert"), (1000, 72, 1.5, 16, "expert"), (3000, 16, 1.0, 9, "expert"),
    (3000, 48, 1.0, 9, "expert"), (4096, 16, 2.0, 1, "token"), (1024, 40, 2.0, 3, "token"), (20000, 16, 2.0, 1, "token"), (9000, 64, 1.0, 2, "token")])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_index_is_a_stable_sort(n, E, c, groups, router, dtype):
    d, N = 16, n * groups
    cfg = B.make_config(n, d, 8, E, c, dtype, groups=groups, router=router)
    gen = torch.Generator(device="cuda").manual_seed(n + E)
    X = torch.empty((N, d), device="cuda").normal_(generator=gen).to(dtype)
    Wg = (torch.empty((d, E), device="cuda").normal_(generator=gen) / 4).to(dtype)
    ws = B.alloc_workspace(cfg)
    ws.fill_(0xA5)                                      # whatever an earlier call left
    route = B.ec_route if router == "expert" else B.ec_route_token_choice
    for _ in range(2):
        r = route(cfg, X, Wg, ws=ws)
        assert B.ec_read_status(ws) == B.EC_OK
        I = r.I.flatten().long()
        filled = (I >= 0).nonzero().flatten()
        order = torch.sort(I[filled], stable=True)[1]
        lengths = torch.bincount(I[filled], minlength=N)
        assert torch.equal(r.row_ptr.long(), torch.cat([lengths.new_zeros(1), lengths.cumsum(0)]))
        assert torch.equal(r.slots.flatten()[:filled.numel()].long(), filled[order])
        assert B.ec_validate_routing(cfg, r.I, r.row_ptr, r.slots, ws) == 0


def _shortest_us(n, E, groups, stages):
    """The shortest of 30 calls' time in the given stages."""
    cfg = B.make_config(n, 256, 8, E, 2.0, torch.bfloat16, groups=groups)
    gen = torch.Generator(device="cuda").manual_seed(n)
    X = torch.empty((n * groups, 256), device="cuda").normal_(generator=gen).bfloat16()
    Wg = (torch.empty((256, E), device="cuda").normal_(generator=gen) / 16).bfloat16()
    ws, times = B.alloc_workspace(cfg), []
    r = B.ec_route(cfg, X, Wg, ws=ws)
    B.ec_profile_enable(True)
    try:
        for _ in range(30):
            B.ec_route(cfg, X, Wg, ws=ws, out=r)
            times.append(sum(ms for stage, ms in B.ec_profile_read() if stage in stages))
    finally:
        B.ec_profile_enable(False)
    return 1e3 * min(times)


def test_columns_beyond_one_per_sm_need_no_second_round():
    """16384 tokens: 256 experts take 1.34 times as long as 128 where an SM holds one CTA of the selection, 1.1 times where it holds two."""
    assert _shortest_us(16384, 256, 1, ("topk",)) < 1.22 * _shortest_us(16384, 128, 1, ("topk",))


def test_many_small_columns_do_not_wait_for_the_index():
    """Sixteen groups of 256 tokens with 64 experts and one of 4096: 2.1 times as long where each of the 1024 CTAs has the threads that
    the index wants."""
    stages = ("topk", "topk_index", "inverse_index")
    assert _shortest_us(256, 64, 16, stages) < 1.4 * _shortest_us(4096, 64, 1, stages)
