"""The combine of results that exceed L2 (rows through a ring in shared memory where they are wide enough): every width class, tokens without slots (a group of
warps that runs ahead of the others) and with more slots than the ring has entries, against 64 bits and the same bits twice."""
import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,E,c,dtype", [(140000, 128, 8, 2.0, torch.bfloat16), (70000, 520, 16, 1.0, torch.float32), (33000, 1024, 64, 1.0, torch.bfloat16),
                                           (20001, 1704, 64, 1.0, torch.bfloat16), (8200, 4096, 32, 1.0, torch.bfloat16), (4300, 8192, 64, 1.0, torch.float32)])
@pytest.mark.parametrize("crowded", [False, True])
def test_combine_through_the_ring(n, d, E, c, dtype, crowded):
    """crowded: every expert takes the same tokens, so that most tokens have no slot and the others E of them."""
    cfg = B.make_config(n, d, 8, E, c, dtype)
    k = B.ec_capacity(cfg)
    assert E * k * d >= 32 << 20
    gen = torch.Generator(device="cuda").manual_seed(n)
    if crowded:
        I = torch.randperm(n, device="cuda", generator=gen)[:k].sort()[0].repeat(E, 1)
    else:
        I = torch.stack([torch.randperm(n, device="cuda", generator=gen)[:k] for _ in range(E)])
    I = I.flatten()
    order = torch.sort(I, stable=True)[1]
    row_ptr = torch.cat([I.new_zeros(1), torch.bincount(I, minlength=n).cumsum(0)]).int()
    X_e = torch.empty((E, k, d), device="cuda").normal_(generator=gen)
    G = torch.rand((E, k), device="cuda", generator=gen)
    out = B.ec_unshuffle(cfg, X_e, G, row_ptr, order.int())
    want, size = torch.zeros((n, d), device="cuda", dtype=torch.float64), torch.zeros((n, d), device="cuda", dtype=torch.float64)
    for e in range(E):
        rows, y = I[e * k:(e + 1) * k], G[e].double()[:, None] * X_e[e].double()
        want[rows] += y
        size[rows] += y.abs()
    eps = 2.0 ** -24 if dtype == torch.float32 else 2.0 ** -8          # of the rounding to the result's type; at most E sums in fp32
    assert ((out.double() - want).abs() <= eps * want.abs() + (E + 1) * 2.0 ** -24 * size).all()
    assert torch.equal(out, B.ec_unshuffle(cfg, X_e, G, row_ptr, order.int()))


def _median_time(call):
    times = []
    for _ in range(12):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return sorted(times)[6]


@pytest.mark.parametrize("n,d,E", [(16384, 1024, 64), (16384, 4096, 64)])
def test_tokens_with_many_slots_side_by_side_cost_no_more(n, d, E):
    """Every expert takes the same first tokens (as with padding rows that are all alike: ties go to the lowest): the same bytes as
    anywhere, and all SMs have to share them.  Times vary by some percent; one SM in thirty at work is a factor of twenty."""
    cfg = B.make_config(n, d, 8, E, 2.0, torch.bfloat16)
    k = B.ec_capacity(cfg)
    gen = torch.Generator(device="cuda").manual_seed(n)
    X_e = torch.empty((E, k, d), device="cuda").normal_(generator=gen)
    G, out = torch.rand((E, k), device="cuda", generator=gen), torch.empty((n, d), device="cuda", dtype=torch.bfloat16)
    took = []
    for I in (torch.stack([torch.randperm(n, device="cuda", generator=gen)[:k] for _ in range(E)]), torch.arange(k, device="cuda").repeat(E, 1)):
        slots = torch.sort(I.flatten(), stable=True)[1].int()
        row_ptr = torch.cat([I.new_zeros(1), torch.bincount(I.flatten(), minlength=n).cumsum(0)]).int()
        took.append(_median_time(lambda: B.ec_unshuffle(cfg, X_e, G, row_ptr, slots, out)))
    assert took[1] <= 3 * took[0]


def test_narrow_rows_take_about_as_long_as_wide_ones():
    """The same bytes in rows of 1024, 256, 64 and 32: a kernel that pays per row would take several times as long."""
    took = []
    for d in (1024, 256, 64, 32):
        n, E = (32 << 20) // (2 * d), 32
        cfg = B.make_config(n, d, 8, E, 2.0, torch.bfloat16)
        k = B.ec_capacity(cfg)
        gen = torch.Generator(device="cuda").manual_seed(d)
        I = torch.stack([torch.randperm(n, device="cuda", generator=gen)[:k] for _ in range(E)]).flatten()
        slots = torch.sort(I, stable=True)[1].int()
        row_ptr = torch.cat([I.new_zeros(1), torch.bincount(I, minlength=n).cumsum(0)]).int()
        X_e, G = torch.empty((E, k, d), device="cuda").normal_(generator=gen), torch.rand((E, k), device="cuda", generator=gen)
        out = torch.empty((n, d), device="cuda", dtype=torch.bfloat16)
        took.append(_median_time(lambda: B.ec_unshuffle(cfg, X_e, G, row_ptr, slots, out)))
    assert max(took) <= 2.5 * took[0], took
