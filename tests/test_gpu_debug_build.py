"""ec_validate_routing, and the index-checking build of the library (-DEC_DEBUG), on a B200.

The debug build stands in for a memory checker: every index a kernel reads from I, row_ptr or slots is compared with
its range first, a bad one is recorded (EC_ERR_INDEX) and the access it would have addressed is skipped.  It must
give the same bits as the normal build on valid inputs, and survive corrupted index structures, which only it is given.
"""
import ctypes
import importlib.util
import os

import pytest
import torch

from paper_2202_09368_b200 import binding as B
from paper_2202_09368_b200 import build as BUILD
from paper_2202_09368_b200 import inputs as IN

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


@pytest.fixture(scope="module")
def D():
    """A second instance of the binding, loaded on libecmoe_debug.so."""
    path = os.path.join(os.path.dirname(B.__file__), "libecmoe_debug.so")
    if not os.path.exists(path):
        BUILD.build(debug=True)
    spec = importlib.util.spec_from_file_location("binding_debug", B.__file__)
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    m._LIB_PATH = path
    assert m.ec_debug_build() and not B.ec_debug_build()
    return m


@pytest.mark.parametrize("router,groups,n,E,c", [("expert", 1, 2048, 16, 2.0), ("expert", 3, 1000, 12, 1.5), ("token", 1, 4096, 8, 2.0),
                                                ("token", 2, 1024, 8, 1.5), ("expert", 1, 40000, 8, 2.0)])
def test_validate_routing_accepts_what_the_router_makes_and_counts_what_is_wrong(router, groups, n, E, c):
    d = 32
    li = IN.make_layer_inputs(groups * n, d, 8, E, BF16, seed=31, with_grad=False, expert_skew=0.5 if router == "token" else 0.0)
    cfg = B.make_config(n, d, 8, E, c, BF16, groups=groups, router=router)
    X, Wg = li.X.cuda(), li.Wg.cuda()
    r = B.ec_route_token_choice(cfg, X, Wg) if router == "token" else B.ec_route(cfg, X, Wg)
    assert B.ec_validate_routing(cfg, r.I, r.row_ptr, r.slots) == 0
    k = B.ec_capacity(cfg) * groups
    filled = int(r.row_ptr[-1])

    def bad(I=None, row_ptr=None, slots=None):
        return B.ec_validate_routing(cfg, r.I if I is None else I, r.row_ptr if row_ptr is None else row_ptr,
                                     r.slots if slots is None else slots)

    I2 = r.I.clone(); I2[1, 3] = groups * n + 5                       # a token that does not exist
    assert bad(I=I2) >= 1
    I2 = r.I.clone(); I2[0, 0] = -7
    assert bad(I=I2) >= 1
    if router == "expert":
        I2 = r.I.clone(); I2[2, 1] = -1                               # empty slots exist only with the token-choice router
        assert bad(I=I2) >= 1
    if groups > 1:
        I2 = r.I.clone(); I2[0, 0] = I2[0, k - 1]                     # a token of the last group in a slot of the first
        assert bad(I=I2) >= 1
    rp = r.row_ptr.clone(); rp[5] = -3
    assert bad(row_ptr=rp) >= 1
    rp = r.row_ptr.clone(); rp[-1] += 1                               # one more slot listed than filled
    assert bad(row_ptr=rp) >= 1
    sl = r.slots.clone(); sl[2] = E * k + 9
    assert bad(slots=sl) >= 1
    if filled >= 4:
        sl = r.slots.clone(); sl[[0, filled - 1]] = sl[[filled - 1, 0]]   # two tokens' slots exchanged
        assert bad(slots=sl) >= 2


@pytest.mark.parametrize("dtype,n,d,dff,E,c,router", [(F32, 300, 36, 100, 3, 1.5, "expert"), (BF16, 1024, 128, 256, 8, 2.0, "expert"),
                                                      (BF16, 2048, 128, 384, 4, 2.6, "token"), (BF16, 1024, 128, 256, 8, 2.0, "capped"),
                                                      (BF16, 1024, 128, 256, 8, 2.0, "fused"), (F32, 300, 36, 100, 3, 1.5, "fused")])
def test_debug_build_gives_the_same_bits_and_reports_nothing_on_valid_inputs(D, dtype, n, d, dff, E, c, router):
    cap = dict(cap_b=3, cap_iters=20) if router == "capped" else dict(fuse_gather=True) if router == "fused" else {}
    rt = "token" if router == "token" else "expert"
    li = IN.make_layer_inputs(n, d, dff, E, dtype, seed=33, expert_skew=1.0 if rt == "token" else 0.0)
    X, Wg, W1, W2, dY = (t.cuda() for t in (li.X, li.Wg, li.W1, li.W2, li.dX_out))
    outs = []
    for lib in (B, D):
        cfg = lib.make_config(n, d, dff, E, c, dtype, router=rt, **cap)
        ws = lib.alloc_workspace(cfg)
        Y, saved = lib.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws)
        assert lib.ec_read_status(ws) == lib.EC_OK
        g = lib.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, ws=ws)
        assert lib.ec_read_status(ws) == lib.EC_OK
        outs.append([Y] + list(g))
    for a, b in zip(*outs):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))


@pytest.mark.parametrize("fuse", [False, True])
@pytest.mark.parametrize("dtype", [F32, BF16])
def test_debug_build_survives_and_reports_corrupted_indices(D, dtype, fuse):
    """Only the debug library is given these: indices far outside their ranges in the saved blob between forward and
    backward, and in the arguments of the stand-alone shuffle and unshuffle.  Every bad access is skipped."""
    n, d, dff, E, c = 1024, 128, 256, 8, 2.0
    li = IN.make_layer_inputs(n, d, dff, E, dtype, seed=35)
    X, Wg, W1, W2, dY = (t.cuda() for t in (li.X, li.Wg, li.W1, li.W2, li.dX_out))
    cfg = D.make_config(n, d, dff, E, c, dtype, fuse_gather=fuse)    # fused: the dW1 product reads rows of X through the bad I
    k = D.ec_capacity(cfg)
    ws = D.alloc_workspace(cfg)
    Y, saved = D.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws)
    assert D.ec_read_status(ws) == D.EC_OK
    v = D.saved_view(cfg, saved)
    v["I"][0, 0] = n + 11; v["I"][3, 5] = -9
    v["slots"][3] = E * k + 5; v["slots"][100] = -2
    v["row_ptr"][7] = -3; v["row_ptr"][500] = E * k + 77
    g = D.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, ws=ws)
    assert D.ec_read_status(ws) == D.EC_ERR_INDEX
    assert all(torch.isfinite(t.float()).all() for t in g)
    # the stand-alone calls have no workspace to report in; they must simply not touch memory they should not
    r = D.ec_route(cfg, X, Wg)
    I = r.I.clone(); I[0, :4] = torch.tensor([n, 2 * n, -5, 2 ** 30], dtype=torch.int32)
    X_in = D.ec_shuffle(cfg, X, I)
    assert torch.equal(X_in[0, 4:], X[r.I[0, 4:].long()]) and not X_in[0, :4].any()
    sl = r.slots.clone(); sl[:3] = torch.tensor([E * k, -1, 2 ** 30], dtype=torch.int32)
    rp = r.row_ptr.clone(); rp[9] = -4
    out = D.ec_unshuffle(cfg, X_in.float(), r.G, rp, sl)
    assert torch.isfinite(out.float()).all()
    torch.cuda.synchronize()


@pytest.mark.parametrize("n,E,groups", [(130, 8, 1), (4736, 32, 1), (9000, 64, 1), (1500, 16, 3), (16384, 128, 1)])
def test_a_solver_wait_that_runs_out_is_reported_and_leaves_a_defined_assignment(D, n, E, groups):
    """Registers and shared memory, one group and three.  One CTA of a group leaves no words from the second pass on and the others
    wait 5 ms: the call ends, the status says so, A holds numbers that a selection can work on, and the next call on the same
    workspace is the right one."""
    cfg = D.make_config(n, 8, 8, E, 2.0, BF16, groups=groups, cap_b=3, cap_iters=20, cap_lambda=1e-2)
    gen = torch.Generator(device="cuda").manual_seed(n)
    S = torch.softmax(torch.empty(n * groups, E, device="cuda").normal_(generator=gen), dim=1)
    want = D.ec_capped_assignment(cfg, S)
    ws = D.alloc_workspace(cfg)
    A = torch.full_like(S, float("nan"))
    call = D.lib().ec_debug_capped_wait
    call.argtypes = [ctypes.POINTER(D.ec_config)] + [ctypes.c_void_p] * 3 + [ctypes.c_size_t, ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p]
    assert call(ctypes.byref(cfg), S.data_ptr(), A.data_ptr(), ws.data_ptr(), ws.numel(), 5_000_000, 1, D._stream()) == D.EC_OK
    assert D.ec_read_status(ws) == D.EC_ERR_TIMEOUT
    assert bool(((A >= 0) & (A <= 1)).all())
    again = D.ec_capped_assignment(cfg, S, ws=ws)
    assert D.ec_read_status(ws) == D.EC_OK and torch.equal(again, want)


@pytest.mark.parametrize("n,E,groups", [(2000, 8, 1), (500, 16, 3), (9000, 64, 1), (20000, 32, 1), (20000, 48, 1)])
def test_a_gate_whose_waits_run_out_leaves_an_index_inside_its_buffers(D, n, E, groups):
    """128 tokens never get scores, on a workspace full of ones (the marks among them): the status says so, the index that the
    selection of whatever S holds leads to is a whole one, and the next call on the same workspace is the right one."""
    cfg = D.make_config(n, 128, 8, E, 2.0, BF16, groups=groups)
    li = IN.make_layer_inputs(n * groups, 128, 8, E, BF16, seed=n)
    X, Wg = li.X.cuda(), li.Wg.cuda()
    ws = D.alloc_workspace(cfg)
    want = D.ec_route(cfg, X, Wg, ws=ws)
    assert D.ec_read_status(ws) == D.EC_OK
    ws.fill_(255)
    fields = ("S", "I", "G", "row_ptr", "slots")
    r = D.Routing(*(torch.zeros_like(getattr(want, f)) for f in fields))
    call = D.lib().ec_debug_gate_wait
    call.argtypes = [ctypes.POINTER(D.ec_config)] + [ctypes.c_void_p] * 8 + [ctypes.c_size_t, ctypes.c_void_p]
    assert call(ctypes.byref(cfg), X.data_ptr(), Wg.data_ptr(), *(getattr(r, f).data_ptr() for f in fields), ws.data_ptr(), ws.numel(), D._stream()) == D.EC_OK
    assert D.ec_read_status(ws) == D.EC_ERR_TIMEOUT
    assert int(r.row_ptr[-1]) == r.I.numel() and D.ec_validate_routing(cfg, r.I, r.row_ptr, r.slots, ws=ws) == 0
    again = D.ec_route(cfg, X, Wg, ws=ws)
    assert D.ec_read_status(ws) == D.EC_OK and all(torch.equal(getattr(again, f), getattr(want, f)) for f in fields)


@pytest.mark.parametrize("kind", [0, 1, 2])
def test_fp32_products_go_to_the_multiply_adds_where_the_tensor_kernel_cannot_run(D, kind):
    """As if the compiler had given it other registers than its split among the warps needs."""
    n, d, dff, E = 2048, 512, 1024, 8
    cfg = D.make_config(n, d, dff, E, 2.0, F32)
    k = D.ec_capacity(cfg)
    gen = torch.Generator(device="cuda").manual_seed(kind)
    rows, b = {0: ((E, k, d), (E, d, dff)), 1: ((E, k, dff), (E, d, dff)), 2: ((E, k, d), (E, k, dff))}[kind]
    A, Bm = (torch.empty(s, device="cuda").normal_(generator=gen) for s in (rows, b))
    want = {0: lambda: A.double() @ Bm.double(), 1: lambda: A.double() @ Bm.double().mT, 2: lambda: A.double().mT @ Bm.double()}[kind]()
    usual = D.ec_expert_gemm(cfg, kind, A, Bm)
    ws, out = D.alloc_workspace(cfg), torch.full_like(usual, float("nan"))
    call = D.lib().ec_debug_expert_gemm_registers
    call.argtypes = [ctypes.POINTER(D.ec_config), ctypes.c_int] + [ctypes.c_void_p] * 4 + [ctypes.c_size_t, ctypes.c_void_p]
    assert call(ctypes.byref(cfg), kind, A.data_ptr(), Bm.data_ptr(), out.data_ptr(), ws.data_ptr(), ws.numel(), D._stream()) == D.EC_OK
    # sums of at most 1024 fp32 products, one after the other: a few 1e-7 of the result in the 2-norm, at most 1024 * 2^-24
    assert float((out - want).norm() / want.norm()) < 1024 * 2.0 ** -24 and not torch.equal(out, usual)


@pytest.mark.parametrize("n,d,E,dtype", [(3000, 768, 8, BF16), (2000, 1024, 16, F32), (1500, 2048, 8, F32), (1000, 4096, 8, BF16), (700, 8192, 4, BF16)])
def test_an_unshuffle_whose_waits_run_out_is_finished_all_the_same(D, n, d, E, dtype):
    """One CTA of the ring gets its first rows only and its warps wait 2 ms for the others: nobody can tell from the result."""
    cfg = D.make_config(n, d, 8, E, 2.0, dtype)
    gen = torch.Generator(device="cuda").manual_seed(n)
    I = torch.stack([torch.randperm(n, device="cuda", generator=gen)[:D.ec_capacity(cfg)] for _ in range(E)]).flatten()
    slots = torch.sort(I, stable=True)[1].int()
    row_ptr = torch.cat([I.new_zeros(1), torch.bincount(I, minlength=n).cumsum(0)]).int()
    X_e = torch.empty((I.numel(), d), device="cuda").normal_(generator=gen)
    G = torch.rand(I.numel(), device="cuda", generator=gen)
    want = D.ec_unshuffle(cfg, X_e, G, row_ptr, slots)
    out = torch.full_like(want, float("nan"))
    call = D.lib().ec_debug_unshuffle_wait
    call.argtypes = [ctypes.POINTER(D.ec_config)] + [ctypes.c_void_p] * 5 + [ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p]
    assert call(ctypes.byref(cfg), X_e.data_ptr(), G.data_ptr(), row_ptr.data_ptr(), slots.data_ptr(), out.data_ptr(), 2_000_000, 1, D._stream()) == D.EC_OK
    assert torch.equal(out, want)


@pytest.mark.parametrize("n,E,dtype,kw", [(2048, 8, BF16, {}), (20000, 8, BF16, {}), (2048, 8, F32, dict(fuse_gather=True)), (2048, 8, BF16, dict(fuse_gather=True)),
                                          (2048, 8, BF16, dict(router="token")), (2048, 8, BF16, dict(cap_b=3, cap_iters=5)),
                                          (20000, 65, BF16, dict(cap_b=3, cap_iters=5)), (1000, 10, F32, dict(groups=2))])
def test_a_layer_with_rows_of_nan_stays_inside_its_buffers(D, n, E, dtype, kw):
    """Half of the tokens are NaN, many more than an expert takes: whatever the values, no index is out of range."""
    d, dff, g = 64, 64, kw.get("groups", 1)
    cfg = D.make_config(n, d, dff, E, 1.0, dtype, **kw)
    li = IN.make_layer_inputs(n * g, d, dff, E, dtype, seed=n)
    X, Wg, W1, W2, dY = (t.cuda() for t in (li.X, li.Wg, li.W1, li.W2, li.dX_out))
    X[::2] = float("nan")
    ws = D.alloc_workspace(cfg)
    Y, saved = D.ec_moe_forward(cfg, X, Wg, W1, W2, ws=ws)
    assert D.ec_read_status(ws) == D.EC_OK
    v = D.saved_view(cfg, saved)
    assert D.ec_validate_routing(cfg, v["I"], v["row_ptr"], v["slots"]) == 0
    D.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, ws=ws)
    assert D.ec_read_status(ws) == D.EC_OK
