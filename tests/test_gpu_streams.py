"""Calls from several host threads and streams at the same time, and results handed from one stream to another: every call gives
the bits it gives alone."""
import threading

import pytest
import torch

from paper_2202_09368_b200 import binding as B

pytestmark = pytest.mark.gpu


def _together(jobs, rounds):
    """jobs: callables that queue work on the current stream.  Runs each in a thread and a stream of its own, `rounds` times."""
    failed = []
    start = threading.Barrier(len(jobs))

    def work(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                for _ in range(rounds):
                    job()
        except Exception as e:
            failed.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(job,)) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed


def _routing(n, E, seed):
    cfg = B.make_config(n, 16, 8, E, 2.0, torch.float32)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    X, Wg = torch.empty(n, 16, device="cuda").normal_(generator=gen), torch.empty(16, E, device="cuda").normal_(generator=gen)
    want, out, ws = B.ec_route(cfg, X, Wg), B.ec_route(cfg, X, Wg), B.alloc_workspace(cfg)

    def check():
        for name in ("S", "I", "G", "row_ptr", "slots"):
            assert torch.equal(getattr(out, name), getattr(want, name))
            getattr(out, name).zero_()

    return lambda: B.ec_route(cfg, X, Wg, ws=ws, out=out), check


def test_routing_of_several_sizes_from_several_threads():
    """The one-launch selection and inverse index ask for as much shared memory as a call's size needs: a small call in one
    thread between the set-up and the launch of a large one in another must not take it away."""
    jobs = [_routing(n, 4, n) for n in (64, 4096, 300, 4000, 16000)]
    _together([j for j, _ in jobs], 2000)
    for _, check in jobs:
        check()


def _layer(n, d, dff, E, dtype, seed, **kw):
    cfg = B.make_config(n, d, dff, E, 2.0, dtype, **kw)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(scale, *shape):
        return (torch.empty(shape, device="cuda").normal_(generator=gen) * scale).to(dtype)

    X, Wg, W1, W2, dY = normal(1, n, d), normal(d ** -0.5, d, E), normal(d ** -0.5, E, d, dff), normal(dff ** -0.5, E, d, dff), normal(1, n, d)
    ws, saved, Y = B.alloc_workspace(cfg), B.alloc_saved(cfg), torch.empty_like(X)
    grads = tuple(torch.empty_like(t) for t in (X, Wg, W1, W2))

    def step():
        B.ec_moe_forward(cfg, X, Wg, W1, W2, X_out=Y, saved=saved, ws=ws)
        assert not kw.get("cap_b") or B.ec_read_status(ws) == B.EC_OK         # the solver's waits, before the backward pass clears the word
        B.ec_moe_backward(cfg, X, Wg, W1, W2, dY, saved, grads=grads, ws=ws)

    step()
    want = [t.clone() for t in (Y,) + grads]

    def check():
        assert B.ec_read_status(ws) == B.EC_OK
        for got, ref in zip((Y,) + grads, want):
            assert torch.equal(got, ref)

    return step, check


def test_layers_on_several_streams_at_once():
    """Kernels that are set up while their predecessor drains, products that fill every SM, and the solver, whose CTAs wait for one
    another, two of it among them."""
    bf16, f32 = torch.bfloat16, torch.float32
    jobs = [_layer(4096, 256, 512, 32, bf16, 1, cap_b=3, cap_iters=20), _layer(2048, 128, 256, 16, bf16, 2, cap_b=3, cap_iters=20),
            _layer(2048, 256, 1024, 8, bf16, 3), _layer(512, 128, 256, 10, f32, 4), _layer(20000, 64, 64, 8, bf16, 5)]
    _together([j for j, _ in jobs], 100)
    for _, check in jobs:
        check()


def test_results_handed_from_stream_to_stream():
    """The steps of the routing chain alternate between two streams that wait for each other's events, on new inputs every time: a kernel
    that is set up early still reads what the other stream wrote before the event."""
    n, d, E = 8192, 512, 16
    cfg = B.make_config(n, d, 8, E, 2.0, torch.bfloat16)
    gen = torch.Generator(device="cuda").manual_seed(3)
    Xs = [torch.empty(n, d, dtype=torch.bfloat16, device="cuda").normal_(generator=gen) for _ in range(4)]
    Wg = (torch.empty(d, E, device="cuda").normal_(generator=gen) / d ** 0.5).to(torch.bfloat16)
    k, ws = B.slots_per_expert(cfg), B.alloc_workspace(cfg)
    wants = []
    for X in Xs:
        r = B.ec_route(cfg, X, Wg, ws=ws)
        X_in = B.ec_shuffle(cfg, X, r.I)
        wants.append((X_in, B.ec_unshuffle(cfg, X_in.float(), r.G, r.row_ptr, r.slots)))
    X, r = torch.zeros_like(Xs[0]), B.ec_route(cfg, Xs[0], Wg, ws=ws)
    X_in, X_e = torch.empty(E, k, d, dtype=torch.bfloat16, device="cuda"), torch.empty(E, k, d, device="cuda")
    outs = [torch.empty_like(w[1]) for w in wants * 10]
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()

    def on(stream, other, f):
        stream.wait_stream(other)
        with torch.cuda.stream(stream):
            f()

    for i, out in enumerate(outs):
        on(one, two, lambda: X.copy_(Xs[i % 4]))
        on(two, one, lambda: B.ec_route(cfg, X, Wg, ws=ws, out=r))
        on(one, two, lambda: B.ec_shuffle(cfg, X, r.I, X_in))
        on(two, one, lambda: X_e.copy_(X_in))
        on(one, two, lambda: B.ec_unshuffle(cfg, X_e, r.G, r.row_ptr, r.slots, out))
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        assert torch.equal(out, wants[i % 4][1])
