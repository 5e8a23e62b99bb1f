"""Calls from several host threads, each on a stream of its own, at the same time: every one gives the bits it gives alone."""
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
