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
