"""Scratch that mp_bb_solve keeps between calls: bounded for all threads together, given back, and the
same results from threads on streams of their own as from one thread."""
import threading

import numpy as np
import pytest
import torch

from gpu_util import require_cuda

pytestmark = pytest.mark.gpu

N_THREADS = 4


def _problem(V, n, seed):
    from paper_1503_01721_gb300 import api
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    DA = torch.rand((n, V), generator=gen, device="cuda") * (torch.rand((n, V), generator=gen, device="cuda") < 0.3)
    f = lambda a: torch.tensor(a, device="cuda")
    vox = api.VoxelParams(torch.randint(0, 3, (V,), generator=gen, device="cuda", dtype=torch.uint8),
                          f([0.6, 0.5, 1.0]), f([0.05, 0.3, 1.0]), f([0.0, 0.0, 1.0]))
    return DA, vox, torch.zeros(n, device="cuda"), torch.empty(V, device="cuda")


def _used():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_threads_and_streams():
    require_cuda()
    import __graft_entry__
    __graft_entry__.build()
    from paper_1503_01721_gb300 import api
    opts = api.BBOptions(30, 1e-9, 1e-12)
    # growing sizes, the largest about 100 MB of scratch
    sizes = [(40000, 3), (90000, 9), (200000, 20), (600000, 40), (50000, 12)]
    streams = [torch.cuda.Stream() for _ in range(N_THREADS)]
    want = {}
    for t in range(N_THREADS):
        for V, n in sizes:
            DA, vox, y, z = _problem(V, n, 10 * t + n)
            rep = api.mp_bb_solve(DA, vox, y, z, opts=opts)
            want[t, V] = (y.cpu(), z.cpu(), rep)
            del DA, vox, y, z
        with torch.cuda.stream(streams[t]):  # the driver's own memory for a stream is there from its first launch on
            api.mp_bb_solve(*_problem(40000, 3, 0), opts=opts)
    ddc = api.Ddc(4, 4, *(torch.zeros(1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.float32)))
    ddc.close()  # gives back what the calls above left
    problems = {(t, V): _problem(V, n, 10 * t + n) for t in range(N_THREADS) for V, n in sizes}
    before = _used()
    go, done, leave, bad = threading.Barrier(N_THREADS), threading.Barrier(N_THREADS + 1), threading.Event(), []

    def work(t):
        try:
            go.wait(60)
            for _ in range(3):
                for V, _n in sizes:
                    DA, vox, y, z = problems[t, V]
                    with torch.cuda.stream(streams[t]):
                        y.zero_()
                        rep = api.mp_bb_solve(DA, vox, y, z, opts=opts)
                    if not (torch.equal(y.cpu(), want[t, V][0]) and torch.equal(z.cpu(), want[t, V][1])
                            and rep == want[t, V][2]):
                        bad.append((t, V))
        except Exception as e:  # noqa: BLE001
            bad.append((t, repr(e)))
        done.wait(120)
        leave.wait(120)  # the thread lives on: what it kept would still be held

    threads = [threading.Thread(target=work, args=(t,)) for t in range(N_THREADS)]
    for th in threads:
        th.start()
    done.wait(120)
    kept = _used() - before
    leave.set()
    for th in threads:
        th.join()
    assert bad == []
    assert kept <= (128 + 64) << 20, f"{kept >> 20} MB kept by {N_THREADS} threads"
    ddc = api.Ddc(4, 4, *(torch.zeros(1, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.float32)))
    ddc.close()
    assert _used() - before <= 64 << 20
