"""One context per host thread, calls of different sizes at the same time: the
kernels' shared-memory limits belong to the device, so no call may lower one
that another thread's launch needs."""
import threading

import pytest

from test_gpu_parity import mt  # noqa: F401

pytestmark = pytest.mark.gpu


def in_threads(calls, reps):
    """Runs every call `reps` times in a thread of its own, all at once; the statuses that are not 0."""
    bad, gate = [], threading.Barrier(len(calls))

    def work(call):
        gate.wait()
        for _ in range(reps):
            s = call()
            if s != 0:
                bad.append(s)

    ts = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return bad


def contexts(count):
    import torch
    from paper_2603_18401_gb300 import Matcher

    return [Matcher(0, stream=torch.cuda.Stream()) for _ in range(count)]


def test_candidate_lists_of_small_and_large_images(mt):
    import torch

    ms = contexts(4)
    calls, keep = [], []
    for m, n in zip(ms, (100_000, 500, 100_000, 500)):
        g = torch.Generator(device="cuda").manual_seed(n)
        size = torch.tensor([640.0, 480.0], dtype=torch.float64, device="cuda")
        xy = [torch.rand(c, 2, dtype=torch.float64, device="cuda", generator=g) * size for c in (64, n)]
        d = [torch.randint(0, 256, (c, 32), dtype=torch.uint8, device="cuda", generator=g) for c in (64, n)]
        F = torch.tensor([0, 0, 0, 0, 0, -1.0, 0, 1.0, 0], dtype=torch.float64, device="cuda")
        o = m._alloc_out(64, True, 64 * n)
        pair, out = m.make_pair(*xy, F, 1.0, *d, 0, 32, 640, 480), m._out_struct(o, 64 * n)
        torch.cuda.synchronize()
        keep.append((xy, d, F, o))
        calls.append(lambda m=m, pair=pair, out=out: m.egm_match_pair(pair, out))
    assert in_threads(calls, 500) == []
    for m in ms:
        m.close()


def test_gms_of_coarse_and_fine_grids(mt):
    import ctypes as C

    import torch

    ms = contexts(4)
    calls, keep = [], []
    for m, grid in zip(ms, (48, 2, 24, 8)):
        xy = torch.rand(300, 2, dtype=torch.float64, device="cuda") * 640
        best = torch.arange(300, dtype=torch.int32, device="cuda")
        fl = torch.ones(300, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        keep.append((xy, best, fl))
        p = [C.c_void_p(t.data_ptr()) for t in (xy, xy, best, fl)]
        calls.append(lambda m=m, p=p, grid=grid: m.lib.egm_gms(m.ctx, p[0], 300, p[1], 300, p[2], p[3], 640, 640, 640,
                                                             640, 1, grid, 6.0))
    assert in_threads(calls, 500) == []
    for m in ms:
        m.close()
