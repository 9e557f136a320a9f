"""GPU: plan memory is reused between plans, by any thread and stream, and given back.

Plans of different shapes are created, applied and destroyed in turn from two threads on
their own streams; every result equals, bit for bit, that of a plan made alone.  Freed
plan memory stays within the documented 2 GiB and returns to the device on request.
"""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_plan_memory_reuse_and_release():
    import torch
    from paper_1604_04374_gb300 import Plan, build, pce
    build.build()
    dev = torch.device("cuda", 0)
    probs = [synth.problem_2d(256, 128, 8, 3, 51, "normal"), synth.problem_2d(1024, 64, 4, 2, 52, "normal"),
             synth.problem_1d(4096, 8, 5, 53)]
    data = [tuple(torch.from_numpy(a).to(dev) for a in (p.w, p.h, p.u)) for p in probs]

    def run(i, stream):
        w, h, u = data[i]
        with torch.cuda.stream(stream):
            plan = Plan(w, h=h)
            y, x = plan.apply(u), plan.apply_adjoint(u)
            stream.synchronize()
            plan.close()
            return y.cpu().numpy(), x.cpu().numpy()

    ref = [run(i, torch.cuda.Stream()) for i in range(len(data))]
    bad = []

    def worker(t):
        s = torch.cuda.Stream()
        for n in range(12):
            i = (n + t) % len(data)
            if not all(np.array_equal(a, b) for a, b in zip(run(i, s), ref[i])):
                bad.append((t, n))

    threads = [threading.Thread(target=worker, args=(t,)) for t in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad

    pce.pce_release_memory()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    big = synth.problem_2d(1024, 1024, 4, 1, 54)
    plan = Plan(torch.from_numpy(big.w).to(dev), h=torch.from_numpy(big.h).to(dev))
    scratch = plan.info()[2]
    assert scratch > 256 << 20
    assert torch.cuda.mem_get_info()[0] <= free0 - scratch
    plan.close()
    slack = 256 << 20   # torch's own cache and allocation granularity
    assert torch.cuda.mem_get_info()[0] >= free0 - (2 << 30) - slack
    pce.pce_release_memory()
    assert torch.cuda.mem_get_info()[0] >= free0 - slack


def test_closed_plans_keep_at_most_two_gib():
    """Plans of about 4 GiB together, all closed: the library keeps some of their memory, but
    no more than 2 GiB, until it is asked for it."""
    import torch
    from paper_1604_04374_gb300 import Plan, build, pce
    build.build()
    dev = torch.device("cuda", 0)
    big = synth.problem_2d(1024, 1024, 4, 1, 55)
    w, h = torch.from_numpy(big.w).to(dev), torch.from_numpy(big.h).to(dev)
    pce.pce_release_memory()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    plans = [Plan(w, h=h) for _ in range(4)]
    held = free0 - torch.cuda.mem_get_info()[0]
    assert held > 3 << 30
    for p in plans:
        p.close()
    torch.cuda.synchronize()
    slack = 256 << 20
    kept = free0 - torch.cuda.mem_get_info()[0]
    assert kept <= (2 << 30) + slack and kept > 0
    pce.pce_release_memory()
    assert torch.cuda.mem_get_info()[0] >= free0 - slack
