"""Calls of several host threads that launch the same kernels with different amounts of shared memory."""
import threading

import numpy as np
import pytest
import torch

from paper_2501_13512_gb300 import inputs, vie

pytestmark = pytest.mark.gpu

K0 = 2 * np.pi
H = 0.05


def test_threads_with_different_shared_memory_sizes():
    """Products of planes and lines of 50 to 200 KB and block solves with different boxes, each thread on its own
    stream: every call returns, with the result of the same call alone."""
    shapes = [(48, 60, 6), (64, 64, 6), (60, 90, 6), (100, 20, 40)]
    errors, jobs = [], []
    for i, n in enumerate(shapes):
        eps_r, bid, x = inputs.random_case(n, seed=i)
        g = vie.Grid(eps_r, H)
        sp = g.spectrum(K0)
        w = inputs.metasurface(cells=1 + i % 2, seed=i)
        m = vie.Grid.from_workload(w)
        ms = m.spectrum(w.k0)
        b = torch.randn((3,) + m.shape, dtype=torch.complex64, device="cuda")
        xs = [torch.as_tensor(x).cuda().to(dt) for dt in (torch.complex128, torch.complex64)]
        jobs.append((g, sp, xs, m, ms, b))

    def calls(job):
        g, sp, xs, m, ms, b = job
        return [g.matvec(sp, x) for x in xs] + [m.precond(ms, b, inner_tol=1e-2)[0]]

    alone = [calls(j) for j in jobs]
    torch.cuda.synchronize()

    def run(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(100):
                    out = calls(jobs[k])
                torch.cuda.current_stream().synchronize()
            for a, b in zip(out, alone[k]):
                assert torch.equal(a, b)
        except Exception as e:  # noqa: BLE001 (reported by the test's own thread)
            errors.append(e)

    threads = [threading.Thread(target=run, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert not errors, errors[0]
