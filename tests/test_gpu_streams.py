"""Products whose launches follow one another across streams, threads and in captured graphs."""
import threading

import numpy as np
import pytest
import torch

from paper_2501_13512_gb300 import inputs, vie

pytestmark = pytest.mark.gpu

K0 = 2 * np.pi
H = 0.05
# planes in one CTA, and separate passes
SHAPES = [(20, 18, 9), (130, 20, 10)]
DTYPES = [torch.complex64, torch.complex128]


def case(n, dtype):
    eps_r, _, x = inputs.random_case(n, seed=sum(n))
    g = vie.Grid(eps_r, H)
    return g, g.spectrum(K0), torch.from_numpy(x).to(device="cuda", dtype=dtype)


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("dtype", DTYPES)
def test_captured_products(dtype, n):
    # two products in a row in a graph (the second reads the first's result), replayed on other data
    g, sp, x = case(n, dtype)
    y, z = torch.empty_like(x), torch.empty_like(x)
    want = g.matvec(sp, g.matvec(sp, 2 * x))
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        g.matvec(sp, x, y)
        g.matvec(sp, y, z)
    x.mul_(2)
    for _ in range(3):
        y.zero_()
        z.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(z, want)


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("dtype", DTYPES)
def test_chain_across_two_streams(dtype, n):
    # each product reads the result of the one before it, on the other stream, joined by events
    g, sp, x = case(n, dtype)
    want = x
    for _ in range(6):
        want = g.matvec(sp, want)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    bufs = [torch.empty_like(x) for _ in range(6)]
    for _ in range(10):
        src, done = x, None
        for k, dst in enumerate(bufs):
            s = streams[k % 2]
            if done is not None:
                s.wait_event(done)
            with torch.cuda.stream(s):
                g.matvec(sp, src, dst)
            done = s.record_event()
            src = dst
        done.synchronize()
        assert torch.equal(bufs[-1], want)
        for t in bufs:
            t.zero_()
        torch.cuda.synchronize()


def test_every_thread_of_several_finishes_with_its_own_result():
    """Products and block solves of grids that need different amounts of shared memory, a thread and a stream each."""
    jobs = []
    for i, n in enumerate([(48, 60, 6), (64, 64, 6), (60, 90, 6), (100, 20, 40)]):
        g, sp, x = case(n, torch.complex128)
        w = inputs.metasurface(cells=1 + i % 2, seed=i)
        m = vie.Grid.from_workload(w)
        b = torch.randn((3,) + m.shape, dtype=torch.complex64, device="cuda")
        jobs.append((g, sp, [x, x.to(torch.complex64)], m, m.spectrum(w.k0), b))

    def calls(job):
        g, sp, xs, m, ms, b = job
        return [g.matvec(sp, x) for x in xs] + [m.precond(ms, b, inner_tol=1e-2)[0]]

    alone = [calls(j) for j in jobs]
    torch.cuda.synchronize()
    done, errors = [], []

    def run(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(20):
                    out = calls(jobs[k])
                    torch.cuda.current_stream().synchronize()
                    for a, b in zip(out, alone[k]):
                        assert torch.equal(a, b)
            done.append(k)
        except Exception as e:  # noqa: BLE001 (reported by the test's own thread)
            errors.append(e)

    threads = [threading.Thread(target=run, args=(k,), daemon=True) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert not errors, errors[0]
    assert sorted(done) == list(range(len(jobs))) and not any(t.is_alive() for t in threads)
