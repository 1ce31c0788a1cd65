"""Forces and link gradients that share one context's scratch: on two streams, by two
threads, through autograd (whose callers cannot choose the context) and beside a
replayed CUDA graph, each result the same bits as when it runs alone."""

import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import autograd, fields, hr  # noqa: E402
from tests.test_gpu_gauge_force import links  # noqa: E402

DIMS = (16, 18, 14, 20)
V = 16 * 18 * 14 * 20


def spinor(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn((V, 4, 2), dtype=torch.complex128, device="cuda", generator=g)


class Job:
    """Link gradient and gauge force of its own fields into its own buffers."""

    def __init__(self, seed):
        self.ctx = autograd.default_context(0)
        self.q = links(DIMS, seed)
        self.a, self.b = (fields.pack_spinor(self.ctx, DIMS, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, spinor(seed + k))
                          for k in (1, 2))
        self.G = torch.zeros((4, V, 4), dtype=torch.float64, device="cuda")
        self.F = torch.zeros((4, V, 3), dtype=torch.float64, device="cuda")

    def run(self, stream=None):
        hr.hr_link_grad(self.ctx, DIMS, self.a, self.b, 1.0, self.G, stream=stream)
        hr.hr_gauge_force(self.ctx, DIMS, 2.3, self.q, 1.0, self.F, stream=stream)

    def clear(self):
        self.G.zero_()
        self.F.zero_()
        torch.cuda.synchronize()

    def result(self):
        torch.cuda.synchronize()
        return self.G.clone(), self.F.clone()


def same(x, y):
    return all(torch.equal(a, b) for a, b in zip(x, y))


def alone(job):
    job.clear()
    job.run()
    return job.result()


def test_two_streams():
    jobs = [Job(10), Job(20)]
    want = [alone(j) for j in jobs]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(10):
        for j in jobs:
            j.clear()
        for j, s in zip(jobs, streams):
            j.run(s)
        assert same(jobs[0].result(), want[0]) and same(jobs[1].result(), want[1])


def test_two_threads():
    jobs = [Job(30), Job(40)]
    want = [alone(j) for j in jobs]
    bad = []

    def work(job, expect):
        s = torch.cuda.Stream()
        for _ in range(10):
            with torch.cuda.stream(s):
                job.G.zero_()
                job.F.zero_()
                job.run()
                s.synchronize()
                if not same((job.G, job.F), expect):
                    bad.append(1)
                s.synchronize()

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=a) for a in zip(jobs, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_autograd_on_two_streams():
    q = [links(DIMS, 50 + k).requires_grad_(True) for k in range(2)]
    psi = [spinor(60 + k).requires_grad_(True) for k in range(2)]
    w = [spinor(70 + k) for k in range(2)]

    def loss(k):
        return (w[k].conj() * autograd.DiracApply.apply(q[k], psi[k], DIMS, 0.2)).sum().real

    want = [torch.autograd.grad(loss(k), (q[k], psi[k])) for k in range(2)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(5):
        torch.cuda.synchronize()
        parts = []
        for k in range(2):
            with torch.cuda.stream(streams[k]):
                parts.append(loss(k))
        torch.cuda.synchronize()
        got = torch.autograd.grad(parts[0] + parts[1], (q[0], psi[0], q[1], psi[1]))
        torch.cuda.synchronize()
        assert same(got[:2], want[0]) and same(got[2:], want[1])


def test_beside_a_replayed_graph():
    captured, eager = Job(80), Job(90)
    want = [alone(captured), alone(eager)]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        captured.G.zero_()
        captured.F.zero_()
        captured.run()
    torch.cuda.synchronize()
    graph.replay()
    first = captured.result()
    # other kernels than outside a graph: 1e-14 of numbers up to 100 and up to 2.3 * 6
    assert (first[0] - want[0][0]).abs().max().item() <= 1e-12
    assert (first[1] - want[0][1]).abs().max().item() <= 1e-13
    s = torch.cuda.Stream()
    for _ in range(10):
        captured.clear()
        eager.clear()
        graph.replay()
        eager.run(s)
        assert same(captured.result(), first) and same(eager.result(), want[1])
