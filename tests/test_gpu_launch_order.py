"""Operators among other work: after a wait for another stream, inside a caller's
CUDA graph with branches, and with two contexts on two streams.  Their kernels may
become resident before the previous kernel of the stream has finished
(programmatic launches), and still see everything that is ordered before them."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import fields, hr  # noqa: E402
from tests.test_gpu_gauge_force import links  # noqa: E402

DIMS = (8, 8, 6, 10)
M0 = 0.2


def _setup(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    V = DIMS[0] * DIMS[1] * DIMS[2] * DIMS[3]
    ctx = hr.Context(0)
    gauge = fields.pack_gauge(ctx, DIMS, hr.HR_FUND, hr.HR_F64, links(DIMS, seed))
    x = fields.pack_spinor(ctx, DIMS, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN,
                           torch.randn((V, 4, 2), dtype=torch.complex128, device="cuda", generator=g))
    return ctx, gauge, x


def _work(ctx):
    return fields.empty_bytes(hr.hr_dirac_workspace_bytes(DIMS, hr.HR_FUND, hr.HR_F64, hr.HR_OP_NORMAL, 1))


def _normal(ctx, gauge, x, y, work, stream=None):
    hr.hr_dirac_eo(ctx, DIMS, M0, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, hr.HR_OP_NORMAL, 1, gauge, x, y, work,
                   stream=stream)


def _chain(ctx, gauge, x, n=6):
    """x -> A x, n times."""
    work, y = _work(ctx), torch.empty_like(x)
    for _ in range(n):
        _normal(ctx, gauge, x, y, work)
        x, y = y, x.clone()
    return x


def test_after_a_wait_for_another_stream():
    ctx, gauge, x = _setup(51)
    want = _chain(ctx, gauge, x.clone())
    big = torch.randn(4096, 4096, device="cuda")
    s = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    work, y = _work(ctx), torch.empty_like(x)
    cur = torch.zeros_like(x)
    for k in range(6):
        # the operand comes late, from the stream that is not the operator's
        with torch.cuda.stream(s[(k + 1) % 2]):
            for _ in range(4):
                big = big @ big * 1e-3
            cur = x.clone() if k == 0 else y.clone()
            ev = torch.cuda.Event()
            ev.record()
        with torch.cuda.stream(s[k % 2]):
            s[k % 2].wait_event(ev)
            y = torch.empty_like(x)
            _normal(ctx, gauge, cur, y, work)
            cur.record_stream(s[k % 2])
            done = torch.cuda.Event()
            done.record()
        s[(k + 1) % 2].wait_event(done)
        y.record_stream(s[(k + 1) % 2])
        y.record_stream(s[k % 2])
    torch.cuda.synchronize()
    assert torch.equal(y, want)


def test_inside_a_callers_graph_with_branches():
    ctx, gauge, x = _setup(52)
    ctx2, gauge2, x2 = _setup(53)
    want = [_chain(ctx, gauge, x.clone(), 2), _chain(ctx2, gauge2, x2.clone(), 2)]
    work, work2 = _work(ctx), _work(ctx2)
    y, z, y2, z2, both = (torch.empty_like(x) for _ in range(5))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        _normal(ctx, gauge, x, y, work)
        with torch.cuda.stream(side):
            _normal(ctx2, gauge2, x2, y2, work2)
            _normal(ctx2, gauge2, y2, z2, work2)
        main.wait_stream(side)      # the next operator follows two kernels
        _normal(ctx, gauge, y, z, work)
        both.copy_(z2)              # a copy, then an operator
        _normal(ctx, gauge, x, y, work)
        _normal(ctx, gauge, y, z, work)
    for _ in range(3):
        z.zero_()
        both.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(z, want[0]) and torch.equal(both, want[1])


def test_two_contexts_on_two_streams():
    a, b = _setup(54), _setup(55)
    want = [_chain(c, g, x.clone(), 12) for c, g, x in (a, b)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    state = []
    for k, (c, g, x) in enumerate((a, b)):
        state.append([x.clone(), torch.empty_like(x), _work(c)])
    torch.cuda.synchronize()
    for _ in range(12):
        for k, (c, g, _x) in enumerate((a, b)):
            _normal(c, g, state[k][0], state[k][1], state[k][2], stream=streams[k])
            state[k][0], state[k][1] = state[k][1], state[k][0]
    torch.cuda.synchronize()
    for k in range(2):
        assert torch.equal(state[k][0], want[k])
