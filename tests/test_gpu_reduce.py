"""Grid reductions of the solvers (a row of sums per block, one finishing
launch) at the sizes where their shape changes: one block and one row, more
rows than one finishing block adds (2048 sums), grids capped by the scratch,
and solve loops that stop inside a group of iterations or a pass.

The reported residual is compared with |b - A x| of the returned x, summed by
torch in FP64.  Both sides carry the operator's error, about 1e-14 of |A x|,
and after a few iterations |b - A x| is above 1e-3 |b|, hence 1e-10.
"""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import fields, hr  # noqa: E402

M0 = 0.3


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return hr.Context(0)


def problem(ctx, dims, n_rhs, seed=3):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    q = torch.randn((4, V, 4), dtype=torch.float64, device="cuda", generator=g)
    q /= q.norm(dim=-1, keepdim=True)
    shape = ((n_rhs,) if n_rhs > 1 else ()) + (V, 4, 2)
    b = torch.randn(shape, dtype=torch.complex128, device="cuda", generator=g)
    return (fields.pack_gauge(ctx, dims, hr.HR_FUND, hr.HR_F64, q),
            fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, b))


def solve(ctx, dims, n_rhs, inner, maxiter, check_every, gauge, b, delta=1e-2, tol=1e-10):
    opts = hr.hr_solver_default_opts()
    opts.inner_prec, opts.n_rhs, opts.maxiter, opts.check_every = inner, n_rhs, maxiter, check_every
    opts.reliable_delta, opts.tol = delta, tol
    x = fields.zeros_spinor(dims, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, n_rhs)
    work = fields.empty_bytes(hr.hr_cg_workspace_bytes(dims, hr.HR_FUND, opts))
    _, info = hr.hr_cg_solve(ctx, dims, M0, hr.HR_FUND, opts, gauge, b, x, work)
    return x, info


@pytest.mark.parametrize("dims,n_rhs", [((4, 4, 4, 4), 1), ((8, 6, 4, 10), 1), ((4, 4, 4, 4), 32), ((16, 16, 16, 16), 1),
                                        ((24, 26, 28, 30), 1), ((32, 32, 32, 34), 1), ((12, 10, 14, 8), 16),
                                        ((24, 24, 22, 26), 16), ((32, 24, 24, 24), 32), ((48, 48, 40, 40), 1)])
def test_reported_residual(ctx, dims, n_rhs):
    gauge, b = problem(ctx, dims, n_rhs)
    x, info = solve(ctx, dims, n_rhs, hr.HR_F64, 3, 0, gauge, b)
    assert info.iters == 3
    ax = fields.empty_spinor(dims, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, n_rhs)
    work = fields.empty_bytes(hr.hr_dirac_workspace_bytes(dims, hr.HR_FUND, hr.HR_F64, hr.HR_OP_NORMAL, n_rhs))
    hr.hr_dirac_eo(ctx, dims, M0, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, hr.HR_OP_NORMAL, n_rhs, gauge, x, ax, work)

    def plain(v):
        u = fields.unpack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_EVEN, v, n_rhs)
        return torch.view_as_real(u).reshape(n_rhs, -1)

    pb = plain(b)
    rel = ((pb - plain(ax)).norm(dim=1) / pb.norm(dim=1)).max().item()
    assert 1e-3 < rel < 1.0
    assert abs(info.true_rel_residual - rel) <= 1e-10 * rel


@pytest.mark.parametrize("maxiter", [1, 2, 3, 4, 5, 7, 8, 9, 13])
@pytest.mark.parametrize("inner", [hr.HR_F64, hr.HR_F32, hr.HR_F16])
def test_iteration_cap_in_both_loops(ctx, inner, maxiter):
    """The cap falls anywhere in a pass of 8 and a group of 4 iterations; delta
    0.5 makes nearly every iteration a reliable update, so that the others skip."""
    dims = (8, 8, 4, 6)
    gauge, b = problem(ctx, dims, 1)
    for delta in (0.5, 1e-2):
        x0, i0 = solve(ctx, dims, 1, inner, maxiter, 0, gauge, b, delta)
        x1, i1 = solve(ctx, dims, 1, inner, maxiter, 1, gauge, b, delta)
        assert i0.iters == i1.iters == maxiter
        # an update due at the cap itself runs in the chunked loop only; for the
        # binary16 solver it then adds the pending increments in another order
        if inner != hr.HR_F16:
            assert torch.equal(x0, x1)


@pytest.mark.parametrize("n_rhs", [1, 4])
@pytest.mark.parametrize("inner,delta", [(hr.HR_F64, 0.1), (hr.HR_F32, 0.5), (hr.HR_F32, 1e-4), (hr.HR_F16, 0.3),
                                         (hr.HR_F16, 1e-2)])
def test_loops_agree_to_convergence(ctx, inner, delta, n_rhs):
    dims = (8, 8, 8, 6)
    gauge, b = problem(ctx, dims, n_rhs, seed=5)
    x0, i0 = solve(ctx, dims, n_rhs, inner, 500, 0, gauge, b, delta)
    x1, i1 = solve(ctx, dims, n_rhs, inner, 500, 3, gauge, b, delta)
    assert i0.true_rel_residual <= 1e-10
    assert (i0.iters, i0.n_reliable_updates) == (i1.iters, i1.n_reliable_updates)
    assert torch.equal(x0, x1)
