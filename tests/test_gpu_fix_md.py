"""The fixed-point molecular-dynamics and clover-build kernels at the edges of
their range against the oracle: smallest extents, links off unit length and
long steps (the native FP64 path), 8-byte aligned fields, large clover
coefficients."""

import numpy as np
import pytest

import oracle
import synth
from oracle import clover as ocl
from oracle import hmc as ohmc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import hr, fields  # noqa: E402

DIMS = [(2, 2, 2, 2), (4, 2, 6, 10), (6, 4, 2, 8)]


def _dev(a, offset=False):
    """The array on the device, 16-byte aligned or (offset) only 8-byte aligned."""
    t = torch.as_tensor(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    if not offset:
        return t
    buf = torch.empty(t.numel() + 1, dtype=torch.float64, device="cuda")
    v = buf[1:].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 8
    return v


def _links(dims, kind, seed):
    q = synth.haar_links(dims, seed)
    if kind == "mixed":  # a few links off unit length: native FP64 beside fixed point
        q = q.copy()
        q[1, 3] *= 1.25
        q[3, 0] *= 0.5
    return q


@pytest.mark.parametrize("offset", [False, True])
@pytest.mark.parametrize("kind", ["unit", "mixed"])
@pytest.mark.parametrize("dims", DIMS)
def test_gauge_force(dims, kind, offset):
    ctx = hr.Context(0)
    q = _links(dims, kind, 81)
    F = torch.ones((4, q.shape[1], 3), dtype=torch.float64, device="cuda")
    hr.hr_gauge_force(ctx, dims, 2.2, _dev(q, offset), -0.5, F)
    want = 1.0 - 0.5 * ohmc.gauge_force(dims, q, 2.2)
    # six staples of three products each, 2^-52 per operation on values up to beta
    assert np.abs(F.cpu().numpy() - want).max() <= 64 * 2.2 * 2.0 ** -52
    ctx.close()


@pytest.mark.parametrize("offset", [False, True])
@pytest.mark.parametrize("eps", [0.0, 1e-9, 0.05, 0.5, 30.0])
@pytest.mark.parametrize("dims", DIMS)
def test_link_update(dims, eps, offset):
    ctx = hr.Context(0)
    q = synth.haar_links(dims, 82)
    p = np.random.default_rng(83).normal(size=(4, q.shape[1], 3))
    p[0, 0] = 0.0
    qd = _dev(q, offset)
    hr.hr_link_update(ctx, dims, eps, _dev(p), qd)
    got = qd.cpu().numpy()
    # the angle eps |p| / 2 rounds at 2^-52 of itself
    assert np.abs(got - ohmc.link_update(q, p, eps)).max() <= (16 + eps * np.abs(p).max() * 4) * 2.0 ** -52
    assert np.abs((got ** 2).sum(-1) - 1.0).max() <= 8 * 2.0 ** -52
    ctx.close()


def test_link_update_renormalises_any_length():
    ctx, dims = hr.Context(0), (4, 2, 6, 10)
    q = _links(dims, "mixed", 84)
    p = np.random.default_rng(85).normal(size=(4, q.shape[1], 3))
    qd = _dev(q)
    hr.hr_link_update(ctx, dims, 0.1, _dev(p), qd)
    unit = q / np.sqrt((q ** 2).sum(-1, keepdims=True))
    assert np.abs(qd.cpu().numpy() - ohmc.link_update(unit, p, 0.1)).max() <= 32 * 2.0 ** -52
    ctx.close()


@pytest.mark.parametrize("prec", [hr.HR_F64, hr.HR_F32])
@pytest.mark.parametrize("kind", [hr.HR_CLOVER_SW, hr.HR_CLOVER_EXP])
@pytest.mark.parametrize("m0,csw", [(-0.2, 1.0), (0.3, -0.7), (40.0, 1.3), (-3.0, 1.0), (0.0, 9.0), (-5.5, 0.4)])
@pytest.mark.parametrize("dims", DIMS)
def test_clover_build(dims, m0, csw, kind, prec):
    """A and A^-1 applied to a full set of spinors: within the fixed-point range
    (the first three), across it (a site block close to singular or a large
    exponent) and outside it (4 + m0 < 0)."""
    ctx = hr.Context(0)
    q = _links(dims, "unit", 86)
    qd = fields.gauge_to_device(q)
    L = oracle.expand_links(dims, 2, q)
    A = ocl.site_term(dims, L, m0, csw, kind)
    clov = fields.build_clover(ctx, dims, hr.HR_FUND, prec, kind, m0, csw, qd)
    psi = synth.gaussian_spinor(dims, 2, 87)
    tol = 2e-14 if prec == hr.HR_F64 else 2e-6
    for parity in (hr.HR_EVEN, hr.HR_ODD):
        src = fields.pack_spinor(ctx, dims, hr.HR_FUND, prec, parity, fields.spinor_to_device(psi))
        dst = fields.empty_spinor(dims, hr.HR_FUND, prec, parity)
        mask = fields.unpack_spinor(ctx, dims, hr.HR_FUND, prec, parity, src).cpu().numpy() != 0
        for inverse in (False, True):
            hr.hr_clover_apply(ctx, dims, hr.HR_FUND, prec, parity, inverse, 1, clov, src, dst)
            got = fields.unpack_spinor(ctx, dims, hr.HR_FUND, prec, parity, dst).cpu().numpy()
            M = np.linalg.inv(A) if inverse else A
            want = ocl.apply_site(M, psi * mask)
            size = np.linalg.norm(M, axis=(-2, -1)).max() * np.abs(psi).max() * 4
            # an inverse carries the site's condition number
            cond = np.linalg.cond(A).max() if inverse else 1.0
            assert np.abs(got - want).max() <= tol * size * cond
    ctx.close()


@pytest.mark.parametrize("links", ["unit", "mixed"])
@pytest.mark.parametrize("kind", ["gauss", "range", "zeros"])
@pytest.mark.parametrize("dims", DIMS)
def test_clover_insertion_force(dims, kind, links):
    """Insertions of very different magnitude from site to site: each link within
    the rounding of the corners of its own plaquettes."""
    ctx = hr.Context(0)
    V = int(np.prod(dims))
    q = _links(dims, links, 88)
    rng = np.random.default_rng(89)
    lam = rng.normal(size=(V, 8, 8)) + 1j * rng.normal(size=(V, 8, 8))
    if kind == "range":
        lam *= (2.0 ** rng.integers(-40, 41, V))[:, None, None]
    elif kind == "zeros":
        lam[rng.random(V) < 0.7] = 0.0
    F = torch.zeros((4, V, 3), dtype=torch.float64, device="cuda")
    work = fields.empty_bytes(hr.hr_clover_force_workspace_bytes(dims))
    hr.hr_clover_insertion_force(ctx, dims, 1.3, _dev(q), torch.tensor(lam, device="cuda"), 0.7, F, work)
    want = 0.91 * ocl.clover_derivative(dims, oracle.expand_links(dims, 2, q), lam)
    n = np.linalg.norm(lam, axis=(1, 2)).reshape(dims)
    for rho in range(4):
        near = sum(np.roll(m, s, sig) for m in (n, np.roll(n, -1, rho)) for sig in range(4) for s in (-1, 0, 1))
        # about 150 products per plaquette of unit links (1.25^4 with the mixed ones)
        assert np.all(np.abs(F[rho].cpu().numpy() - want[rho]) <= 2.0 ** -45 * near.reshape(V, 1) + 1e-300)
    ctx.close()
