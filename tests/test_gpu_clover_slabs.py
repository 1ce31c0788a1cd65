"""The clover build from plaquette vectors where they go through the scratch in
slabs of time slices: two slabs, one slice a slab, slices too large for the
scratch (links instead), unaligned links; A applied to a spinor against its definition
in torch FP64, and A^-1 after A.

The packed field holds 2^-48 of each number, as the operators of the other clover
tests: 1e-13 of the result's norm.
"""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import fields, hr  # noqa: E402

M0, CSW = 0.3, 1.1


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return hr.Context(0)


def qmul(a, b):
    a0, a1, a2, a3 = a.unbind(-1)
    b0, b1, b2, b3 = b.unbind(-1)
    return torch.stack((a0 * b0 - a1 * b1 - a2 * b2 - a3 * b3, a0 * b1 + b0 * a1 - (a2 * b3 - a3 * b2),
                        a0 * b2 + b0 * a2 - (a3 * b1 - a1 * b3), a0 * b3 + b0 * a3 - (a1 * b2 - a2 * b1)), -1)


def conj(a):
    return a * torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=a.dtype, device=a.device)


def gammas():
    s = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128)
    z, e = torch.zeros((2, 2), dtype=torch.complex128), torch.eye(2, dtype=torch.complex128)
    return [torch.cat((torch.cat((z, e), 1), torch.cat((e, z), 1)))] + \
           [torch.cat((torch.cat((z, -1j * k), 1), torch.cat((1j * k, z), 1))) for k in s]


def clover_times(q, dims, psi):
    """(4 + m0 + c_sw sum (i/2) sigma F) psi."""
    Q = q.reshape(4, *dims, 4)
    g = [m.cuda() for m in gammas()]
    out = (4.0 + M0) * psi
    for mu in range(4):
        for nu in range(mu + 1, 4):
            a, b = Q[mu], torch.roll(Q[nu], -1, mu)
            c, d = conj(torch.roll(Q[mu], -1, nu)), conj(Q[nu])
            p = qmul(qmul(a, b), qmul(c, d))
            p = p + torch.roll(qmul(qmul(b, c), qmul(d, a)), 1, mu)
            p = p + torch.roll(qmul(qmul(c, d), qmul(a, b)), (1, 1), (mu, nu))
            p = p + torch.roll(qmul(qmul(d, a), qmul(b, c)), 1, nu)
            v = p.reshape(-1, 4)[:, 1:] / 4.0
            zero = torch.zeros_like(v[:, 0])
            F = torch.stack((torch.complex(zero, v[:, 2]), torch.complex(v[:, 1], v[:, 0]),
                             torch.complex(-v[:, 1], v[:, 0]), torch.complex(zero, -v[:, 2])), -1).reshape(-1, 2, 2)
            s = 0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])
            out = out + CSW * 0.5j * torch.einsum("st,vtc->vsc", s, torch.einsum("vcd,vtd->vtc", F, psi))
    return out


@pytest.mark.parametrize("dims,shift", [((4, 6, 4, 8), 0), ((24, 28, 26, 28), 0), ((24, 28, 26, 28), 1),
                                        ((4, 48, 64, 64), 0), ((2, 64, 64, 64), 0)])
def test_site_term(ctx, dims, shift):
    g = torch.Generator(device="cuda")
    g.manual_seed(31)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    q = 0.4 * torch.randn((4, V, 4), dtype=torch.float64, device="cuda", generator=g)
    q[..., 0] += 1.0
    q /= q.norm(dim=-1, keepdim=True)
    buf = torch.empty(q.numel() + shift, dtype=torch.float64, device="cuda")
    links = buf[shift:].reshape(q.shape)
    links.copy_(q)
    psi = torch.randn((V, 4, 2), dtype=torch.complex128, device="cuda", generator=g)
    want = clover_times(q, dims, psi)
    F64, FUND = hr.HR_F64, hr.HR_FUND
    clover = fields.build_clover(ctx, dims, FUND, F64, hr.HR_CLOVER_SW, M0, CSW, links)
    total = torch.zeros_like(psi)
    for parity in (hr.HR_EVEN, hr.HR_ODD):
        x = fields.pack_spinor(ctx, dims, FUND, F64, parity, psi)
        y, z = (fields.empty_spinor(dims, FUND, F64, parity) for _ in range(2))
        hr.hr_clover_apply(ctx, dims, FUND, F64, parity, False, 1, clover, x, y)
        hr.hr_clover_apply(ctx, dims, FUND, F64, parity, True, 1, clover, y, z)
        back = fields.unpack_spinor(ctx, dims, FUND, F64, parity, z)
        keep = fields.unpack_spinor(ctx, dims, FUND, F64, parity, x)
        assert (back - keep).norm() <= 1e-13 * keep.norm()
        total += fields.unpack_spinor(ctx, dims, FUND, F64, parity, y)
    assert (total - want).norm() <= 1e-13 * want.norm()
