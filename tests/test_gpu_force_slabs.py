"""Link derivatives whose fields' digits go through the scratch slab by slab: the
whole lattice at once, several slices, one slice a slab, slices too large for
the scratch, against torch's derivative of Re<a, H b> in FP64.

The packed fields carry 2^-49 of each number, a component of the gradient sums 64
products of two of them: about 1e-14 in root mean square for unit Gaussians, up
to some 3e-13 over ten million components; the largest component is near 60, hence
1e-14 of it.
"""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import fields, hr  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return hr.Context(0)


def gammas():
    s = torch.tensor([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=torch.complex128)
    z, e = torch.zeros((2, 2), dtype=torch.complex128), torch.eye(2, dtype=torch.complex128)
    return [torch.cat((torch.cat((z, e), 1), torch.cat((e, z), 1)))] + \
           [torch.cat((torch.cat((z, -1j * k), 1), torch.cat((1j * k, z), 1))) for k in s]


def gradient(q, a, b, dims, mu):
    """d Re<a, H b> / dq[mu], one direction (the memory of four would be wasted)."""
    qm = q[mu].clone().requires_grad_(True)
    a0, a1, a2, a3 = qm.unbind(-1)
    U = torch.stack((torch.complex(a0, a3), torch.complex(a2, a1), torch.complex(-a2, a1), torch.complex(a0, -a3)),
                    -1).reshape(-1, 1, 2, 2)
    g = gammas()[mu].to(q.device)
    one = torch.eye(4, dtype=torch.complex128, device=q.device)

    def up(v):
        return torch.roll(v.reshape(*dims, 4, 2), -1, mu).reshape(-1, 4, 2)

    def mul(M, v):
        return (M @ v.unsqueeze(-1)).squeeze(-1)

    f = (a.conj() * torch.einsum("st,vtc->vsc", one - g, mul(U, up(b)))).sum().real
    f = f + (up(a).conj() * torch.einsum("st,vtc->vsc", one + g, mul(U.mH, b))).sum().real
    return torch.autograd.grad(f, qm)[0]


@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (16, 18, 14, 20), (32, 32, 30, 28), (4, 48, 48, 50), (6, 60, 50, 44)])
def test_gradient_and_force(ctx, dims):
    g = torch.Generator(device="cuda")
    g.manual_seed(21)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    q = torch.randn((4, V, 4), dtype=torch.float64, device="cuda", generator=g)
    q /= q.norm(dim=-1, keepdim=True)
    a, b = (torch.randn((V, 4, 2), dtype=torch.complex128, device="cuda", generator=g) * 2 ** 0.5 for _ in range(2))
    pa, pb = (fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, v) for v in (a, b))
    grad = torch.full_like(q, 0.5)
    hr.hr_link_grad(ctx, dims, pa, pb, -0.75, grad)
    force = torch.zeros((4, V, 3), dtype=torch.float64, device="cuda")
    gauge = fields.pack_gauge(ctx, dims, hr.HR_FUND, hr.HR_F64, q)
    hr.hr_force(ctx, dims, gauge, pa, pb, 1.0, force)
    for mu in range(4):
        G = gradient(q, a, b, dims, mu)
        top = G.abs().max().item()
        assert (grad[mu] - 0.5 + 0.75 * G).abs().max().item() <= 1e-14 * top
        # U -> exp(i w.s/2) U: F = (q0 G - G0 q - q x G) / 2 on the vector parts
        F = (q[mu, :, :1] * G[:, 1:] - G[:, :1] * q[mu, :, 1:] - torch.cross(q[mu, :, 1:], G[:, 1:], dim=1)) / 2
        assert (force[mu] - F).abs().max().item() <= 1e-14 * top
