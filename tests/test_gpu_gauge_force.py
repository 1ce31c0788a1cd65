"""The gauge force from plaquette vectors against its definition in torch FP64:
slabs of time slices (the whole lattice, several, one slice each, slices too
large for the scratch), one thread per site and one per link, unaligned links,
links off unit length, accumulation into a nonzero force.

The reference's six staples of three products each carry at most about 8e-15 in
FP64 (12 roundings of 1.1e-16 a staple and its sum), the fixed-point kernels
less; both are scaled by beta / 2, hence 1e-14 beta.
"""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import hr  # noqa: E402


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


def reference(q, dims, beta):
    Q = q.reshape(4, *dims, 4)
    out = []
    for mu in range(4):
        S = 0
        for nu in range(4):
            if nu == mu:
                continue
            up = qmul(qmul(torch.roll(Q[nu], -1, mu), conj(torch.roll(Q[mu], -1, nu))), conj(Q[nu]))
            dn = qmul(qmul(conj(torch.roll(Q[nu], -1, mu)), conj(Q[mu])), Q[nu])
            S = S + up + torch.roll(dn, 1, nu)
        out.append(0.5 * beta * qmul(Q[mu], S)[..., 1:])
    return torch.stack(out).reshape(4, -1, 3)


def links(dims, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    q = torch.randn((4, V, 4), dtype=torch.float64, device="cuda", generator=g)
    return q / q.norm(dim=-1, keepdim=True)


def check(ctx, dims, q, beta=2.3, coeff=-0.7):
    F = torch.full((4, q.shape[1], 3), 0.25, dtype=torch.float64, device="cuda")
    hr.hr_gauge_force(ctx, dims, beta, q, coeff, F)
    err = (F - 0.25 - coeff * reference(q, dims, beta)).abs().max().item()
    assert err <= 1e-14 * beta


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 4), (6, 2, 10, 4), (18, 20, 16, 18), (22, 18, 20, 18),
                                  (32, 40, 40, 40), (34, 24, 36, 30), (4, 60, 60, 64), (6, 2, 300, 300),
                                  (2, 64, 64, 64), (48, 4, 4, 4)])
def test_shapes(ctx, dims):
    check(ctx, dims, links(dims, 11))


@pytest.mark.parametrize("dims", [(8, 6, 4, 6), (20, 18, 20, 20)])
def test_links_outside_the_fast_range(ctx, dims):
    """Off unit length below and above the correction's limit of 2^-29, beyond
    1 %, components above 2, and a zero link."""
    q = links(dims, 12)
    for k, f in enumerate((1 + 4e-10, 1 - 9e-10, 1 + 1.1e-9, 1 - 1e-6, 1.004, 0.9, 1.7, 5.0, 0.0)):
        q[k % 4, 7 + 13 * k] *= f
    F = torch.zeros((4, q.shape[1], 3), dtype=torch.float64, device="cuda")
    hr.hr_gauge_force(ctx, dims, 2.0, q, 1.0, F)
    ref = reference(q, dims, 2.0)
    # sizes up to 5: the bound scales with the largest staple
    assert (F - ref).abs().max().item() <= 2e-14 * max(1.0, ref.abs().max().item())


def test_unaligned_links(ctx):
    for dims in [(8, 6, 4, 6), (18, 20, 20, 20)]:
        q = links(dims, 13)
        buf = torch.empty(q.numel() + 1, dtype=torch.float64, device="cuda")
        buf[1:] = q.reshape(-1)
        check(ctx, dims, buf[1:].reshape(q.shape))
