"""Gauge force, link update and clover build of links near the identity (cold
starts, smooth and perturbative fields, short steps): what they compute is as
small as the links' vector parts and holds binary64's accuracy relative to
those, in fields that are weak everywhere, in part, or on one link.

Bounds: the native formulas make at most some 60 roundings of 2^-53 on terms as
large as the largest vector component they read (a scalar part near 1 times a vector
part), and so does the reference in torch or NumPy binary64.
"""

import numpy as np
import pytest

from oracle import hmc as ohmc
from tests.test_gpu_clover_slabs import CSW, M0, clover_times
from tests.test_gpu_gauge_force import links, reference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import fields, hr  # noqa: E402

ULP = 2.0 ** -52


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return hr.Context(0)


def weak_links(dims, kind, seed):
    """Unit links on the device: 1 + eps noise, or partly rough."""
    q = links(dims, seed)  # Haar
    V = q.shape[1]
    eps = kind if isinstance(kind, float) else 1e-7
    w = torch.zeros_like(q)
    w[..., 1:] = eps * q[..., 1:]
    w[..., 0] = (1.0 - (w[..., 1:] ** 2).sum(-1)).sqrt()
    if kind == "half":  # weak in the first half of the time slices
        w[:, V // 2:] = q[:, V // 2:]
    elif kind == "one":  # the identity but for one link
        keep = w[2, V // 3].clone()
        w.zero_()
        w[..., 0] = 1.0
        w[2, V // 3] = keep
    elif kind == "cold":
        w.zero_()
        w[..., 0] = 1.0
    return w


def neighbourhood(q, dims):
    """Per link: the largest vector component among the links of its six plaquettes."""
    n = q[..., 1:].abs().amax(-1).reshape(4, *dims)
    out = []
    for mu in range(4):
        m = n[mu]
        for nu in range(4):
            if nu != mu:
                ahead = torch.roll(n[nu], -1, mu)
                for t in (n[nu], ahead, torch.roll(n[mu], -1, nu), torch.roll(n[nu], 1, nu), torch.roll(n[mu], 1, nu),
                          torch.roll(ahead, 1, nu)):
                    m = torch.maximum(m, t)
        out.append(m)
    return torch.stack(out).reshape(4, -1, 1)


KINDS = [0.2, 0.05, 1e-3, 1e-6, 1e-13, "half", "one", "cold"]


# one thread per link and per site, several slabs, slices too large for the scratch
@pytest.mark.parametrize("dims", [(4, 2, 6, 10), (22, 18, 20, 18), (4, 60, 60, 64), (2, 64, 64, 64)])
@pytest.mark.parametrize("kind", KINDS)
def test_gauge_force(ctx, dims, kind):
    q = weak_links(dims, kind, 41)
    F = torch.zeros((4, q.shape[1], 3), dtype=torch.float64, device="cuda")
    hr.hr_gauge_force(ctx, dims, 2.3, q, 1.0, F)
    err = (F - reference(q, dims, 2.3)).abs()
    assert bool((err <= 64 * 2.3 * ULP * neighbourhood(q, dims)).all())


def test_gauge_force_unaligned(ctx):
    dims = (18, 16, 20, 26)
    q = weak_links(dims, "half", 42)
    buf = torch.empty(q.numel() + 1, dtype=torch.float64, device="cuda")
    buf[1:] = q.reshape(-1)
    F = torch.full((4, q.shape[1], 3), 0.0, dtype=torch.float64, device="cuda")
    hr.hr_gauge_force(ctx, dims, 2.3, buf[1:].reshape(q.shape), 1.0, F)
    assert bool(((F - reference(q, dims, 2.3)).abs() <= 64 * 2.3 * ULP * neighbourhood(q, dims)).all())


@pytest.mark.parametrize("eps", [0.3, 1e-3, 1e-12, 1e-18, 1e-200, 0.0])
@pytest.mark.parametrize("kind", [0.2, 1e-6, 1e-13, "half", "cold"])
def test_link_update(ctx, kind, eps):
    dims = (6, 4, 2, 8)
    q = weak_links(dims, kind, 43).cpu().numpy()
    p = np.random.default_rng(44).normal(size=(4, q.shape[1], 3))
    p[1, 5] = 0.0
    qd = torch.tensor(q, device="cuda")
    hr.hr_link_update(ctx, dims, eps, torch.tensor(p, device="cuda"), qd)
    got, want = qd.cpu().numpy(), ohmc.link_update(q, p, eps)
    size = np.maximum(np.abs(q[..., 1:]).max(-1), 0.5 * eps * np.abs(p).max(-1))
    assert np.abs(got[..., 0] - want[..., 0]).max() <= 16 * ULP
    assert np.all(np.abs(got[..., 1:] - want[..., 1:]) <= 16 * ULP * size[..., None])


def test_short_steps_from_the_identity_add_up(ctx):
    dims = (4, 4, 4, 4)
    q = weak_links(dims, "cold", 45)
    p = torch.randn((4, q.shape[1], 3), dtype=torch.float64, device="cuda")
    for _ in range(100):
        hr.hr_link_update(ctx, dims, 2e-17, p, q)
    assert (q[..., 1:] - 1e-15 * p).abs().max().item() <= 1e-12 * 1e-15 * p.abs().max().item()


def columns(ctx, dims, clover, inverse=False, only=range(8)):
    """A or A^-1 of every site: [V, 8, 8], column 2 spin + colour (the others zero)."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    out = torch.zeros((V, 8, 8), dtype=torch.complex128, device="cuda")
    for c in only:
        psi = torch.zeros((V, 4, 2), dtype=torch.complex128, device="cuda")
        psi.reshape(V, 8)[:, c] = 1.0
        for parity in (hr.HR_EVEN, hr.HR_ODD):
            x = fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, parity, psi)
            y = fields.empty_spinor(dims, hr.HR_FUND, hr.HR_F64, parity)
            hr.hr_clover_apply(ctx, dims, hr.HR_FUND, hr.HR_F64, parity, inverse, 1, clover, x, y)
            out[:, :, c] += fields.unpack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, parity, y).reshape(V, 8)
    return out


def build(ctx, dims, q, kind=hr.HR_CLOVER_SW, m0=M0, c_sw=CSW):
    return fields.build_clover(ctx, dims, hr.HR_FUND, hr.HR_F64, kind, m0, c_sw, q)


# slabs, and slices too large for the scratch
@pytest.mark.parametrize("dims", [(4, 6, 4, 8), (24, 28, 26, 28), (2, 64, 64, 64)])
@pytest.mark.parametrize("kind", [0.1, 1e-5, 1e-9, 1e-14, "half", "one", "cold"])
def test_clover_build(ctx, dims, kind):
    """Off-diagonal numbers of A (the diagonal: test_gpu_clover_slabs)."""
    q = weak_links(dims, kind, 46)
    V = q.shape[1]
    clover = build(ctx, dims, q)
    # the leaves of a site read the links within one step in two directions
    near = q[..., 1:].abs().amax(-1).amax(0).reshape(dims)
    for mu in range(4):
        near = torch.maximum(near, torch.maximum(torch.roll(near, 1, mu), torch.roll(near, -1, mu)))
    near = near.reshape(V, 1)
    for c in (0, 7):
        psi = torch.zeros((V, 4, 2), dtype=torch.complex128, device="cuda")
        psi.reshape(V, 8)[:, c] = 1.0
        want = clover_times(q, dims, psi).reshape(V, 8)
        err = (columns(ctx, dims, clover, only=(c,))[:, :, c] - want).abs()
        err[:, c] = 0.0
        # the packed pairs hold 2^-48 of each number
        assert bool((err <= 64 * ULP * near + 2.0 ** -47 * want.abs()).all())


@pytest.mark.parametrize("eps", [1e-3, 1e-7, 1e-12])
def test_clover_inverse_and_exponential(ctx, eps):
    """Off-diagonal numbers of A^-1 and of both forms of the exponential, from X = A / a - 1
    of the linear form (test_clover_build) and their power series."""
    dims = (4, 6, 4, 8)
    q = weak_links(dims, eps, 48)
    a = 4.0 + M0
    lin, exp = build(ctx, dims, q), build(ctx, dims, q, hr.HR_CLOVER_EXP)
    one = torch.eye(8, dtype=torch.complex128, device="cuda")
    X = columns(ctx, dims, lin) / a - one
    assert X.abs().max().item() < 8 * eps

    def series(coefficients):
        s, p = torch.zeros_like(X), one.expand_as(X)
        for c in coefficients:
            s, p = s + c * p, p @ X
        return s

    fact = [1.0, 1.0, 1 / 2, 1 / 6, 1 / 24, 1 / 120, 1 / 720]
    for clover, inverse, want in ((lin, True, series([(-1.0) ** k for k in range(7)]) / a),
                                  (exp, False, series(fact) * a),
                                  (exp, True, series([f * (-1.0) ** k for k, f in enumerate(fact)]) / a)):
        err = (columns(ctx, dims, clover, inverse) - want).abs() * (1.0 - one.real)
        # X and the result are pairs of 2^-48 of numbers up to 8 eps, X's diagonal 2^-48 of 1
        assert err.max().item() <= 2.0 ** -46 * 8 * eps * a


@pytest.mark.parametrize("c_sw", [1e-3, 1e-9, 1e-13])
def test_clover_build_small_coefficient(ctx, c_sw):
    """A's off-diagonal numbers scale with c_sw."""
    dims = (4, 6, 4, 8)
    q = links(dims, 47)
    off = 1.0 - torch.eye(8, dtype=torch.float64, device="cuda")
    full, small = (columns(ctx, dims, build(ctx, dims, q, c_sw=c)) * off for c in (1.0, c_sw))
    # two pairs of 2^-48 each, on numbers up to 2
    assert (small - c_sw * full).abs().max().item() <= 2.0 ** -45 * c_sw


def test_clover_build_rows_of_different_size(ctx):
    """Planes (0 1) and (2 3) smooth beside rough ones: A's numbers of the row they make
    are small beside the others of the block."""
    dims = (4, 6, 4, 8)
    V = 4 * 6 * 4 * 8
    q = torch.zeros((4, V, 4), dtype=torch.float64, device="cuda")
    x = torch.tensor([[i // (6 * 4 * 8) % 4, i // 32 % 6, i // 8 % 4, i % 8] for i in range(V)], device="cuda")
    noise = links(dims, 49)[..., 1:] * 1e-8
    for mu in range(4):  # diagonal links, the field strengths F_02 and F_13 of order 1
        angle = 0.7 * torch.sin(x[:, {0: 2, 1: 3, 2: 0, 3: 1}[mu]].double() + mu)
        q[mu, :, 0], q[mu, :, 3] = angle.cos(), angle.sin()
        q[mu, :, 1:] += noise[mu]
    q /= q.norm(dim=-1, keepdim=True)
    psi = torch.zeros((V, 4, 2), dtype=torch.complex128, device="cuda")
    psi[:, 0, 0] = 1.0
    want = clover_times(q, dims, psi).reshape(V, 8)
    got = columns(ctx, dims, build(ctx, dims, q), only=(0,))[:, :, 0]
    err = (got - want).abs()
    err[:, 0] = 0.0
    assert bool((err <= 64 * ULP + 2.0 ** -47 * want.abs()).all())
