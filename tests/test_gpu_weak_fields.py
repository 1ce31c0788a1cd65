"""Gauge force and link update of links near the identity (cold
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
from tests.test_gpu_gauge_force import links, reference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import hr  # noqa: E402

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
