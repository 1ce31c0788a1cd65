"""The fixed-point link derivatives over the value range: sites of very
different magnitude, zero sites, coherent spinors (the largest possible sums),
non-unit links, and fields below the fixed-point range (the native FP64 path),
each link against the oracle within the rounding of its own factors."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import hr, fields  # noqa: E402

DIMS = [(2, 2, 2, 2), (4, 2, 6, 10), (6, 4, 4, 8)]


def _fields(kind, dims, seed):
    V = int(np.prod(dims))
    rng = np.random.default_rng(seed)
    a, b = synth.gaussian_spinor(dims, 2, seed), synth.gaussian_spinor(dims, 2, seed + 1)
    if kind == "range":
        a = a * (2.0 ** rng.integers(-60, 61, V))[:, None, None]
        b = b * (2.0 ** rng.integers(-60, 61, V))[:, None, None]
    elif kind == "zeros":
        a[rng.random(V) < 0.5] = 0.0
        b[rng.random(V) < 0.5] = 0.0
    elif kind == "coherent":
        a[:], b[:] = 1.0 + 1.0j, -1.0 + 1.0j
    elif kind == "tiny":  # below 2^-105 on half of the sites: the native path beside the fixed-point one
        a[rng.random(V) < 0.5] *= 2.0 ** -112
    return a, b


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("kind", ["gauss", "range", "zeros", "coherent", "tiny"])
def test_link_derivatives_over_the_value_range(dims, kind):
    ctx = hr.Context(0)
    V = int(np.prod(dims))
    q = synth.haar_links(dims, 61)
    if kind == "gauss":
        q = q * np.random.default_rng(5).uniform(0.01, 30.0, (4, V, 1))  # hr_force is linear in the links
    a, b = _fields(kind, dims, 62)
    dev = fields.spinor_to_device
    gauge = fields.pack_gauge(ctx, dims, hr.HR_FUND, hr.HR_F64, fields.gauge_to_device(q))
    ap = fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, dev(a))
    bp = fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, dev(b))
    # what the pairs hold: 48 bits (less below 2^-102)
    a = fields.unpack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, ap).cpu().numpy()
    b = fields.unpack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, bp).cpu().numpy()
    F = torch.zeros((4, V, 3), dtype=torch.float64, device="cuda")
    G = torch.zeros((4, V, 4), dtype=torch.float64, device="cuda")
    hr.hr_force(ctx, dims, gauge, ap, bp, 1.0, F)
    hr.hr_link_grad(ctx, dims, ap, bp, 1.0, G)
    wantg = oracle.link_grad(dims, a, b)
    u = q[:, :, 1:]
    wantf = 0.5 * (q[:, :, :1] * wantg[:, :, 1:] - wantg[:, :, :1] * u - np.cross(u, wantg[:, :, 1:]))
    na, nb = np.sqrt((np.abs(a) ** 2).sum((1, 2))).reshape(dims), np.sqrt((np.abs(b) ** 2).sum((1, 2))).reshape(dims)
    for mu in range(4):
        # 32 products of factors rounded at 2^-48 (links) or better: 2^-45 of the two terms' norms
        bound = (na * np.roll(nb, -1, mu) + np.roll(na, -1, mu) * nb).reshape(V, 1) * 2.0 ** -45 + 1e-300
        assert np.all(np.abs(G[mu].cpu().numpy() - wantg[mu]) <= bound)
        size = np.linalg.norm(q[mu], axis=1, keepdims=True)
        assert np.all(np.abs(F[mu].cpu().numpy() - wantf[mu]) <= bound * size)
    ctx.close()


def test_nan_and_inf_reach_the_links_that_hold_them():
    ctx, dims = hr.Context(0), (4, 4, 2, 4)
    V = int(np.prod(dims))
    a, b = _fields("gauss", dims, 70)
    a[5, 0, 0] = np.nan
    b[40, 2, 1] = np.inf
    dev = fields.spinor_to_device
    ap = fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, dev(a))
    bp = fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, dev(b))
    G = torch.zeros((4, V, 4), dtype=torch.float64, device="cuda")
    hr.hr_link_grad(ctx, dims, ap, bp, 1.0, G)
    got = ~torch.isfinite(G).all(-1).cpu().numpy()
    hit = np.zeros((4,) + dims, bool)
    for site in (5, 40):
        x = np.unravel_index(site, dims)
        for mu in range(4):
            hit[mu][x] = True
            y = list(x)
            y[mu] = (y[mu] - 1) % dims[mu]
            hit[mu][tuple(y)] = True
    assert np.array_equal(got, hit.reshape(4, V))
    ctx.close()
