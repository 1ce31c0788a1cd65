"""Link derivatives of fields whose spins differ much in size within a site, so that
a link's derivative is far below the product of the largest components, and of zero
fields beside very small links."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2411_18511_gb300 import fields, hr  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return hr.Context(0)


def _pack(ctx, dims, v):
    return fields.pack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, fields.spinor_to_device(v))


# the whole lattice in the scratch, slabs of it, slices too large for it
@pytest.mark.parametrize("dims", [(4, 2, 6, 10), (6, 60, 50, 44), (2, 64, 64, 64)])
@pytest.mark.parametrize("small", [2.0 ** -6, 2.0 ** -20, 2.0 ** -40])
def test_spins_of_different_size(ctx, dims, small):
    """a large where b is small: spins 0 and 2 of a, 1 and 3 of b.  Directions 0 and 3
    pair spins (0, 2) and (1, 3) only, so their derivatives are of the size `small`."""
    V = int(np.prod(dims))
    a, b = synth.gaussian_spinor(dims, 2, 91), synth.gaussian_spinor(dims, 2, 92)
    a[:, 1::2] *= small
    b[:, 0::2] *= small
    ap, bp = _pack(ctx, dims, a), _pack(ctx, dims, b)
    # what the pairs hold
    a, b = (fields.unpack_spinor(ctx, dims, hr.HR_FUND, hr.HR_F64, hr.HR_FULL, v).cpu().numpy() for v in (ap, bp))
    q = synth.haar_links(dims, 93)
    gauge = fields.pack_gauge(ctx, dims, hr.HR_FUND, hr.HR_F64, fields.gauge_to_device(q))
    G = torch.zeros((4, V, 4), dtype=torch.float64, device="cuda")
    F = torch.zeros((4, V, 3), dtype=torch.float64, device="cuda")
    hr.hr_link_grad(ctx, dims, ap, bp, 1.0, G)
    hr.hr_force(ctx, dims, gauge, ap, bp, 1.0, F)
    wantg = oracle.link_grad(dims, a, b)
    u = q[:, :, 1:]
    wantf = 0.5 * (q[:, :, :1] * wantg[:, :, 1:] - wantg[:, :, :1] * u - np.cross(u, wantg[:, :, 1:]))

    def size(v, s):  # norm of one of the two spins that a direction pairs
        return np.sqrt((np.abs(v[:, s::2]) ** 2).sum((1, 2))).reshape(dims)

    for mu in range(4):
        # 32 products of numbers that carry 2^-48 (links) or are exact (fields): 2^-45 of
        # the terms' sizes, spin by spin where the direction pairs these two
        split = (0, 1) if mu in (0, 3) else (slice(None),)
        bound = 0.0
        for s in split:
            na, nb = (size(v, s) if isinstance(s, int) else np.sqrt((np.abs(v) ** 2).sum((1, 2))).reshape(dims)
                      for v in (a, b))
            bound = bound + na * np.roll(nb, -1, mu) + np.roll(na, -1, mu) * nb
        bound = bound.reshape(V, 1) * 2.0 ** -45
        assert np.all(np.abs(G[mu].cpu().numpy() - wantg[mu]) <= bound)
        assert np.all(np.abs(F[mu].cpu().numpy() - wantf[mu]) <= bound)


@pytest.mark.parametrize("dims", [(4, 2, 6, 10), (2, 64, 64, 64)])
def test_zero_fields_leave_the_force_alone(ctx, dims):
    """Links of any size and zero fields: nothing is added."""
    V = int(np.prod(dims))
    q = synth.haar_links(dims, 94) * (2.0 ** (np.arange(V) % 80 - 79.0))[None, :, None]
    gauge = fields.pack_gauge(ctx, dims, hr.HR_FUND, hr.HR_F64, fields.gauge_to_device(q))
    z = _pack(ctx, dims, np.zeros((V, 4, 2), complex))
    F = torch.full((4, V, 3), 0.75, dtype=torch.float64, device="cuda")
    hr.hr_force(ctx, dims, gauge, z, z, 1.0, F)
    assert bool((F == 0.75).all())
