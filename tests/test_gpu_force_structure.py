"""Link derivatives of zero fields beside very small links."""

import numpy as np
import pytest

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
