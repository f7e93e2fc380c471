"""The gradient energy where |k|^2 |c_hat|^2, or |c_hat|^2 itself, leaves FP32: very small
voxels (h = 4e-18: |k|^2 up to 2e36) and very small amplitudes (1e-23, with a kappa that
makes the gradient part the energy), against the oracle. 1e-5: FP32 transforms of the field."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_21748_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(300, 8, 12), (48, 40, 36), (64, 64, 64)])
@pytest.mark.parametrize("amp,h,kappa", [(0.4, 4e-18, 1.0), (1e-23, 1.0, 1e50)])
def test_energy(shape, amp, h, kappa):
    import torch
    from paper_2507_21748_gb300 import evx
    c0 = inputs.uniform_field(shape, seed=6, offset=0.0, lo=-amp, hi=amp)
    with evx.Grid(shape, dt=0.1, M=1.0, kappa=kappa, h=h) as g:
        g.set_field(torch.from_numpy(c0).cuda())
        E = g.energy()[0]
    ref = O.energy(c0, kappa, h)
    assert np.isfinite(E) and abs(E - ref) <= 1e-5 * abs(ref)
