"""Modes whose denominator 1 + dt M kappa |k|^4 leaves FP32 are damped to zero on every
length: grids of very small voxels (SI units) come back as their mean, to the rounding of
the FP32 field (2^-24 of |c| <= 1, and the transform's 2^-20). h = 1e-10: |k|^4 reaches
1e42; h = 1e-20: |k|^2 itself is infinite (Allen-Cahn's denominator)."""
import numpy as np
import pytest

from paper_2507_21748_gb300 import inputs

pytestmark = pytest.mark.gpu

# two radices along x (300, 486), grouped stages (40), four-step (64, 256)
LENGTHS = [300, 486, 40, 64, 256]


@pytest.mark.parametrize("nx", LENGTHS)
@pytest.mark.parametrize("model,h", [("ch", 1e-10), ("block", 1e-10), ("ac", 1e-20)])
def test_field_stays_finite(nx, model, h):
    import torch
    from paper_2507_21748_gb300 import evx
    shape = (nx, 8, 12)
    c0 = inputs.uniform_field(shape, seed=4, offset=0.1, lo=-0.4, hi=0.4)
    with evx.Grid(shape, dt=0.1, M=1.0, kappa=1.0, h=h, model="ac" if model == "ac" else "ch") as g:
        g.set_field(torch.from_numpy(c0).cuda())
        if model == "block":
            g.block(5)
        else:
            g.step(3)
        out, mean = g.get_field().cpu().numpy(), g.mean()
    assert np.isfinite(out).all()
    assert np.abs(out - mean).max() <= 2e-6
