"""Within a segment an adjoint step reads Lambda as the two parts the step before left; at a
segment's end they are added up. With one step per segment only sums are read, with more the
parts: the same additions, so the gradients agree to the bit. Mixed-radix x lengths (the
oracle checks them in test_gpu_adjoint.py), with and without two-radix y and z, and a tuned one."""
import numpy as np
import pytest

from paper_2507_21748_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(972, 8, 10), (300, 18, 10), (24, 150, 288), (64, 20, 36)])
def test_parts_and_sums_agree(shape):
    import torch
    from paper_2507_21748_gb300 import evx
    c0 = torch.from_numpy(inputs.uniform_field(shape, seed=8, lo=-0.3, hi=0.3)).cuda()
    dL = torch.from_numpy(np.random.default_rng(1).standard_normal(shape).astype(np.float32)).cuda()
    with evx.Grid(shape, dt=0.1, M=1.0, kappa=1.0, h=1.0) as g:
        one = g.adjoint(c0, 5, 1, dL)
        for ckpt in (2, 5):
            d0, gk, gm = g.adjoint(c0, 5, ckpt, dL)
            assert torch.equal(d0, one[0]) and gk == one[1] and gm == one[2]
