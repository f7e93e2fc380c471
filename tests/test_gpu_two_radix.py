"""The two-radix passes (csrc/evx_mixed_*.cu) by value against the FP64 oracle: every class of
kernels (largest radix 12, 16, 20 or 32, second radix up to 16 and above), every radix as
either factor along some axis, every mode: solver step, Allen-Cahn step with its mean, the
preconditioner, the block propagator, the adjoint, the energies, the transforms alone. An
edge above 128 keeps its axis off the grouped-stage kernels; the factors below 12 appear on
grids of more than 2^22 voxels, which take none of those. The lengths without two radices (972 and
1000 along x and y) are here too.

Bars as in the models' own tests: relative L2 1e-5 of the field and 1e-4 of its increment
after a step, 1e-5 of the energy, 1e-9 of the Allen-Cahn mean, 1e-4 of the gradients."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_21748_gb300 import inputs

pytestmark = pytest.mark.gpu

XY = [(162, 180, 20), (240, 300, 8), (300, 384, 12), (324, 600, 10), (486, 640, 8), (750, 216, 10), (900, 144, 12),
      (960, 324, 8), (8, 768, 18), (972, 8, 10), (10, 1000, 12)]
Z = [(18, 20, 288), (10, 16, 300), (12, 18, 324), (8, 20, 480), (20, 10, 540), (8, 10, 600), (16, 12, 750),
     (10, 8, 810), (8, 12, 900), (10, 16, 960), (12, 18, 972), (8, 10, 1000)]
LARGE = [(8, 1024, 540), (10, 900, 480), (900, 18, 270), (480, 30, 300), (1024, 512, 10), (900, 486, 12), (960, 300, 16),
         (600, 150, 54), (450, 250, 40)]
P = dict(dt=0.1, M=0.9, kappa=1.1, h=1.0)


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def run(shape, model, advance):
    """(initial field, field after advance(grid), energy, mean)"""
    import torch
    from paper_2507_21748_gb300 import evx
    c0 = inputs.uniform_field(shape, seed=31, offset=0.2, lo=-0.4, hi=0.4)
    with evx.Grid(shape, model=model, **P) as g:
        g.set_field(torch.from_numpy(c0).cuda())
        if model != "vm":
            assert np.abs(g.get_field().cpu().numpy() - c0).max() <= 2e-6
        advance(g)
        return c0, g.get_field().cpu().numpy(), g.energy()[0], g.mean()


def close(c0, got, ref):
    assert rel(got, ref) <= 1e-5
    assert rel(got - c0.astype(np.float64), ref - c0) <= 1e-4


@pytest.mark.parametrize("model", ["ch", "ac", "vm"])
@pytest.mark.parametrize("shape", XY + Z + LARGE)
def test_step(shape, model):
    c0, got, E, mean = run(shape, model, lambda g: g.step(1))
    ref = {"ch": O.ch_step, "ac": O.ac_step, "vm": O.vm_step}[model](c0, P["dt"], P["M"], P["kappa"], P["h"], 1)
    close(c0, got, ref)
    Eref = (O.vm_energy if model == "vm" else O.energy)(ref, P["kappa"])
    assert abs(E - Eref) <= 1e-5 * abs(Eref)
    if model == "ac":
        assert abs(mean - ref.mean()) <= 1e-9


@pytest.mark.parametrize("shape", XY + Z)
def test_block(shape):
    c0, got, _, _ = run(shape, "ch", lambda g: g.block(10))
    close(c0, got, O.ch_block_step(c0, P["dt"], P["M"], P["kappa"], P["h"], 10))


@pytest.mark.parametrize("shape", [(162, 180, 20), (10, 16, 300), (12, 18, 324), (20, 10, 540), (900, 8, 288), (972, 10, 12)])
def test_adjoint(shape):
    import torch
    from paper_2507_21748_gb300 import evx
    c0 = inputs.uniform_field(shape, seed=33, lo=-0.3, hi=0.3, offset=0.1)
    cN, target = (O.ch_step(c0, P["dt"], m, k, P["h"], 5) for m, k in ((P["M"], P["kappa"]), (0.8, 1.5)))
    dL = (cN - target).astype(np.float32)
    ref = O.ch_adjoint(c0, dL.astype(np.float64), P["dt"], P["M"], P["kappa"], P["h"], 5)
    with evx.Grid(shape, **P) as g:
        d0, gk, gm = g.adjoint(torch.from_numpy(c0).cuda(), 5, 3, torch.from_numpy(dL).cuda())
    assert rel(d0.cpu().numpy(), ref[0]) <= 1e-4
    for got, want in ((gk, ref[1]), (gm, ref[2])):
        assert abs(got - want) <= 1e-4 * abs(want)
