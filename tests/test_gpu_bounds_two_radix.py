"""The bounds-checked build (see test_gpu_bounds.py) on grids whose passes run the two-radix
and the grouped-stage kernels: every class of radices along x, y and z, row counts that leave
the last CTA short, and the grouped stages next to both. No access outside a buffer, and the
fields and energies of the normal build."""
import os
import subprocess
import sys

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_21748_gb300", "csrc")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import sys
sys.path.insert(0, %r)
import numpy as np, torch
from paper_2507_21748_gb300 import evx, inputs
res = {}
for shape in [(300, 18, 10), (324, 8, 36), (960, 8, 10), (162, 180, 300), (8, 768, 540), (16, 150, 320), (10, 972, 12),
              (18, 20, 1000), (20, 50, 54)]:
    c0 = torch.from_numpy(inputs.uniform_field(shape, seed=1, offset=0.1, lo=-0.4, hi=0.4)).cuda()
    for model in ("ch", "ac", "vm"):
        with evx.Grid(shape, model=model) as g:
            g.set_field(c0)
            g.step(3)
            out = [torch.tensor(g.energy()[0])]
            if model == "ch":
                g.block(4)
            out.append(g.get_field().cpu())
            if model == "ch" and c0.numel() < 2 ** 21:
                d0, gk, gm = g.adjoint(c0, 3, 2, torch.ones_like(c0))
                out += [d0.cpu(), torch.tensor([gk, gm])]
        res[(shape, model)] = out
torch.save(res, sys.argv[1])
print("BOUNDS", *evx.debug_bounds())
''' % ROOT


def test_every_checked_file_is_reported():
    with open(os.path.join(CSRC, "evx_runtime.cu")) as f:
        runtime = f.read()
    for name, text in ((n, open(os.path.join(CSRC, n)).read()) for n in sorted(os.listdir(CSRC)) if n.endswith(".cu")):
        if "EVX_IN(" in text or "EVX_AT(" in text or "evx_mixed.cuh" in text:
            take = "bounds_line_" + name[len("evx_"):-len(".cu")]
            assert "int %s(bool clear)" % take in text and take in runtime, name


@pytest.mark.gpu
def test_two_radix_kernels_stay_in_bounds(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300.build import build_lib
    libs = [build_lib(debug_bounds=True), build_lib()]
    got = []
    for i, lib in enumerate(libs):
        out = str(tmp_path / ("%d.pt" % i))
        env = dict(os.environ, EVX_LIB=lib)
        env.pop("EVX_GENERIC", None)
        r = subprocess.run([sys.executable, "-c", SCRIPT, out], env=env, capture_output=True, text=True, timeout=900)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
        assert r.stdout.splitlines()[-1] == "BOUNDS %d 0" % (1 - i), r.stdout[-500:]
        got.append(torch.load(out))
    for key, a in got[0].items():
        for x, y in zip(a, got[1][key]):
            assert torch.isfinite(x).all() and float((x - y).norm()) <= 1e-6 * float(y.norm()), key
