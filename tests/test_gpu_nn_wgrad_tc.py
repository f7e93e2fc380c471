"""Weight gradient of the 32 -> 32 convolutions on the tensor-memory kernel against FP64
sums, at the edges of its units: one row, wrapped neighbours, dY ring wraps (more than 11
rows), half chunks, several segments per column, fewer partial sums than CTAs. FP32
accumulation over n voxels of random products: bound 2^-23 sqrt(n) relative, at least 1e-6."""
import numpy as np
import pytest

from oracle import nn as N

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,ctas", [((1, 1, 2, 64), 304), ((1, 2, 2, 128), 304), ((1, 2, 30, 64), 1),
                                        ((2, 3, 26, 192), 304), ((1, 1, 100, 128), 3), ((1, 20, 16, 320), 304)])
def test_wgrad_matches_fp64(shape, ctas):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    rng = np.random.default_rng(sum(shape))

    def bf16(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16)

    x, dy = bf16(rng.standard_normal(shape + (32,))), bf16(rng.standard_normal(shape + (32,)))
    xd, dyd = x.cuda(), dy.cuda()
    part = torch.empty(ctas * 27 * 1024, dtype=torch.float32, device="cuda")
    dw = torch.empty((27, 32, 32), dtype=torch.float32, device="cuda")
    S._ck(S.lib.evx_nn_conv3d_wgrad(S._p(dyd), S._p(xd), S._p(dw), S._p(part), part.numel(), *shape, 32, 32, S._stream()))
    S.check()
    ref = N.conv_wgrad(dy.double().numpy(), x.double().numpy())
    bound = max(1e-6, 2.0 ** -23 * np.sqrt(np.prod(shape)))
    assert np.linalg.norm(dw.double().cpu().numpy() - ref) <= bound * np.linalg.norm(ref)
