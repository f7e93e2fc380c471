"""32 -> 32 convolutions whose rows end in a 64-voxel chunk (Z an odd multiple of 64) and
whose columns are split into uneven y segments, against the FP64 oracle. Bounds: BF16
operands and outputs, so half a BF16 ulp per value (2^-9) plus FP32 accumulation."""
import numpy as np
import pytest

from oracle import nn as N

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 2, 64), (1, 3, 50, 64), (2, 2, 24, 192), (1, 2, 10, 320), (3, 40, 34, 64)])
@pytest.mark.parametrize("epi", [0, 1, 5])
def test_half_chunks_match_the_oracle(shape, epi):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    rng = np.random.default_rng(sum(shape) + epi)

    def bf16(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16)

    B, X, Y, Z = shape
    x, w = bf16(rng.standard_normal(shape + (32,))), bf16(rng.standard_normal((27, 32, 32)) * 0.1)
    b = torch.from_numpy(rng.standard_normal(32).astype(np.float32))
    stream = torch.from_numpy(rng.standard_normal(shape + (32,)).astype(np.float32))
    out = torch.zeros(shape + (32,), dtype=torch.bfloat16, device="cuda")
    pre = stream.cuda() if epi == 5 else torch.zeros_like(out)
    xd, wd, bd = x.cuda(), w.cuda(), b.cuda()
    S._ck(S.lib.evx_nn_conv3d(S._p(xd), S._p(wd), S._p(bd), S._p(out), S._p(pre), None, B, X, Y, Z, 32, 32, epi,
                              S._stream()))
    S.check()
    ref = N.conv(x.double().numpy(), w.double().numpy(), b.double().numpy())
    if epi == 1:
        assert np.linalg.norm(pre.double().cpu().numpy() - ref) < 2.0 ** -8 * np.linalg.norm(ref)
        ref = N.gelu(ref)
    if epi == 5:
        ref = ref + stream.double().numpy()
        assert np.linalg.norm(pre.double().cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)
    assert np.linalg.norm(out.double().cpu().numpy() - ref) < 2.0 ** -8 * np.linalg.norm(ref)
