"""The FP32-stream lift and projection at the edges of their tiles (16 / ZW rows x 32 ZW columns;
16 rows x 32 columns walked along x) against the FP64 oracle: rows that end inside a tile,
X = 1 wraps, several segments per column, a scale. 27 to 864 FP32 terms per value: 1e-5
relative, as for the BF16 forms; the lift's BF16 copy within half an ulp (2^-8)."""
import numpy as np
import pytest

from oracle import nn as N

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 2, 32), (1, 3, 18, 96), (2, 9, 34, 64), (1, 20, 6, 128), (3, 33, 16, 32)])
@pytest.mark.parametrize("scale", [1.0, 0.75])
def test_lift32_and_project32(shape, scale):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    rng = np.random.default_rng(sum(shape))

    def bf16(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16)

    B, X, Y, Z = shape
    f = rng.standard_normal(shape).astype(np.float32)
    w0, wp = bf16(rng.standard_normal((27, 32, 16)) * 0.2), bf16(rng.standard_normal((27, 16, 32)) * 0.1)
    b0 = torch.from_numpy(rng.standard_normal(32).astype(np.float32))
    fd, w0d, wpd, b0d = torch.from_numpy(f).cuda(), w0.cuda(), wp.cuda(), b0.cuda()
    h = torch.empty(shape + (32,), dtype=torch.bfloat16, device="cuda")
    h32, d = torch.empty(shape + (32,), device="cuda"), torch.empty(shape, device="cuda")
    S._ck(S.lib.evx_nn_lift32(S._p(fd), scale, S._p(w0d), 16, 32, S._p(b0d), S._p(h), S._p(h32), *shape, S._stream()))
    act = np.zeros(shape + (16,))
    act[..., 0] = f * np.float32(scale)
    ref = N.conv(act, w0.double().numpy(), b0.double().numpy())
    assert np.linalg.norm(h32.double().cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)
    assert np.linalg.norm(h.double().cpu().numpy() - ref) < 2.0 ** -8 * np.linalg.norm(ref)
    S._ck(S.lib.evx_nn_project32(S._p(h32), S._p(wpd), 32, 16, S._p(b0d), S._p(d), *shape, S._stream()))
    S.check()
    ref = N.conv(h32.double().cpu().numpy(), wp.double().numpy(), b0[:16].double().numpy())[..., 0]
    assert np.linalg.norm(d.double().cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)
