"""Calls that must not take longer than a kernel of the same arithmetic, best of ten. The
FP32-stream projection against the BF16 one (both 864 FMAs per voxel; the walking kernel
alone took 3.9 times as long here), half as much again allowed. The BF16 lift against the
FP32-stream one, which stores three times the bytes (1.19 times as long when every lane
rounded every input). A 32 -> 32 convolution of one short column per CTA against mma.sync
(1.22 times as long with columns of eight rows). A tenth allowed in these two."""
import numpy as np
import pytest

from oracle import nn as N

pytestmark = pytest.mark.gpu


def best_us(call):
    import torch
    times = []
    for _ in range(10):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(20):
            call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 50.0)
    return min(times)


@pytest.mark.parametrize("shape", [(1, 24, 24, 64), (1, 32, 32, 64), (1, 24, 24, 128), (1, 64, 64, 64)])
def test_project32(shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    rng = np.random.default_rng(3)
    h32 = torch.from_numpy(rng.standard_normal(shape + (32,)).astype(np.float32)).cuda()
    h, w = h32.to(torch.bfloat16), torch.from_numpy(rng.standard_normal((27, 16, 32)).astype(np.float32)).to(torch.bfloat16).cuda()
    out = torch.empty(shape, device="cuda")
    t16 = best_us(lambda: S._ck(S.lib.evx_nn_project(S._p(h), S._p(w), 32, 16, None, S._p(out), *shape, S._stream())))
    t32 = best_us(lambda: S._ck(S.lib.evx_nn_project32(S._p(h32), S._p(w), 32, 16, None, S._p(out), *shape, S._stream())))
    S.check()
    ref = N.conv(h32.double().cpu().numpy(), w.double().cpu().numpy())[..., 0]
    assert np.linalg.norm(out.double().cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)
    assert t32 <= 1.5 * t16, (t32, t16)


def test_lift():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    shape = (4, 64, 64, 64)
    f, w = torch.randn(shape, device="cuda"), torch.randn((27, 32, 16), device="cuda").to(torch.bfloat16)
    h, h32 = torch.empty(shape + (32,), dtype=torch.bfloat16, device="cuda"), torch.empty(shape + (32,), device="cuda")
    t16 = best_us(lambda: S._ck(S.lib.evx_nn_lift(S._p(f), 1.0, S._p(w), 16, 32, None, S._p(h), *shape, S._stream())))
    t32 = best_us(lambda: S._ck(S.lib.evx_nn_lift32(S._p(f), 1.0, S._p(w), 16, 32, None, S._p(h), S._p(h32), *shape,
                                                    S._stream())))
    assert t16 <= 1.1 * t32, (t16, t32)


@pytest.mark.parametrize("epi", ["PLAIN", "GELU"])
def test_conv_short_columns(epi):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    shape = (1, 8, 8, 64)
    x, pre, out = (torch.randn(shape + (32,), device="cuda").to(torch.bfloat16) for _ in range(3))
    w = torch.randn((27, 32, 32), device="cuda").to(torch.bfloat16)
    before, t = S.lib.evx_nn_conv_engine(), {}
    for engine in (S.ENGINE_TCGEN05, S.ENGINE_MMA_SYNC):
        S._ck(S.lib.evx_nn_set_conv_engine(engine))
        try:
            t[engine] = best_us(lambda: S._ck(S.lib.evx_nn_conv3d(
                S._p(x), S._p(w), None, S._p(out), S._p(pre), None, *shape, 32, 32, getattr(S, "EPI_" + epi), S._stream())))
        finally:
            S._ck(S.lib.evx_nn_set_conv_engine(before))
    S.check()
    assert t[S.ENGINE_TCGEN05] <= 1.1 * t[S.ENGINE_MMA_SYNC], t
