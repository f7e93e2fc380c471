"""The 32 -> 32 weight gradient on the tensor-memory kernel is no further from FP64 than on
the mma.sync kernel, over batches with few and many input rows per CTA (the tensor core's
FP32 accumulation truncates, so the error grows with the rows that one accumulator adds)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 96, 80, 64), (1, 120, 128, 64), (1, 64, 96, 128), (4, 32, 64, 128), (2, 128, 64, 192)])
def test_error_against_fp64(shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    gen = torch.Generator(device="cuda").manual_seed(5)
    x, dy = (torch.randn(shape + (32,), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(2))
    part = torch.empty(304 * 27 * 1024, dtype=torch.float32, device="cuda")
    ref = torch.empty((27, 32, 32), dtype=torch.float64, device="cuda")
    flat = dy.double().reshape(-1, 32).T
    for t in range(27):
        off = (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)
        ref[t] = flat @ torch.roll(x.double(), [-o for o in off], (1, 2, 3)).reshape(-1, 32)
    err = {}
    before = S.lib.evx_nn_conv_engine()
    for engine in (S.ENGINE_TCGEN05, S.ENGINE_MMA_SYNC):
        S._ck(S.lib.evx_nn_set_conv_engine(engine))
        try:
            dw = torch.empty((27, 32, 32), dtype=torch.float32, device="cuda")
            S._ck(S.lib.evx_nn_conv3d_wgrad(S._p(dy), S._p(x), S._p(dw), S._p(part), part.numel(), *shape, 32, 32, S._stream()))
            S.check()
        finally:
            S._ck(S.lib.evx_nn_set_conv_engine(before))
        err[engine] = float((dw.double() - ref).norm() / ref.norm())
    assert 0.0 < err[S.ENGINE_TCGEN05] <= err[S.ENGINE_MMA_SYNC], err
