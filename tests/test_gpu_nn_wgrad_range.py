"""Weight gradients whose partial sums are infinite, or finite with a total beyond FP32:
both give infinity of the right sign, not NaN (the total is an FP64 sum, rounded to FP32 at the end)."""
import pytest

pytestmark = pytest.mark.gpu

SHAPE = (1, 32, 64, 64)  # 2^17 voxels


# 2^100 * 2^100 overflows by itself; 2^58 * 2^58 over 2^17 voxels only in the total (2^133; a
# CTA's share is 2^124 to 2^127)
@pytest.mark.parametrize("log2", [100, 58])
@pytest.mark.parametrize("cin,cout,engine", [(32, 32, 0), (32, 32, 1), (16, 32, 0), (32, 16, 0)])
def test_overflow_is_infinite(cin, cout, engine, log2):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    x = torch.full(SHAPE + (cin,), 2.0 ** log2, device="cuda").bfloat16()
    dy = torch.full(SHAPE + (cout,), -2.0 ** log2, device="cuda").bfloat16()
    part = torch.empty(304 * 27 * cin * cout, dtype=torch.float32, device="cuda")
    dw = torch.empty((27, cout, cin), dtype=torch.float32, device="cuda")
    old = S.conv_engine()
    try:
        S.set_conv_engine(engine)
        S._ck(S.lib.evx_nn_conv3d_wgrad(S._p(dy), S._p(x), S._p(dw), S._p(part), part.numel(), *SHAPE, cin, cout,
                                        S._stream()))
        S.check()
    finally:
        S.set_conv_engine(old)
    assert bool((dw == -float("inf")).all())
