"""The FP32-stream projection on both sides of its rule: the walking kernel (full tiles, rows
that end inside a tile, uneven segments, several columns per CTA, a wrap onto itself) and the
lane-per-channel one, which a base off 16 bytes takes on any grid. The two add the same
products in the same order, so their results are equal to the bit; 864 FP32 terms per value
against FP64: 1e-5 relative."""
import pytest

pytestmark = pytest.mark.gpu

WALK = [(8, 20, 46, 96), (2, 65, 64, 128), (16, 24, 48, 32), (1, 70, 158, 96), (152, 12, 16, 64)]
LANE = [(1, 24, 24, 64), (2, 9, 34, 64), (1, 64, 64, 64)]


def planes_and_rounds(shape, sms):
    """The rule of evx_nn_project32, restated: the walk where planes < 3 rounds."""
    B, X, Y, Z = shape
    ncol, best = B * -(-Y // 16) * (Z // 32), None
    for s in [1] + list(range(2, X // 8 + 1)):
        planes = -(-ncol * s // sms) * (-(-X // s) + 2)
        best = planes if best is None or planes < best else best
    return best, -(-(B * X * (Y // 2) * (Z // 32)) // (16 * sms))


@pytest.mark.parametrize("shape", WALK + LANE)
def test_same_bits(shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate as S
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        planes, rounds = planes_and_rounds(shape, 152)
        assert (planes < 3 * rounds) == (shape in WALK), (planes, rounds)
    gen = torch.Generator(device="cuda").manual_seed(7)
    n = shape[0] * shape[1] * shape[2] * shape[3]
    buf = torch.empty(n * 32 + 4, device="cuda")
    h = torch.randn(shape + (32,), generator=gen, device="cuda")
    w = torch.randn((27, 16, 32), generator=gen, device="cuda").mul_(0.1).to(torch.bfloat16)
    b = torch.randn(16, generator=gen, device="cuda")
    out = []
    for shift in (0, 1):
        x = buf[shift:shift + n * 32].view(shape + (32,))
        x.copy_(h)
        assert (x.data_ptr() % 16 == 0) == (shift == 0)
        d = torch.empty(shape, device="cuda")
        S._ck(S.lib.evx_nn_project32(S._p(x), S._p(w), 32, 16, S._p(b), S._p(d), *shape, S._stream()))
        S.check()
        out.append(d)
    assert torch.equal(out[0], out[1])
    ref = torch.full(shape, float(b[0]), dtype=torch.float64, device="cuda")
    for t in range(27):
        off = (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)
        ref += torch.roll(h, [-o for o in off], (1, 2, 3)).double() @ w[t, 0].double()
    assert float((out[0] - ref).norm()) < 1e-5 * float(ref.norm())
