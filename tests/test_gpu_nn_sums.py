"""The surrogate's FP64 reductions on FP32 pairs against numpy in FP64: ragged lengths,
buffers off the 16-byte grid, values whose squares leave FP32's range, infinities and NaN.
A pair holds a value to 2^-46, so sums agree to 1e-13 of the sum of magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_21748_gb300 import surrogate
    return surrogate


def field(n, kind, seed):
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1, 1, n)
    scale = {"unit": 1.0, "tiny": 1e-25, "large": 1e25, "mixed": 10.0 ** rng.integers(-12, 3, n).astype(float)}[kind]
    return (x * scale).astype(np.float32)


@pytest.mark.parametrize("n,off,kind", [(1, 0, "unit"), (33, 1, "unit"), (100003, 0, "mixed"), (65536, 3, "tiny"),
                                        (300001, 0, "large"), (1 << 20, 0, "unit")])
def test_sums(S, n, off, kind):
    import torch
    x, t = field(n, kind, n), field(n, kind, n + 1)
    buf = [torch.zeros(n + 4, device="cuda") for _ in range(3)]
    for b, a in zip(buf, (x, t)):
        b[off:off + n] = torch.from_numpy(a).cuda()
    xd, td, gd = (b[off:off + n] for b in buf)
    part, out = torch.empty(304, dtype=torch.float64, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
    S._ck(S.lib.evx_nn_abs_sum(S._p(xd), n, S._p(part), 304, S._p(out), S._stream()))
    ref = np.abs(x.astype(np.float64)).sum()
    assert abs(out.item() - ref) <= 1e-13 * ref
    S._ck(S.lib.evx_nn_mse(S._p(xd), S._p(td), n, 0.5, S._p(gd), S._p(part), 304, S._p(out), S._stream()))
    d = x - t  # FP32, as the kernel
    ref = np.square(d.astype(np.float64)).sum()
    assert abs(out.item() - ref) <= 1e-13 * ref
    assert np.array_equal(gd.cpu().numpy(), np.float32(0.5) * d)


@pytest.mark.parametrize("V,amp,mean", [(4096, 0.05, 0.0), (5003, 1e-11, 0.0), (4097, 0.5, -0.3), (4096, 40.0, 3.0)])
def test_nl_scale_and_zero_mean(S, V, amp, mean):
    import torch
    B = 3
    c = (mean + amp * np.random.default_rng(V).uniform(-1, 1, (B, V))).astype(np.float32)
    cd = torch.from_numpy(c).cuda()
    part = torch.empty(3 * 304 * B, dtype=torch.float64, device="cuda")
    sc = torch.empty(B, dtype=torch.float64, device="cuda")
    S._ck(S.lib.evx_nn_nl_scale(S._p(cd), B, V, S._p(part), 304, S._p(sc), S._stream()))
    c64 = c.astype(np.float64)
    m = c64.mean(1, keepdims=True)
    d = c64 - m
    N = d * d * (3 * m + d)
    ref = np.minimum(1.0, np.sqrt((N * N).sum(1) / (d * d).sum(1)))
    assert np.all(np.abs(sc.cpu().numpy() - ref) <= 1e-11 * ref)
    out = torch.empty_like(cd)
    S._ck(S.lib.evx_nn_zero_mean_add_scaled(S._p(cd), S._p(cd), S._p(sc), B, V, S._p(part), 304, S._p(out), S._stream()))
    want = c64 + ref[:, None] * d
    assert np.max(np.abs(out.cpu().numpy() - want)) <= 4 * 2.0 ** -24 * np.max(np.abs(c64) + np.abs(d))


def test_non_finite_values_pass_through(S):
    import torch
    x = torch.ones(1000, device="cuda")
    part, out = torch.empty(304, dtype=torch.float64, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
    x[17] = float("inf")
    S._ck(S.lib.evx_nn_abs_sum(S._p(x), 1000, S._p(part), 304, S._p(out), S._stream()))
    assert out.item() == float("inf")
    x[18] = float("nan")
    S._ck(S.lib.evx_nn_abs_sum(S._p(x), 1000, S._p(part), 304, S._p(out), S._stream()))
    assert np.isnan(out.item())


@pytest.mark.parametrize("nvox,c", [(5, 16), (1001, 32), (64, 8), (7, 3)])
def test_field_to_act(S, nvox, c):
    import torch
    f = torch.from_numpy(field(nvox, "unit", nvox)).cuda()
    act = torch.full((nvox, c), 7.0, dtype=torch.bfloat16, device="cuda")
    S._ck(S.lib.evx_nn_field_to_act(S._p(f), nvox, c, 0.5, S._p(act), S._stream()))
    want = torch.zeros_like(act)
    want[:, 0] = (f * 0.5).bfloat16()
    assert torch.equal(act, want)
