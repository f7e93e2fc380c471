"""CPU model of the two-radix passes (csrc/evx_mixed*.cu, csrc/evx_mixed.cuh): the radix
split of every length, the exchange slots and the transforms they make up against
numpy's FFT, the real-row passes, and the index maps of the composite register DFTs.
Every shared-memory slot is checked against the buffer the launch allocates."""
import numpy as np
import pytest

RADICES = [1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32]
SMOOTH = sorted(2 ** a * 3 ** b * 5 ** c for a in range(11) for b in range(7) for c in range(5)
                if 4 <= 2 ** a * 3 ** b * 5 ** c <= 1024)


def split(L):
    for r1 in RADICES:
        if L % r1 == 0 and L // r1 <= r1 and L // r1 in RADICES:
            return r1, L // r1
    return None


def dft(v, d):
    n = np.arange(len(v))
    return np.exp(d * 2j * np.pi * np.outer(n, n) / len(v)) @ v


def tw(L, m, d):
    return np.exp(d * 2j * np.pi * m / L)


def test_every_edge_has_a_split_but_two():
    edges = [n for n in SMOOTH if n % 2 == 0 and n >= 8]
    assert [n for n in edges if split(n) is None] == [972, 1000]
    assert [n // 2 for n in edges if split(n // 2) is None] == []


@pytest.mark.parametrize("L", [n for n in SMOOTH if split(n)])
def test_column_passes(L):
    R1, R2 = split(L)
    R2p, slots = R2 | 1, R1 * (R2 | 1)
    rng = np.random.default_rng(L)
    x = rng.standard_normal(L) + 1j * rng.standard_normal(L)
    for d in (-1, 1):
        buf = np.full(slots, np.nan, complex)
        for n2 in range(R2):  # ColLoad
            v = dft(x[n2 + R2 * np.arange(R1)], d)
            for k in range(R1):
                assert n2 * k < L
                buf[k * R2p + n2] = v[k] * tw(L, n2 * k, d)
        out = np.empty(L, complex)
        for k1 in range(R1):  # ColStore
            out[k1 + R1 * np.arange(R2)] = dft(buf[k1 * R2p + np.arange(R2)], d)
        ref = np.fft.fft(x) if d < 0 else np.fft.ifft(x) * L
        assert np.allclose(out, ref, atol=1e-10 * L)
    # ColUpdate's inverse half and ColStoreInv: X (item k1, k2) back to x
    X, buf = np.fft.fft(x), np.full(slots, np.nan, complex)
    for k1 in range(R1):
        v = dft(X[k1 + R1 * np.arange(R2)], 1)
        buf[k1 * R2p + np.arange(R2)] = v * tw(L, np.arange(R2) * k1, 1)
    out = np.empty(L, complex)
    for n2 in range(R2):
        out[n2 + R2 * np.arange(R1)] = dft(buf[np.arange(R1) * R2p + n2], 1)
    assert np.allclose(out / L, x, atol=1e-12 * L)


def zstride(M, Zp, R1, R2):
    rs = max(Zp, R1 * (R2 | 1))
    return rs + ((((R1 + 1) & ~1) - rs) % 16)


@pytest.mark.parametrize("M", [n for n in SMOOTH if n <= 512 and split(n)])
def test_row_passes(M):
    R1, R2 = split(M)
    R2p, Zp = R2 | 1, (M + 1 + 7) // 8 * 8
    RS = zstride(M, Zp, R1, R2)
    assert RS % 2 == 0 and RS >= M + 1 and RS >= R1 * R2p and RS % 16 == ((R1 + 1) & ~1) % 16
    rng = np.random.default_rng(M)
    c = rng.standard_normal(2 * M)
    X = np.fft.rfft(c)
    row = np.full(RS, np.nan, complex)
    row[:M + 1] = X
    k = np.arange(M)
    w = tw(2 * M, k, -1)
    # ZInvA: pre-processing of k = n2 + R2 i, then the exchange
    P, Q = row[k] + np.conj(row[M - k]), row[k] - np.conj(row[M - k])
    Z = P + 1j * np.conj(w) * Q
    ex = np.full(RS, np.nan, complex)
    for n2 in range(R2):
        v = dft(Z[n2 + R2 * np.arange(R1)], 1)
        ex[np.arange(R1) * R2p + n2] = v * tw(M, n2 * np.arange(R1), 1)
    z = np.empty(M, complex)
    for k1 in range(R1):  # ZMiddle / ZInvB: real samples m = k1 + R1 k
        z[k1 + R1 * np.arange(R2)] = dft(ex[k1 * R2p + np.arange(R2)], 1)
    got = np.stack([z.real, z.imag], 1).reshape(-1) / (2 * M)
    assert np.allclose(got, c, atol=1e-11 * M)
    # ZMiddle / ZFwdB forward half, ZFwdA, post-processing
    s = c[0::2] + 1j * c[1::2]
    for k1 in range(R1):
        v = dft(s[k1 + R1 * np.arange(R2)], -1)
        ex[k1 * R2p + np.arange(R2)] = v * tw(M, np.arange(R2) * k1, -1)
    nat = np.empty(M, complex)
    for n2 in range(R2):
        nat[n2 + R2 * np.arange(R1)] = dft(ex[np.arange(R1) * R2p + n2], -1)
    assert np.allclose(nat, np.fft.fft(s), atol=1e-10 * M)
    out = np.full(M + 1, np.nan, complex)
    for kk in range(M // 2 + 1):
        if kk == 0:
            out[0], out[M] = nat[0].real + nat[0].imag, nat[0].real - nat[0].imag
            continue
        P, Q = nat[kk] + np.conj(nat[M - kk]), nat[kk] - np.conj(nat[M - kk])
        u = -1j * tw(2 * M, kk, -1) * Q
        out[kk] = (P + u) / 2
        if M - kk != kk:
            out[M - kk] = np.conj(P - u) / 2
    assert np.allclose(out, X, atol=1e-10 * M)


@pytest.mark.parametrize("N1,N2", [(2, 3), (4, 3), (3, 5), (2, 9), (8, 3), (2, 15)])
def test_coprime_register_dfts(N1, N2):
    N = N1 * N2
    x = np.random.default_rng(N).standard_normal(N) + 0j
    for d in (-1, 1):
        t = np.array([dft(np.array([x[(N2 * n1 + N1 * n2) % N] for n2 in range(N2)]), d) for n1 in range(N1)])
        t = np.array([dft(t[:, k2], d) for k2 in range(N2)]).T
        out = np.empty(N, complex)
        for k in range(N):
            out[k] = t[k % N1, k % N2]
        assert np.allclose(out, dft(x, d))


def root(m, n):
    """root_of_unity of csrc/evx_fft.cuh."""
    m %= n
    o = 8 * m // n
    num = 8.0 * m - o * n
    if o & 1:
        num = n - num
    x = num / n * 0.78539816339744830962
    c = s = 0.0
    tc, ts = 1.0, x
    for k in range(12):
        c, s = c + tc, s + ts
        tc *= -x * x / ((2 * k + 1) * (2 * k + 2))
        ts *= -x * x / ((2 * k + 2) * (2 * k + 3))
    return [(c, s), (s, c), (-s, c), (-c, s), (-c, -s), (-s, -c), (s, -c), (c, -s)][o]


def test_compile_time_roots():
    for n in range(2, 33):
        for m in range(-n, 2 * n):
            c, s = root(m, n)
            a = 8 * np.arctan(np.longdouble(1)) * (m % n) / n  # extended precision: the reference's argument is exact
            assert abs(c - np.cos(a)) < 4e-16 and abs(s - np.sin(a)) < 4e-16
