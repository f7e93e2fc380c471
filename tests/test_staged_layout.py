"""CPU model of the grouped-stage passes (csrc/evx_staged.cu): the leading and trailing
groups apply the operations of the stage-by-stage Stockham transform (csrc/evx_fft.cuh),
so the two models agree to the last bit; slots stay inside the exchange."""
import numpy as np
import pytest

GROUPS = [1, 2, 3, 4, 5, 6, 8, 9, 12, 15, 16, 20, 25, 27, 32]


def plan(L):
    r, n = [], L
    for p in (5, 3, 16):
        while n % p == 0:
            r.append(p)
            n //= p
    return r + ([n] if n > 1 else [])


def lead(R):
    return 5 if R % 5 == 0 else 3 if R % 3 == 0 else 16 if R % 16 == 0 else R


def cut(L):
    best, r1, pl = None, 1, plan(L)
    for r in pl:
        r1 *= r
        r2 = L // r1
        if r1 in GROUPS and r2 in GROUPS and (best is None or max(r1, r2) < max(best)):
            best = (r1, r2)
    return best


def dft(u, d):  # one fixed order of operations per radix
    n = len(u)
    out = np.zeros(n, complex)
    for k in range(n):
        acc = 0j
        for t in range(n):
            acc = acc + u[t] * np.exp(d * 2j * np.pi * (t * k % n) / n)
        out[k] = acc
    return out


def stockham(x, d):
    L, y, Ns = len(x), list(x), 1
    tw = [np.exp(d * 2j * np.pi * m / L) for m in range(L)]
    for r in plan(L):
        o = [None] * L
        for j in range(L // r):
            kk = j % Ns
            u = [y[j + t * (L // r)] for t in range(r)]
            if Ns > 1:
                u = [u[0]] + [u[t] * tw[t * kk * (L // (Ns * r))] for t in range(1, r)]
            u = dft(u, d)
            for t in range(r):
                o[(j - kk) * r + kk + t * Ns] = u[t]
        y, Ns = o, Ns * r
    return np.array(y)


def group(v, Ns, kk, L, d):
    R, nsi, rest, v = len(v), 1, len(v), list(v)
    while rest > 1:
        r = lead(rest)
        o = [None] * R
        for j in range(R // r):
            ki = j % nsi
            u = [v[j + t * (R // r)] for t in range(r)]
            if Ns * nsi > 1:
                step = L // (Ns * nsi * r) * (kk + ki * Ns)
                assert (r - 1) * step < L
                u = [u[0]] + [u[t] * np.exp(d * 2j * np.pi * (t * step) / L) for t in range(1, r)]
            u = dft(u, d)
            for t in range(r):
                o[(j - ki) * r + ki + t * nsi] = u[t]
        v, nsi, rest = o, nsi * r, rest // r
    return v


LENGTHS = [L for L in range(4, 129) if all(p in (2, 3, 5) for p in
           [q for q in range(2, L + 1) if L % q == 0 and all(q % s for s in range(2, q))])]


@pytest.mark.parametrize("L", LENGTHS)
def test_groups_are_the_stages(L):
    c = cut(L)
    if c is None:
        pytest.skip("no cut: the two-radix kernels take this length")
    R1, R2 = c
    R2p = R2 | 1
    x = np.random.default_rng(L).standard_normal(2 * L).view(complex)
    for d in (-1, 1):
        ex = [None] * (R1 * R2p)
        for n2 in range(R2):
            v = group([x[n2 + R2 * t] for t in range(R1)], 1, 0, L, d)
            for u in range(R1):
                ex[u * R2p + n2] = v[u]
        out = np.zeros(L, complex)
        for k1 in range(R1):
            v = group([ex[k1 * R2p + t] for t in range(R2)], R1, k1, L, d)
            for u in range(R2):
                out[k1 + R1 * u] = v[u]
        assert np.array_equal(out, stockham(x, d))
        assert np.allclose(out, np.fft.fft(x) if d < 0 else np.fft.ifft(x) * L, atol=1e-10 * L)
    # LeadFromRows: element n2 + R2 t of a spectrum left in rows (k at (k mod R1) R2p + k / R1)
    dq, dm = R2 // R1, R2 % R1
    for n2 in range(R2):
        q, m = divmod(n2, R1)
        for t in range(R1):
            k = n2 + R2 * t
            assert (m, q) == (k % R1, k // R1) and m * R2p + q < R1 * R2p
            q, m = q + dq, m + dm
            if m >= R1:
                m, q = m - R1, q + 1


def test_lengths_the_surrogate_trains_on_have_a_cut():
    assert all(cut(L) for L in (24, 30, 32, 36, 40, 48, 50, 54, 60, 72, 80, 90, 96, 100, 108, 120))
