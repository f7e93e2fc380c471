"""CPU model of vm_fd_kernel (csrc/evx_kernels.cu): thread map, shared-memory planes, the
register columns and the plane schedule, executed plane by plane with poisoned slots (NaN)
so that a read of a plane that is not there, of a wrong halo or of a slot already reused
shows in the result, which must equal the stencils evaluated directly."""
import numpy as np
import pytest

TY, TZ = 16, 64
Q, CZ, CY, MZ, MY = TZ // 4, TZ + 8, TY + 4, TZ + 8, TY + 2
MAIN = (TY + 2) * Q
KH2, M0 = 1.3, 0.8


def mob(v):
    return M0 * np.maximum(1 - v * v, 0)


def direct(c):
    def nb(f, d, s):
        return np.roll(f, -s, d)
    mu = c ** 3 - c - KH2 * (sum(nb(c, d, s) for d in range(3) for s in (1, -1)) - 6 * c)
    m = mob(c)
    return sum(0.5 * (m + nb(m, d, s)) * (nb(mu, d, s) - mu) for d in range(3) for s in (1, -1))


def cta(c, rhs, y0, z0, x0, xc):
    nx, ny, nz = c.shape
    xe, nzv = min(x0 + xc, nx), min(TZ, nz - z0)
    cs = np.full((4, CY * CZ), np.nan)
    ms, bs = np.full((2, MY * MZ), np.nan), np.full((2, MY * MZ), np.nan)

    def load(xp):
        cs[xp & 3] = np.nan
        for r in range(CY):
            y = (y0 + r - 2) % ny
            for q in range(Q):
                if 4 * q < nzv:
                    cs[xp & 3, r * CZ + 4 + 4 * q: r * CZ + 8 + 4 * q] = c[xp % nx, y, z0 + 4 * q: z0 + 4 * q + 4]
            zl, zr = (z0 - 2) % nz, (z0 + nzv) % nz
            assert zl % 2 == 0 and zr % 2 == 0
            cs[xp & 3, r * CZ + 2: r * CZ + 4] = c[xp % nx, y, zl: zl + 2]
            cs[xp & 3, r * CZ + 4 + nzv: r * CZ + 6 + nzv] = c[xp % nx, y, zr: zr + 2]

    threads = []
    for tid in range(MAIN + 32):
        main, e = tid < MAIN, tid - MAIN
        r, q = (tid // Q if main else 1 + (e >> 1)), tid % Q
        if not (4 * q < nzv if main else (e >> 1) < TY):
            continue
        n = 4 if main else 1
        col = 4 + 4 * q if main else (4 + nzv if e & 1 else 3)
        inner = main and 1 <= r <= TY and y0 + r - 1 < ny
        ce, me = (r + 1) * CZ + col, r * MZ + col
        assert CZ <= ce and ce + n - 1 + CZ < CY * CZ and me + n <= MY * MZ
        threads.append(dict(n=n, r=r, q=q, ce=ce, me=me, inner=inner))

    def own(t, xp):
        return cs[xp & 3, t["ce"]: t["ce"] + t["n"]].copy()

    def mu_plane(t, xp):
        s, n = cs[xp & 3], t["n"]
        a, d = s[t["ce"] + CZ: t["ce"] + CZ + n], s[t["ce"] - CZ: t["ce"] - CZ + n]
        zl, zr = s[t["ce"] - 1], s[t["ce"] + n]
        v = t["c0"]
        up = np.append(v[1:], zr) + np.append(zl, v[:-1])
        t["up"] = v ** 3 - v - KH2 * (t["cp"] + t["cm"] + a + d + up - 6 * v)
        t["bp"] = mob(v)
        ms[xp & 1, t["me"]: t["me"] + n], bs[xp & 1, t["me"]: t["me"] + n] = t["up"], t["bp"]

    for xp in range(x0 - 2, x0 + 2):
        load(xp)
    for t in threads:
        t["cm"], t["c0"], t["cp"] = own(t, x0 - 2), own(t, x0 - 1), own(t, x0)
        mu_plane(t, x0 - 1)
        t["um"], t["bm"], t["cm"], t["c0"] = t["up"], t["bp"], t["c0"], t["cp"]
        t["cp"] = own(t, x0 + 1)
        mu_plane(t, x0)
        t["u0"], t["b0"], t["cm"], t["c0"] = t["up"], t["bp"], t["c0"], t["cp"]
    load(x0 + 2)
    for x in range(x0, xe):
        if x + 3 <= xe + 1:
            load(x + 3)  # while other warps may still run iteration x - 1: it reads planes x and x + 1 only
            assert (x + 3) & 3 not in (x & 3, (x + 1) & 3)
        ms[(x + 1) & 1], bs[(x + 1) & 1] = np.nan, np.nan
        for t in threads:
            t["cp"] = own(t, x + 2)
            mu_plane(t, x + 1)
        for t in threads:
            if t["inner"]:
                o, u, b = t["me"], ms[x & 1], bs[x & 1]
                mi, ui = t["b0"], t["u0"]
                out = 0.5 * (mi + t["bp"]) * (t["up"] - ui) + 0.5 * (mi + t["bm"]) * (t["um"] - ui)
                for s in (MZ, -MZ):
                    out += 0.5 * (mi + b[o + s: o + s + 4]) * (u[o + s: o + s + 4] - ui)
                out += 0.5 * (mi + np.append(mi[1:], b[o + 4])) * (np.append(ui[1:], u[o + 4]) - ui)
                out += 0.5 * (mi + np.append(b[o - 1], mi[:-1])) * (np.append(u[o - 1], ui[:-1]) - ui)
                z = z0 + 4 * t["q"]
                rhs[x, y0 + t["r"] - 1, z: z + 4] = out
            t["um"], t["u0"], t["bm"], t["b0"] = t["u0"], t["up"], t["b0"], t["bp"]
            t["cm"], t["c0"] = t["c0"], t["cp"]


@pytest.mark.parametrize("shape,xc", [((8, 8, 8), 8), ((10, 18, 12), 64), ((20, 40, 68), 8), ((9, 16, 64), 64),
                                      ((17, 10, 132), 16)])
def test_march(shape, xc):
    nx, ny, nz = shape
    c = np.random.default_rng(nx).uniform(-1.2, 1.2, shape)
    rhs = np.full(shape, np.nan)
    for y0 in range(0, ny, TY):
        for z0 in range(0, nz, TZ):
            for x0 in range(0, nx, xc):
                cta(c, rhs, y0, z0, x0, xc)
    assert np.allclose(rhs, direct(c), rtol=0, atol=1e-12)
