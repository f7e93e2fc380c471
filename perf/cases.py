"""The work that users of the framework have it do, as cases that can be timed and compared.

A case is one pass through the public entry points: a solver run (load the
initial field, step, read the result back, with the energy where a run monitors
it), a differentiable solve with its gradients, one convolution layer of the
learned surrogate forward and backward, one training step of the network, one
guarded surrogate block. ``listed()`` holds the cases that are followed,
``draw(rng)`` makes more of the same ranges, ``prepare`` makes what the caller
has in hand (seeded inputs, grid, network), ``run`` is the pass, ``exact`` the
same outputs in 64 bits from plain torch and ``work`` the bytes and operations a
pass cannot do without.
"""
import math

import torch

from paper_2507_21748_gb300 import evx, surrogate

DT, KAPPA, MOB = 0.1, 1.0, 1.0
SPREAD = 0.05  # the initial noise: offset + U(-0.05, 0.05) per voxel

# the edges a grid may have: even, 8 .. 1024, prime factors 2, 3 and 5 only
EDGES = sorted(2 ** a * 3 ** b * 5 ** c for a in range(1, 11) for b in range(7) for c in range(5)
               if 8 <= 2 ** a * 3 ** b * 5 ** c <= 1024)


def listed():
    return [
        # the smallest call: a coarse ragged grid stepped a few times, with its energy (interactive
        # use and parameter scans; every launch and synchronisation shows)
        dict(name="ch_48x40x36", kind="solve", model="ch", nx=48, ny=40, nz=36, steps=20, mean=0.0, energy=True,
             host=False),
        # the 64^3 reference configuration, 100 steps from noise
        dict(name="ch_64", kind="solve", model="ch", nx=64, ny=64, nz=64, steps=100, mean=0.0, energy=False,
             host=False),
        # 256^3, the energy monitored every 20 steps: one such stretch of a long run
        dict(name="ch_256", kind="solve", model="ch", nx=256, ny=256, nz=256, steps=20, mean=0.0, energy=True,
             host=False),
        # a segmented microstructure seldom has power-of-two edges: a ragged box, 20 steps
        dict(name="ch_300x240x200", kind="solve", model="ch", nx=300, ny=240, nz=200, steps=20, mean=0.1,
             energy=False, host=False),
        # 400^3 end to end: the field comes from and goes back to pinned host memory
        dict(name="ch_400_host", kind="solve", model="ch", nx=400, ny=400, nz=400, steps=20, mean=0.0, energy=False,
             host=True),
        # the throughput configuration: 1024^3, an off-critical mixture
        dict(name="ch_1024", kind="solve", model="ch", nx=1024, ny=1024, nz=1024, steps=10, mean=0.3, energy=False,
             host=False),
        # Allen-Cahn on the same engine (its mean moves: per-step FP64 sums), uneven edges
        dict(name="ac_128x256x512", kind="solve", model="ac", nx=128, ny=256, nz=512, steps=20, mean=0.2,
             energy=False, host=False),
        # variable mobility: finite-difference right-hand side, spectral preconditioner
        dict(name="vm_320x384x320", kind="solve", model="vm", nx=320, ny=384, nz=320, steps=10, mean=0.2,
             energy=False, host=False),
        # the inverse run: forward from noise, checkpoints every 20 steps, gradients for c0, kappa and M
        dict(name="inverse_128", kind="inverse", nx=128, ny=128, nz=128, steps=60, ckpt=20),
        # one 32 -> 32 layer of the surrogate, training: GELU convolution, then the data, weight and
        # bias gradients
        dict(name="layer_1x64x96x128", kind="layer", batch=1, nx=64, ny=96, nz=128),
        # one optimiser step of the surrogate on a batch of four boxes
        dict(name="train_4x64", kind="train", batch=4, nx=64, ny=64, nz=64),
        # one guarded block of the surrogate at its inference configuration
        dict(name="rollout_8x256", kind="rollout", batch=8, nx=256, ny=256, nz=256),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _edge(rng, lo, hi, multiple=2):
    """A supported edge near a log-uniform draw."""
    ok = [e for e in EDGES if lo <= e <= hi and e % multiple == 0]
    want = _log_uniform(rng, lo, hi)
    return min(ok, key=lambda e: abs(math.log(e / want)))


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["inverse", "layer", "train", "rollout"])
    if kind == "solve":
        model = rng.choice(["ch", "ch", "ch", "ac", "vm"])
        n = _log_uniform(rng, 40, 480)  # edges within a factor of two of each other, as boxes in use are
        nx, ny, nz = (_edge(rng, max(8, n / 1.5), min(1024, n * 1.5)) for _ in range(3))
        if rng.random() < 0.4:  # many users keep to powers of two
            nx, ny, nz = (2 ** max(3, round(math.log2(e))) for e in (nx, ny, nz))
        most = 4e9 / (nx * ny * nz)  # voxel-steps: well under the largest listed case
        steps = max(2, min(40, int(_log_uniform(rng, 5, 40)), int(most)))
        return dict(kind=kind, model=model, nx=nx, ny=ny, nz=nz, steps=steps, mean=rng.choice([0.1, 0.2, 0.3]),
                    energy=rng.random() < 0.4, host=rng.random() < 0.25)
    if kind == "inverse":
        nx, ny, nz = (_edge(rng, 32, 160) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, steps=rng.randrange(20, 61), ckpt=rng.choice([5, 10, 20]))
    nx, ny = _edge(rng, 24, 128), _edge(rng, 24, 128)
    nz = rng.choice([64, 128, 192, 256])
    most = 2 ** (24 if kind == "rollout" else 20) // (nx * ny * nz)  # a backward pass: up to the batch of four 64^3
    return dict(kind=kind, batch=rng.randrange(1, max(1, min(4, most)) + 1), nx=nx, ny=ny, nz=nz)


# ------------------------------------------------------------------ inputs
def _noise(shape, seed, mean=0.0, spread=SPREAD, dtype=torch.float32):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32)
    return f.mul_(2.0 * spread).add_(mean - spread).to(dtype)


def _normal(shape, seed, gain=1.0, dtype=torch.float32):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(gain).to(dtype)


def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _evolved(shape, batch, seed, steps):
    """Solver states of `batch` runs of mean compositions spread over [-0.3, 0.3]."""
    out = torch.empty((batch,) + shape, dtype=torch.float32, device="cuda")
    with evx.Grid(shape, dt=DT, M=MOB, kappa=KAPPA) as g:
        for i in range(batch):
            g.set_field(_noise(shape, seed * 64 + i, mean=-0.3 + 0.6 * (i + 0.5) / batch))
            g.step(steps)
            g.get_field(out[i])
    torch.cuda.synchronize()
    return out


def _layer_inputs(case, seed):
    shape = (case["batch"],) + _shape(case)
    bf = torch.bfloat16
    return dict(x=_normal(shape + (32,), 8 * seed, dtype=bf), dy=_normal(shape + (32,), 8 * seed + 1, 0.1, bf),
                w=_normal((27, 32, 32), 8 * seed + 2, math.sqrt(2.0 / (27 * 32)), bf),
                b=_normal((32,), 8 * seed + 3, 0.1), u=_normal(shape + (32,), 8 * seed + 4, dtype=bf))


def prepare(case, seed):
    kind, shape = case["kind"], _shape(case)
    if kind == "solve":
        c0 = _noise(shape, seed, case["mean"])
        grid = evx.Grid(shape, dt=DT, M=MOB, kappa=KAPPA, model=case["model"])
        if case["host"]:
            c0 = c0.cpu().pin_memory()
            out = torch.empty(shape, dtype=torch.float32).pin_memory()
        else:
            out = torch.empty_like(c0)
        return dict(case=case, c0=c0, out=out, grid=grid)
    if kind == "inverse":
        c0 = _noise(shape, seed)
        grid = evx.Grid(shape, dt=DT, M=0.8, kappa=1.5)
        grid.set_field(c0)
        grid.step(case["steps"])
        target = grid.get_field()
        c0.requires_grad_(True)
        kappa = torch.tensor(KAPPA, dtype=torch.float64, requires_grad=True)
        mob = torch.tensor(MOB, dtype=torch.float64, requires_grad=True)
        return dict(case=case, c0=c0, kappa=kappa, mob=mob, target=target, grid=grid)
    if kind == "layer":
        s = _layer_inputs(case, seed)
        S = surrogate
        act = s["x"].shape
        nparts = 2 * torch.cuda.get_device_properties(0).multi_processor_count
        s["wflip"] = torch.empty_like(s["w"])
        S.lib.evx_nn_flip_weights(S._p(s["w"]), 32, 32, S._p(s["wflip"]), S._stream())
        for name in ("pre", "act", "du"):
            s[name] = torch.empty(act, dtype=torch.bfloat16, device="cuda")
        s["dw"] = torch.empty((27, 32, 32), dtype=torch.float32, device="cuda")
        s["db"] = torch.empty(32, dtype=torch.float32, device="cuda")
        s["wpart"] = torch.empty(nparts * 27 * 32 * 32, dtype=torch.float32, device="cuda")
        s["dpart"] = torch.empty(nparts * 32, dtype=torch.float64, device="cuda")
        s["nparts"], s["case"] = nparts, case
        return s
    c = _evolved(shape, case["batch"], seed, 100)
    if kind == "rollout":
        net = surrogate.Net(shape, batch=case["batch"], seed=seed, train=False, proj_gain=1e-3)
        return dict(case=case, c=c, net=net)
    base, target = torch.empty_like(c), torch.empty_like(c)
    with evx.Grid(shape, dt=DT, M=MOB, kappa=KAPPA) as g:
        for i in range(case["batch"]):
            surrogate.block_base(g, c[i], base[i])
            g.set_field(c[i])
            g.step(10)
            g.get_field(target[i])
    torch.cuda.synchronize()
    net = surrogate.Net(shape, batch=case["batch"], seed=seed, train=True, proj_gain=1e-3)
    return dict(case=case, c=c, base=base, target=target, net=net)


# ------------------------------------------------------------------- passes
def _run_solve(s):
    case, g = s["case"], s["grid"]
    if case["host"]:
        g.set_field_host(s["c0"])
        g.step(case["steps"])
        out = [g.get_field_host(s["out"])]
    else:
        g.set_field(s["c0"])
        g.step(case["steps"])
        out = [g.get_field(s["out"])]
    if case["energy"]:
        out += list(g.energy())
    return out


def _run_inverse(s):
    for t in (s["c0"], s["kappa"], s["mob"]):
        t.grad = None
    c = evx.ch_solve(s["c0"], s["kappa"], s["mob"], s["grid"], s["case"]["steps"], s["case"]["ckpt"])
    loss = 0.5 * (c - s["target"]).square().sum()
    loss.backward()
    return dict(c=c.detach(), dc0=s["c0"].grad, dkappa=s["kappa"].grad.float(), dM=s["mob"].grad.float())


def _run_layer(s):
    S, case = surrogate, s["case"]
    B, (X, Y, Z), p, st = case["batch"], _shape(case), S._p, S._stream()
    ck = S._ck
    ck(S.lib.evx_nn_conv3d(p(s["x"]), p(s["w"]), p(s["b"]), p(s["act"]), p(s["pre"]), None, B, X, Y, Z, 32, 32,
                           S.EPI_GELU, st))
    ck(S.lib.evx_nn_conv3d(p(s["dy"]), p(s["wflip"]), None, p(s["du"]), p(s["u"]), None, B, X, Y, Z, 32, 32,
                           S.EPI_GELU_BWD, st))
    ck(S.lib.evx_nn_conv3d_wgrad(p(s["dy"]), p(s["x"]), p(s["dw"]), p(s["wpart"]), s["wpart"].numel(), B, X, Y, Z,
                                 32, 32, st))
    ck(S.lib.evx_nn_bias_grad(p(s["dy"]), B * X * Y * Z, 32, p(s["dpart"]), s["nparts"], p(s["db"]), st))
    return {k: s[k] for k in ("pre", "act", "du", "dw", "db")}


def _run_train(s):
    net = s["net"]
    pred = net.forward(s["c"], s["base"])
    loss = net.backward(s["target"])
    net.adam(5e-4)
    # the correction has zero mean, so the projection's bias has no gradient: what the sum
    # leaves in "bp" is rounding alone, and Adam scales even that to a full step
    names = [n for n in net.names if n != "bp"]
    return dict(pred=pred, loss=loss, grads={n: net.g[n] for n in names}, params={n: net.p[n] for n in names})


def _run_rollout(s):
    c, stats = surrogate.rollout(s["net"], s["c"], 1, base=True)
    return dict(c=c, fallbacks=stats["fallbacks"])


def run(state):
    kind = state["case"]["kind"]
    return dict(solve=_run_solve, inverse=_run_inverse, layer=_run_layer, train=_run_train,
                rollout=_run_rollout)[kind](state)


# ------------------------------------------------------------------ 64 bits
def _k2(shape):
    k = [2.0 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device="cuda") for n in shape[:2]]
    k.append(2.0 * math.pi * torch.fft.rfftfreq(shape[2], dtype=torch.float64, device="cuda"))
    return k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2


def _vm_rhs(c):
    """div(M(c) grad mu), conservative second-order differences on unit voxels."""
    mu = c * (c * c - 1.0)
    mu += 6.0 * KAPPA * c
    for d in range(3):
        mu -= KAPPA * (torch.roll(c, 1, d) + torch.roll(c, -1, d))
    m = MOB * torch.clamp(1.0 - c * c, min=0.0)
    rhs = torch.zeros_like(c)
    for d in range(3):
        flux = 0.5 * (m + torch.roll(m, -1, d)) * (torch.roll(mu, -1, d) - mu)
        rhs += flux - torch.roll(flux, 1, d)
    return rhs


def _exact_solve(case, seed):
    shape, model = _shape(case), case["model"]
    if shape[0] * shape[1] * shape[2] * case["steps"] > 2e10:
        return None
    c = _noise(shape, seed, case["mean"]).double()
    k2 = _k2(shape)
    if model == "vm":
        pre = DT / (1.0 + DT * MOB * KAPPA * k2 * k2)
        for _ in range(case["steps"]):
            c += torch.fft.irfftn(pre * torch.fft.rfftn(_vm_rhs(c)), s=shape)
    else:
        num = -DT * MOB * (k2 if model == "ch" else torch.ones_like(k2))
        den = 1.0 / (1.0 + DT * MOB * KAPPA * (k2 * k2 if model == "ch" else k2))
        for _ in range(case["steps"]):
            h = torch.fft.rfftn(c)
            h += num * torch.fft.rfftn(c * c * c - c)
            h *= den
            c = torch.fft.irfftn(h, s=shape)
            del h
    out = [c.cpu() if case["host"] else c]
    if case["energy"]:
        e = float(((c * c - 1.0) ** 2).sum()) / 4.0
        if model == "vm":
            for d in range(3):
                e += 0.5 * KAPPA * float(((torch.roll(c, -1, d) - c) ** 2).sum())
        else:
            w = torch.full((shape[2] // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
            w[0] = w[-1] = 1.0
            e += 0.5 * KAPPA * float((w * k2 * torch.fft.rfftn(c).abs().square()).sum()) / c.numel()
        out += [e, float(c.sum())]
    return out


def _exact_inverse(case, seed):
    shape = _shape(case)
    k2 = _k2(shape)

    def solve(c, kappa, mob):
        for _ in range(case["steps"]):
            h = torch.fft.rfftn(c) - DT * mob * k2 * torch.fft.rfftn(c * c * c - c)
            c = torch.fft.irfftn(h / (1.0 + DT * mob * kappa * k2 * k2), s=shape)
        return c

    c0 = _noise(shape, seed).double()
    with torch.no_grad():
        target = solve(c0, 1.5, 0.8).float().double()
    c0.requires_grad_(True)
    kappa = torch.tensor(KAPPA, dtype=torch.float64, device="cuda", requires_grad=True)
    mob = torch.tensor(MOB, dtype=torch.float64, device="cuda", requires_grad=True)
    c = solve(c0, kappa, mob)
    (0.5 * (c - target).square().sum()).backward()
    return dict(c=c.detach(), dc0=c0.grad, dkappa=kappa.grad, dM=mob.grad)


def _taps():
    return [(t, (t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1)) for t in range(27)]


def _shifted(x, off):
    """x(v + off), periodic, of [B][X][Y][Z][C]."""
    return torch.roll(x, [-o for o in off], (1, 2, 3))


def _exact_layer(case, seed):
    s = _layer_inputs(case, seed)
    x, dy, w, b, u = (s[k].double() for k in ("x", "dy", "w", "b", "u"))
    pre, du, dw = b.expand_as(x).clone(), torch.zeros_like(x), torch.zeros_like(w)
    for t, off in _taps():
        xs = _shifted(x, off)
        pre += xs @ w[t].T
        dw[t] = dy.reshape(-1, 32).T @ xs.reshape(-1, 32)
        du += _shifted(dy, [-o for o in off]) @ w[t]
        del xs
    phi = 0.5 * (1.0 + torch.erf(u / math.sqrt(2.0)))
    du *= phi + u * torch.exp(-0.5 * u * u) / math.sqrt(2.0 * math.pi)
    act = 0.5 * pre * (1.0 + torch.erf(pre / math.sqrt(2.0)))
    return dict(pre=pre, act=act, du=du, dw=dw, db=dy.sum((0, 1, 2, 3)))


def exact(case, seed):
    """None where a value in 64 bits needs a whole network or too long."""
    if case["kind"] == "solve":
        return _exact_solve(case, seed)
    if case["kind"] == "inverse":
        return _exact_inverse(case, seed)
    if case["kind"] == "layer":
        return _exact_layer(case, seed)
    return None


# --------------------------------------------------------------------- work
def work(case):
    V = case["nx"] * case["ny"] * case["nz"]
    fft = 2.5 * V * math.log2(V)  # one real transform
    if case["kind"] == "solve":
        n = case["steps"]
        # the field in and out; every step reads and writes the state and transforms twice
        return dict(bytes=8.0 * V + 8.0 * V * n, flops=n * (2 * fft + 20.0 * V))
    if case["kind"] == "inverse":
        n = case["steps"]
        # forward; backward: the forward states again and the adjoint state, each read and written per step
        return dict(bytes=16.0 * V + 8.0 * V * n * 3, flops=n * (2 + 2 + 4) * fft)
    nvox = V * case["batch"]
    conv = 2.0 * 27 * 32 * 32 * nvox
    act = 64.0 * nvox
    if case["kind"] == "layer":
        # x, dy and u in; the pre-activation, the activation and du out
        return dict(bytes=6 * act, flops=3 * conv)
    if case["kind"] == "train":
        # fields in and out; the activations a backward pass needs, written and read once (lift, and two per block)
        return dict(bytes=4.0 * 4 * nvox + 2 * 9 * act, flops=(8 * 3 + 4 * 2.0 / 32) * conv)
    # base, guard energies (two transforms each way and one) and the network's eight layers
    return dict(bytes=4.0 * 4 * nvox, flops=(8 + 2.0 / 32) * conv + case["batch"] * 8 * fft)
