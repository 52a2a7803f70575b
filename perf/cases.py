"""The solver calls whose speed is measured, with inputs, minimal work and 64-bit results.

Every case is a call that a program using this package makes: real- or imaginary-time steps of a spinor or
a batch, a relaxation, host spinors, the diagnostics between two runs, and training and inference of the
warm-start network.  Grid sizes are powers of two (the package takes no others); raggedness is nx != ny,
odd instance counts and batches of several grid sizes.

The calls step their spinor in place, so a second pass on a state goes on from the first, as the time loop
of a program does.  Outputs of complex64 runs that the library hands out as FP64 sums (energies) are
returned in single precision: they carry no more digits than the spinor.
"""
import functools
import math

import numpy as np
import torch

import paper_2010_15069_gb300 as sp

MODES = {"total": sp.SPGPE_NORM_TOTAL, "per": sp.SPGPE_NORM_PER_COMPONENT}
FNO_IN, FNO_OUT = 6, 4


def listed():
    return [
        # The plain method's 64^2 problem in complex128: the smallest grid, where every launch counts.
        dict(name="imag-64-c128", kind="imag", dtype="c128", nx=64, ny=64, ninst=1, steps=100, box=10.0, dt=1e-3,
             g=100.0, g12=95.0, omega=0.0, slope=0.0, kL=0.0, pot="sep", norm="per", lagged=False, start="gauss"),
        # Spin-Hall geometry at 256^2, one instance in real time: a run of a single experiment.
        dict(name="real-256-c64", kind="real", dtype="c64", nx=256, ny=256, ninst=1, steps=100, box=10.0, dt=5e-4,
             g=200.0, g12=200.0, omega=2.0, slope=0.5, kL=1.0, pot="sep", start="cloud"),
        # Ground-state search of the paper's 1024^2 example with the exact renormalisation.
        dict(name="imag-1024-c64", kind="imag", dtype="c64", nx=1024, ny=1024, ninst=1, steps=20, box=24.0, dt=1e-3,
             g=1000.0, g12=900.0, omega=4.0, slope=0.2, kL=2.0, pot="sep", norm="total", lagged=False, start="vortex"),
        # The parameter sweep over three grid sizes, lagged renormalisation: the main batched workload.
        dict(name="sweep-c64", kind="sweep", dtype="c64", n256=64, n512=16, n1024=4, steps=10, dt=5e-3, where="gpu"),
        # One eighth of the sweep in complex128 through relax(): the polish stage that decides a residual of 1e-8.
        dict(name="relax-c128", kind="relax", dtype="c128", n256=8, n512=2, n1024=1, steps=20, check=10, dt=5e-3),
        # 256 instances of the 256^2 problem in real time: an ensemble of noisy initial states.
        dict(name="real-256x256-c64", kind="real", dtype="c64", nx=256, ny=256, ninst=256, steps=10, box=10.0, dt=5e-4,
             g=200.0, g12=200.0, omega=2.0, slope=0.5, kL=1.0, pot="sep", start="cloud"),
        # The 2048^2 trap quench: the largest grid that is run for thousands of steps.
        dict(name="real-2048-c64", kind="real", dtype="c64", nx=2048, ny=2048, ninst=1, steps=20, box=24.0, dt=5e-4,
             g=1000.0, g12=900.0, omega=2.0, slope=0.2, kL=1.0, pot="sep", start="vortex"),
        # An elongated grid with potentials given as 2D arrays (trap, detuning and Raman profile), three instances.
        dict(name="real-1024x512-2d", kind="real", dtype="c64", nx=1024, ny=512, ninst=3, steps=20, box=16.0, dt=5e-4,
             g=500.0, g12=450.0, omega=2.0, slope=0.3, kL=1.0, pot="2d", start="cloud"),
        # The sweep batch kept in pinned host memory, one step per call: copies in and out with every call.
        dict(name="sweep-host", kind="sweep", dtype="c64", n256=64, n512=16, n1024=4, steps=1, dt=5e-3, where="host"),
        # Diagnostics between two runs of a batch: energies, atom numbers and the observables of the ground states.
        dict(name="diagnose-512", kind="diag", dtype="c64", nx=512, ny=512, ninst=16, box=12.0, g=500.0, g12=450.0,
             omega=3.0, slope=0.5, kL=1.0),
        # Training of the warm-start network at its full size: optimiser steps, then the weights out.
        dict(name="fno-train", kind="train", n=256, batch=4, width=64, modes=32, layers=4, hidden=128, steps=8, lr=1e-4),
        # Its proposals for a batch of 512^2 solves.
        dict(name="fno-infer-512", kind="infer", n=512, batch=4, width=64, modes=32, layers=4, hidden=128),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["real", "real", "imag", "imag", "sweep", "relax", "diag", "train", "infer"])
    c128 = rng.random() < 0.3
    if kind in ("real", "imag", "diag"):
        cap = 2 ** 20 if c128 else 2 ** 23  # grid points of one component, all instances
        while True:
            nx, ny = (2 ** rng.randint(6, 12) for _ in range(2))
            if nx * ny <= cap and max(nx, ny) <= 16 * min(nx, ny):
                break
        ninst = _log_int(rng, 1, max(1, min(256, cap // (nx * ny))))
        c = dict(kind=kind, dtype="c128" if c128 else "c64", nx=nx, ny=ny, ninst=ninst, box=rng.uniform(8.0, 24.0),
                 g=math.exp(rng.uniform(math.log(50.0), math.log(2000.0))), omega=rng.choice([0.0, rng.uniform(0.0, 6.0)]),
                 slope=rng.uniform(0.0, 1.0), kL=rng.uniform(0.0, 2.0))
        c["g12"] = c["g"] * rng.uniform(0.8, 1.2)
        if kind == "diag":
            return c
        most = (2 ** 22 if c128 else 2 ** 26) // (nx * ny * ninst)
        c.update(steps=_log_int(rng, 2, max(2, min(200, most))), dt=rng.uniform(2e-4, 1e-3), pot=rng.choice(["sep", "sep", "2d"]),
                 start=rng.choice(["gauss", "cloud", "vortex"]))
        if kind == "imag":
            c.update(norm=rng.choice(["total", "per"]), lagged=rng.random() < 0.5, dt=rng.uniform(1e-3, 5e-3))
        return c
    if kind == "sweep":
        host = rng.random() < 0.3
        return dict(kind="sweep", dtype="c64", n256=rng.randint(1, 64), n512=rng.randint(1, 16), n1024=rng.randint(1, 4),
                    steps=1 if host else rng.randint(2, 10), dt=rng.uniform(1e-3, 5e-3), where="host" if host else "gpu")
    if kind == "relax":
        dt = "c128" if c128 else "c64"
        check = rng.randint(4, 10)
        return dict(kind="relax", dtype=dt, n256=rng.randint(1, 8), n512=rng.randint(1, 2), n1024=rng.randint(0, 1), steps=2 * check,
                    check=check, dt=rng.uniform(1e-3, 5e-3))
    n, width = 2 ** rng.randint(6, 9 if kind == "infer" else 8), rng.choice([32, 64])
    c = dict(kind=kind, n=n, batch=rng.randint(1, 8 if n < 256 else 4), width=width, modes=rng.choice([12, 16, 24, 32]),
             layers=rng.choice([2, 3, 4]), hidden=2 * width)
    if kind == "train":
        c.update(steps=rng.randint(2, 8), lr=1e-4)
    return c


# ---------------------------------------------------------------- inputs

def _rng(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (2 ** 62))


def _axes(n, box):
    return -box + (2.0 * box / n) * torch.arange(n, dtype=torch.float64, device="cuda")


def _spinor(nx, ny, box, start, gen, g):
    """One seeded spinor (2, ny, nx), complex128, each component with half an atom."""
    x, y = _axes(nx, box)[None, :], _axes(ny, box)[:, None]
    r2 = x * x + y * y
    if start == "vortex":  # a wide envelope with 20 vortices, opposite windings in the two components
        radius = 0.42 * box
        u = torch.rand(20, 2, generator=gen, dtype=torch.float64, device="cuda")
        z = torch.ones(ny, nx, dtype=torch.complex128, device="cuda")
        for r, t in u.tolist():
            a, b = radius * math.sqrt(r) * math.cos(2 * math.pi * t), radius * math.sqrt(r) * math.sin(2 * math.pi * t)
            z *= torch.complex((x - a).expand(ny, nx), (y - b).expand(ny, nx))
            z /= z.abs() + 1e-30
        env = torch.exp(-r2 / (2 * radius * radius))
        psi = torch.stack([env * z, env * z.conj()])
    else:  # the Gaussian of the trap, or the density profile of a repulsive cloud; 1e-3 phase noise
        if start == "gauss":
            env = torch.exp(-r2 / 2)
        else:
            mu = math.sqrt(g / math.pi)
            env = torch.sqrt(torch.nn.functional.softplus(mu - r2 / 2, beta=4.0))
        ph = 1e-3 * (2 * torch.rand(2, ny, nx, generator=gen, dtype=torch.float64, device="cuda") - 1)
        psi = env * torch.exp(1j * ph)
    w = (2 * box / nx) * (2 * box / ny)
    return psi * torch.sqrt(0.5 / (w * (psi.abs() ** 2).sum((1, 2), keepdim=True)))


def _ctype(case):
    return torch.complex64 if case["dtype"] == "c64" else torch.complex128


def _grids(case):
    """[(nx, ny, ninst, box, [(g, g12, omega, slope, kL) per instance])], one entry per grid size."""
    if case["kind"] in ("sweep", "relax"):
        out, rnd = [], np.random.RandomState(3)  # the sweep's parameters: the batch's, not the seed's
        for n, k in ((256, case["n256"]), (512, case["n512"]), (1024, case["n1024"])):
            u = rnd.rand(k, 4)
            p = [(50.0 * 40.0 ** a, 50.0 * 40.0 ** a * (0.8 + 0.4 * b), 6.0 * o, s, 1.0) for a, b, o, s in u.tolist()]
            if k:
                out.append((n, n, k, 12.0, p))
        return out
    p = (case["g"], case["g12"], case["omega"], case["slope"], case["kL"])
    return [(case["nx"], case["ny"], case["ninst"], case["box"], [p] * case["ninst"])]


def _spinors(case, seed):
    """The batch's spinors, a list of (ninst, 2, ny, nx) tensors in the case's precision."""
    start = case.get("start", "vortex" if case["kind"] != "diag" else "cloud")
    out = []
    for k, (nx, ny, n, box, prm) in enumerate(_grids(case)):
        t = torch.empty(n, 2, ny, nx, dtype=_ctype(case), device="cuda")
        for i in range(n):
            t[i] = _spinor(nx, ny, box, start, _rng(seed, 4096 * k + i), prm[i][0])
        out.append(t)
    return out


def _pieces(nx, ny, box, prm):
    """Potential pieces as FP64 numpy arrays: (Vx, Vy, delta_y, Omega_y)."""
    x, y = _axes(nx, box).cpu().numpy(), _axes(ny, box).cpu().numpy()
    return 0.5 * x * x, 0.5 * y * y, prm[3] * y, np.full(ny, prm[2])


def _maps(case):
    """2D trap, detuning and Raman arrays (ny, nx): an anharmonic trap, a detuning gradient with a ripple and a
    Raman beam of finite waist."""
    nx, ny, box = case["nx"], case["ny"], case["box"]
    x, y = _axes(nx, box).cpu().numpy()[None, :], _axes(ny, box).cpu().numpy()[:, None]
    V = 0.5 * (x * x + y * y) * (1.0 + 1e-3 * x * x)
    delta = case["slope"] * y + 0.1 * np.cos(x)
    return V, np.broadcast_to(delta, V.shape).copy(), case["omega"] * np.exp(-(x * x + y * y) / (box * box))


def _features(case, seed):
    """Input fields and targets (samples, channels, n, n) of the warm-start network: coordinates, detuning and
    couplings of a draw of the sweep, and a trapped spinor of such an instance."""
    n, box, gen = case["n"], 12.0, _rng(seed, 7)
    count = case["batch"] * case.get("steps", 1)
    u = torch.rand(count, 4, generator=gen, dtype=torch.float64, device="cuda")
    x, y = _axes(n, box)[None, :] / box, _axes(n, box)[:, None] / box
    a = torch.empty(count, FNO_IN, n, n, device="cuda")
    t = torch.empty(count, FNO_OUT, n, n, device="cuda")
    for i, (g, b, o, s) in enumerate(u.tolist()):
        a[i, 0], a[i, 1], a[i, 2] = x, y, s * y
        a[i, 3], a[i, 4], a[i, 5] = o, g, 2.0 * b - 1.0
        z = 10.0 * _spinor(n, n, box, "cloud", gen, 50.0 * 40.0 ** g)
        turn = torch.exp(1j * (3.0 * o * x - 2.0 * s * y))
        t[i] = torch.stack([(z[0] * turn).real, (z[0] * turn).imag, (z[1] * turn.conj()).real, (z[1] * turn.conj()).imag])
    return a, t


def _layout(case):
    """[(name, shape, scale)] of the network's flat parameter vector."""
    W, M, H = case["width"], case["modes"], case["hidden"]
    out = [("P", (W, FNO_IN), 1 / math.sqrt(FNO_IN)), ("p", (W,), 0.05)]
    for k in range(case["layers"]):
        out += [("W%d" % k, (W, W), 1 / math.sqrt(W)), ("w%d" % k, (W,), 0.05), ("R%d" % k, (2 * M, M, W, W, 2), 1 / W)]
    return out + [("Q1", (H, W), 1 / math.sqrt(W)), ("q1", (H,), 0.05), ("Q2", (FNO_OUT, H), 1 / math.sqrt(H)),
                  ("q2", (FNO_OUT,), 0.05)]


def _weights(case, seed):
    gen = _rng(seed, 11)
    return torch.cat([s * (2 * torch.rand(math.prod(shape), generator=gen, device="cuda") - 1)
                      for _, shape, s in _layout(case)])


# ------------------------------------------------------------------- cases

@functools.cache
def _solver_stream():
    """The one stream that the program runs its solver on (not the legacy default stream: relax() replays graphs)."""
    return torch.cuda.Stream()


def prepare(case, seed):
    if case["kind"] in ("train", "infer"):
        net = sp.FNO(FNO_IN, FNO_OUT, width=case["width"], modes=case["modes"], layers=case["layers"], hidden=case["hidden"],
                     seed=1)
        net.set_params(_weights(case, seed).cpu().numpy())
        a, t = _features(case, seed)
        B = case["batch"]
        return dict(case=case, net=net, a=[x.contiguous() for x in a.split(B)], t=[x.contiguous() for x in t.split(B)])
    psi, grids, stream = _spinors(case, seed), _grids(case), _solver_stream()
    if case["kind"] in ("sweep", "relax"):
        ctx = sp.Context.multi([(nx, ny, n, box, box) for nx, ny, n, box, _ in grids], case["dtype"], stream=stream)
        psi = torch.cat([t.reshape(-1) for t in psi])
    else:
        nx, ny, n, box, _ = grids[0]
        ctx, psi = sp.Context(nx, ny, box, box, case["dtype"], ninst=n, stream=stream), psi[0]
    if case.get("pot") == "2d":
        V, delta, Omega = _maps(case)
        ctx.set_potentials(V, delta, Omega, g11=case["g"], g22=case["g"], g12=case["g12"], kL=case["kL"])
    else:
        i = 0
        for nx, ny, n, box, prm in grids:
            for k in range(n) if case["kind"] in ("sweep", "relax") else [None]:
                q = prm[k or 0]
                vx, vy, dy, oy = _pieces(nx, ny, box, q)
                ctx.set_potentials_separable(-1 if k is None else i, Vx=vx, Vy=vy, delta_y=dy, Omega_y=oy, g11=q[0], g22=q[0],
                                             g12=q[1], kL=q[4])
                i += 1
    if case.get("where") == "host":
        host = torch.empty(psi.shape, dtype=psi.dtype, pin_memory=True)
        host.copy_(psi)
        psi = host.numpy()
    torch.cuda.synchronize()
    return dict(case=case, ctx=ctx, psi=psi)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        losses = [state["net"].train_step(a, t, case["lr"]) for a, t in zip(state["a"], state["t"])]
        return dict(loss=losses, weights=state["net"].get_params())
    if kind == "infer":
        return state["net"].forward(state["a"][0])
    ctx, psi = state["ctx"], state["psi"]
    if kind == "real":
        return ctx.step_real(psi, case["dt"], case["steps"])
    if kind == "imag":
        ctx.step_imag(psi, case["dt"], case["steps"], MODES[case["norm"]], lagged=case["lagged"])
        return psi
    if kind == "sweep":
        ctx.step_imag(psi, case["dt"], case["steps"], lagged=True)
        return psi
    if kind == "relax":  # a tolerance that no run of so few steps reaches
        res, steps = ctx.relax(psi, case["dt"], 1e-13, case["steps"], check_every=case["check"], lagged=True)
        return dict(psi=psi, residual=res.astype(_real(case)), steps=list(steps))
    energy, norm, obs = ctx.energy(psi), ctx.norm(psi), ctx.observables(psi)
    return dict(energy=energy.astype(_real(case)), norm=norm, observables=obs)


def _real(case):
    return np.float32 if case["dtype"] == "c64" else np.float64


def work(case):
    if case["kind"] in ("train", "infer"):
        n, B, W, M, L, H = (case[k] for k in ("n", "batch", "width", "modes", "layers", "hidden"))
        P, params = n * n, sum(math.prod(s) for _, s, _ in _layout(case))
        spectral = 2 * (2 * W * n * (2 * M) * n + 4 * W * 2 * M * M * n) + 8 * W * W * 2 * M * M
        fwd = 2 * P * (FNO_IN * W + L * W * W + W * H + H * FNO_OUT) + L * spectral
        if case["kind"] == "infer":
            return dict(bytes=B * P * 4 * (FNO_IN + FNO_OUT) + 2 * params, flops=B * fwd)
        S = case["steps"]  # the optimiser reads and writes weights and two moments each step, and the weights go out
        return dict(bytes=S * (B * P * 4 * (FNO_IN + FNO_OUT) + 24 * params) + 4 * params, flops=S * B * 3 * fwd)
    es = 8 if case["dtype"] == "c64" else 16
    byt = fl = 0.0
    for nx, ny, n, _, _ in _grids(case):
        pts, ffts = nx * ny * n, 10.0 * math.log2(nx * ny)  # one 2D transform of both components, per point
        byt += 2 * pts * es * (1 if case["kind"] == "diag" else 2)
        if case["kind"] == "diag":
            fl += pts * (ffts + 60)
        else:
            fl += pts * case["steps"] * (2 * ffts + 2 * 48 + 12)
    return dict(bytes=byt, flops=fl)


# ------------------------------------------------------- results in 64 bits

class _Model:
    """The split step of one grid size and its instances, in complex128 with torch's transforms."""

    def __init__(self, case, nx, ny, box, prm):
        self.w = (2 * box / nx) * (2 * box / ny)
        x, y = _axes(nx, box)[None, None, :], _axes(ny, box)[None, :, None]
        col = lambda k: torch.tensor([p[k] for p in prm], dtype=torch.float64, device="cuda")[:, None, None]  # noqa: E731
        self.g, self.g12, kL = col(0), col(1), col(4)
        if case.get("pot") == "2d":
            self.V, self.delta, self.Omega = (torch.from_numpy(m).cuda()[None] for m in _maps(case))
        else:
            self.V, self.delta, self.Omega = 0.5 * (x * x + y * y), col(3) * y, col(2)
        kx = 2 * math.pi * torch.fft.fftfreq(nx, 2 * box / nx, dtype=torch.float64, device="cuda")[None, None, :]
        ky = 2 * math.pi * torch.fft.fftfreq(ny, 2 * box / ny, dtype=torch.float64, device="cuda")[None, :, None]
        k2 = 0.5 * (kx * kx + ky * ky)
        self.T = torch.stack([k2 - kL * kx, k2 + kL * kx], 1)

    def half(self, psi, f, dt):
        """R(dt/2) = X(dt/4) D(dt/2) X(dt/4); f = -i in real time, -1 in imaginary time."""
        th = f * self.Omega * (dt / 8)
        c, s = torch.cosh(th), torch.sinh(th)
        u, d = c * psi[:, 0] + s * psi[:, 1], s * psi[:, 0] + c * psi[:, 1]
        ru, rd = u.abs() ** 2, d.abs() ** 2
        u = u * torch.exp(f * (dt / 2) * (self.V + self.delta / 2 + self.g * ru + self.g12 * rd))
        d = d * torch.exp(f * (dt / 2) * (self.V - self.delta / 2 + self.g * rd + self.g12 * ru))
        return torch.stack([c * u + s * d, s * u + c * d], 1)

    def kinetic(self, psi, f, dt):
        return torch.fft.ifft2(torch.exp(f * dt * self.T) * torch.fft.fft2(psi))

    def real(self, psi, dt, steps):
        f = torch.tensor(-1j, dtype=torch.complex128, device="cuda")
        for _ in range(steps):
            psi = self.half(self.kinetic(self.half(psi, f, dt), f, dt), f, dt)
        return psi

    def scale(self, psi, norm):
        n = self.w * (psi.abs() ** 2).sum((2, 3), keepdim=True)
        return torch.sqrt(0.5 / n) if norm == "per" else torch.sqrt(1.0 / n.sum(1, keepdim=True)).expand_as(n)

    def imag(self, psi, dt, steps, norm, lagged, residual=False):
        """Imaginary-time steps; lagged: a boundary hands the next step the spinor scaled by the scale of the
        boundary before, and the ratio of the two follows after the opening half step (the first boundary of a
        call, the one before a step whose residual is measured and the last are exact)."""
        f, prev, late, before = -1.0, None, None, psi
        for n in range(1, steps + 1):
            psi = self.half(psi, f, dt)
            if late is not None:
                psi, late = psi * late, None
            psi = self.half(self.kinetic(psi, f, dt), f, dt)
            s = self.scale(psi, norm)
            if lagged and 1 < n < steps - (1 if residual else 0):
                psi, late = psi * prev, s / prev
            else:
                psi = psi * s
            prev = s
            if n == steps - 1:
                before = psi
        if not residual:
            return psi, None
        num, den = ((q.abs() ** 2).sum((1, 2, 3)) for q in (psi - before, before))
        return psi, torch.sqrt(num / den) / dt

    def energy(self, psi):
        nx, ny = psi.shape[3], psi.shape[2]
        ru, rd = psi[:, 0].abs() ** 2, psi[:, 1].abs() ** 2
        kin = (self.T * torch.fft.fft2(psi).abs() ** 2).sum((1, 2, 3)) / (nx * ny)
        e = [kin, (self.V * (ru + rd)).sum((1, 2)), (0.5 * self.delta * (ru - rd)).sum((1, 2)),
             (self.Omega * (psi[:, 0].conj() * psi[:, 1]).real).sum((1, 2)),
             (0.5 * self.g * (ru * ru + rd * rd) + self.g12 * ru * rd).sum((1, 2))]
        return self.w * torch.stack([sum(e)] + e, 1)


def _network(case, theta, a):
    """Output fields of the network: weights rounded to bfloat16, everything else in 64 bits."""
    P, o = {}, 0
    for name, shape, _ in _layout(case):
        k = math.prod(shape)
        P[name], o = theta[o:o + k].reshape(shape), o + k
    n, M, dev = case["n"], case["modes"], "cuda"
    idx = torch.arange(n, device=dev, dtype=torch.float64)
    ky = torch.cat([torch.arange(M), torch.arange(n - M, n)]).to(dev).double()
    Ex = torch.exp(-2j * math.pi * torch.remainder(torch.outer(idx, torch.arange(M, device=dev).double()), n) / n)
    Ey = torch.exp(-2j * math.pi * torch.remainder(torch.outer(ky, idx), n) / n)
    wt = torch.full((M,), 2.0, dtype=torch.float64, device=dev)
    wt[0] = 1.0
    lin = lambda w, b, v: torch.einsum("oc,bcyx->boyx", w, v) + b[None, :, None, None]  # noqa: E731
    v = lin(P["P"], P["p"], a)
    for k in range(case["layers"]):
        vh = Ey @ (v.to(torch.complex128) @ Ex)
        oh = torch.einsum("jkoc,bcjk->bojk", torch.view_as_complex(P["R%d" % k].contiguous()), vh) * wt
        s = (Ey.conj().T @ oh @ Ex.conj().T).real / (n * n)
        v = lin(P["W%d" % k], P["w%d" % k], v) + s
        if k < case["layers"] - 1:
            v = torch.nn.functional.gelu(v)
    return lin(P["Q2"], P["q2"], torch.nn.functional.gelu(lin(P["Q1"], P["q1"], v)))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "infer"):
        a, t = _features(case, seed)
        w = _weights(case, seed).double()
        rounded = lambda: w.float().bfloat16().double()  # noqa: E731
        B = case["batch"]
        if kind == "infer":
            with torch.no_grad():
                return torch.cat([_network(case, rounded(), a[i:i + 1].double()) for i in range(B)])
        m, v, losses = torch.zeros_like(w), torch.zeros_like(w), []
        for k in range(case["steps"]):
            th = rounded().requires_grad_()
            total = 0.0
            for i in range(k * B, (k + 1) * B):
                out, y = _network(case, th, a[i:i + 1].double()), t[i:i + 1].double()
                part = ((out - y) ** 2).sum() / (y ** 2).sum() / B
                part.backward()
                total += part.item()
            losses.append(torch.tensor(total, dtype=torch.float64))
            m = 0.9 * m + 0.1 * th.grad
            v = 0.999 * v + 0.001 * th.grad ** 2
            w = w - case["lr"] * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1 - 0.999 ** (k + 1))) + 1e-8)
        return dict(loss=losses, weights=w)
    outs, residuals, energies, norms, shapes = [], [], [], [], []
    for (nx, ny, n, box, prm), psi in zip(_grids(case), _spinors(case, seed)):
        m = _Model(case, nx, ny, box, prm)
        psi = psi.to(torch.complex128)
        if kind == "real":
            psi = m.real(psi, case["dt"], case["steps"])
        elif kind == "imag":
            psi, _ = m.imag(psi, case["dt"], case["steps"], case["norm"], case["lagged"])
        elif kind == "sweep":
            psi, _ = m.imag(psi, case["dt"], case["steps"], "total", True)
        elif kind == "relax":
            for _ in range(case["steps"] // case["check"]):
                psi, r = m.imag(psi, case["dt"], case["check"], "total", True, residual=True)
            residuals.append(r)
        else:
            energies.append(m.energy(psi))
            norms.append(m.w * (psi.abs() ** 2).sum((2, 3)))
            shapes.append((nx, ny, box, psi))
        outs.append(psi)
    if kind == "diag":
        return dict(energy=torch.cat(energies), norm=torch.cat(norms), observables=None)
    if kind == "relax":
        return dict(psi=torch.cat([p.reshape(-1) for p in outs]), residual=torch.cat(residuals), steps=None)
    if kind == "sweep":
        return torch.cat([p.reshape(-1) for p in outs])
    return outs[0]
