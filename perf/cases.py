"""The work that a program built on this package has it do, for timing and for
comparison between builds.

A case names its sizes and options; `prepare` makes what a program holds before
the call (particles or a density on the GPU, a solver handle), `run` is one
pass through the public entry points, `work` what a pass cannot do without,
and `exact` the same outputs from plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1611_09638_gb300 import Recon, reconstruct, solve_batch

# Seeds of the inputs are spread so that cases and members of a batch differ.
_STRIDE = 7919


# ----------------------------------------------------------------- the cases

def listed():
    return [
        # The smallest call: gridding a sparse catalogue on a coarse grid;
        # launches and the input checks' readback are all of it.
        {"name": "deposit_small", "kind": "deposit", "n": 64, "np": 100003, "mass": False, "cell": 3.125},
        # Gridding a large catalogue with masses, an odd number of particles.
        {"name": "deposit_large", "kind": "deposit", "n": 256, "np": 20000003, "mass": True, "cell": 1.5625},
        # One coarse mock from particles to the reconstructed density: bound by
        # launches and by the coarse end of the V-cycle.
        {"name": "mixed_32", "kind": "solve", "n": 32, "cell": 3.125, "order": 1, "precision": "mixed", "steps": 8,
         "update": 0},
        # The middle mock size: the finest level streams, the rest is small.
        {"name": "mixed_64", "kind": "solve", "n": 64, "cell": 3.125, "order": 1, "precision": "mixed", "steps": 8,
         "update": 0},
        # The ordinary single solve.
        {"name": "mixed_128", "kind": "solve", "n": 128, "cell": 1.5625, "order": 1, "precision": "mixed",
         "steps": 12, "update": 0},
        # A production grid, 2LPT, enough steps for the limiters to act.
        {"name": "mixed_256", "kind": "solve", "n": 256, "cell": 1.5625, "order": 2, "precision": "mixed",
         "steps": 10, "update": 0},
        # The largest: the paper's grid, the first steps of the solve.
        {"name": "mixed_512", "kind": "solve", "n": 512, "cell": 1.5625, "order": 2, "precision": "mixed",
         "steps": 4, "update": 0},
        # All arithmetic in FP64: what a user runs to check the mixed mode.
        {"name": "fp64_128", "kind": "solve", "n": 128, "cell": 1.5625, "order": 1, "precision": "fp64", "steps": 5,
         "update": 0},
        # App. A's own density update instead of moving tracers.
        {"name": "literal_128", "kind": "solve", "n": 128, "cell": 1.5625, "order": 1, "precision": "mixed",
         "steps": 8, "update": 1},
        # A survey slab on an anisotropic grid, from a density grid: nodal
        # coarse levels, none of the cubic-grid paths.
        {"name": "slab", "kind": "slab", "n0": 128, "n1": 64, "n2": 32, "precision": "mixed", "steps": 6},
        # Mock catalogues of three sizes solved together on their own streams.
        {"name": "batch", "kind": "batch", "small": 6, "middle": 4, "large": 2, "steps": 8},
        # A gradient: the differentiable reconstruction, forward and backward.
        {"name": "adjoint_128", "kind": "adjoint", "n": 128, "cell": 1.5625, "precision": "mixed", "steps": 6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["deposit", "solve", "solve", "solve", "slab", "batch", "adjoint"])
    cell = round(rng.uniform(1.5625, 3.125), 3)
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    if kind == "deposit":
        return {"kind": kind, "n": rng.choice([32, 64, 128, 256]), "np": _log_int(rng, 50001, 20000000) | 1,
                "mass": rng.random() < 0.5, "cell": cell}
    if kind == "solve":
        n = rng.choice([32, 64, 128, 256] if precision == "mixed" else [32, 64, 128])
        update = 1 if rng.random() < 0.2 else 0
        most = 12 if precision == "mixed" else 8
        return {"kind": kind, "n": n, "cell": cell, "order": rng.choice([1, 2]), "precision": precision,
                "steps": rng.randint(2, most), "update": update}
    if kind == "slab":
        n0, n1, n2 = (rng.choice([16, 32, 64, 128]) for _ in range(3))
        return {"kind": kind, "n0": n0, "n1": n1, "n2": n2, "precision": precision, "steps": rng.randint(2, 6)}
    if kind == "batch":
        return {"kind": kind, "small": rng.randint(1, 6), "middle": rng.randint(1, 4), "large": rng.randint(0, 2),
                "steps": rng.randint(3, 8)}
    return {"kind": kind, "n": rng.choice([32, 64, 128]), "cell": cell, "precision": precision,
            "steps": rng.randint(2, 6)}


# ------------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _wavenumbers(n, box):
    kf = 2.0 * math.pi / box
    k1 = torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) * kf
    kr = torch.fft.rfftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64) * kf
    return k1[:, None, None], k1[None, :, None], kr[None, None, :]


def _spectrum(n, box, seed):
    """Fourier modes of a Gaussian field with the BBKS spectrum (Gamma = 0.2,
    n_s = 1) and the variance of sigma_8 = 0.8; no mean and no Nyquist modes."""
    white = torch.randn((n, n, n), generator=_generator(seed), device="cuda", dtype=torch.float64)
    modes = torch.fft.rfftn(white)
    del white
    kx, ky, kz = _wavenumbers(n, box)
    k = torch.sqrt(kx * kx + ky * ky + kz * kz)
    q = k / 0.2
    t = torch.log1p(2.34 * q) / (2.34 * q) * (1.0 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
    power = k * torch.where(q > 0, t, torch.ones_like(t)) ** 2
    # the amplitude that sigma_8 = 0.8 asks for, by the trapezoidal rule over ln k
    lnk = np.linspace(math.log(1e-6), math.log(1e3), 20001)
    kk = np.exp(lnk)
    qq = kk / 0.2
    tt = np.log1p(2.34 * qq) / (2.34 * qq) * (1 + 3.89 * qq + (16.1 * qq) ** 2 + (5.46 * qq) ** 3 + (6.71 * qq) ** 4) ** -0.25
    x = 8.0 * kk
    f = kk ** 4 * tt ** 2 * (3.0 * (np.sin(x) - x * np.cos(x)) / x ** 3) ** 2 / (2.0 * math.pi ** 2)
    sigma2 = float(np.sum(0.5 * (f[1:] + f[:-1]) * np.diff(lnk)))
    scale = torch.sqrt(power * (0.64 / sigma2 * n ** 3 / box ** 3))
    scale[n // 2], scale[:, n // 2], scale[:, :, n // 2] = 0.0, 0.0, 0.0
    scale[0, 0, 0] = 0.0
    return modes * scale


def _particles(n, cell, order, seed):
    """One particle per node of an n^3 grid, moved by the Zel'dovich (order 1)
    or second-order displacement of such a field; positions in box units."""
    box = n * cell
    modes = _spectrum(n, box, seed)
    ks = _wavenumbers(n, box)
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    phi1 = -modes / k2
    del modes
    pot = -phi1
    if order >= 2:
        def second(a, b):
            return torch.fft.irfftn(-ks[a] * ks[b] * phi1, s=(n, n, n))
        xx, yy = second(0, 0), second(1, 1)
        src = xx * yy
        xx += yy
        del yy
        src += xx * second(2, 2)
        del xx
        for a, b in ((0, 1), (0, 2), (1, 2)):
            src -= second(a, b) ** 2
        phi2 = -torch.fft.rfftn(src) / k2
        del src
        phi2[0, 0, 0] = 0.0
        phi2[n // 2], phi2[:, n // 2], phi2[:, :, n // 2] = 0.0, 0.0, 0.0
        pot -= (3.0 / 7.0) * phi2
        del phi2
    del phi1, k2
    q = torch.arange(n, device="cuda", dtype=torch.float64) * cell
    pos = torch.empty((n, n, n, 3), device="cuda", dtype=torch.float64)
    for a, shape in enumerate(((n, 1, 1), (1, n, 1), (1, 1, n))):
        pos[..., a] = torch.fft.irfftn(1j * ks[a] * pot, s=(n, n, n)) + q.reshape(shape)
    return torch.remainder(pos.reshape(-1, 3), box).contiguous()


def _clustered(n, cell, count, mass, seed):
    """A catalogue of any number of particles: those of a displaced grid, each
    picked at random and scattered by a fraction of a cell."""
    base = _particles(min(n, 128), n * cell / min(n, 128), 1, seed)
    g = _generator(seed + 1)
    pick = torch.randint(0, base.shape[0], (count,), generator=g, device="cuda")
    pos = base[pick] + cell * 0.7 * torch.randn((count, 3), generator=g, device="cuda", dtype=torch.float64)
    pos = torch.remainder(pos, n * cell).contiguous()
    m = 0.5 + torch.rand((count,), generator=g, device="cuda", dtype=torch.float64) if mass else None
    return pos, m


def _lognormal(shape, seed):
    """A positive density on an anisotropic grid: smoothed noise, exponentiated."""
    w = torch.fft.rfftn(torch.randn(shape, generator=_generator(seed), device="cuda", dtype=torch.float64))
    for a, n in enumerate(shape):
        k = (torch.fft.rfftfreq if a == 2 else torch.fft.fftfreq)(n, device="cuda", dtype=torch.float64) * 2.0 * math.pi
        w = w * torch.exp(-0.5 * (1.2 * k) ** 2).reshape([-1 if b == a else 1 for b in range(3)])
    f = torch.fft.irfftn(w, s=shape)
    return torch.exp(0.7 * f / f.std()).contiguous()


def _mocks(case):
    sizes = [32] * case["small"] + [64] * case["middle"] + [128] * case["large"]
    return [(n, i) for i, n in enumerate(sizes)]


def _options(case):
    o = {"precision": case["precision"], "k_max": case["steps"]}
    if case.get("update"):
        o["density_update"] = 1
    return o


def prepare(case, seed):
    kind = case["kind"]
    if kind == "deposit":
        n = case["n"]
        pos, mass = _clustered(n, case["cell"], case["np"], case["mass"], seed)
        return {"kind": kind, "recon": Recon((n, n, n), box=n * case["cell"]), "pos": pos, "mass": mass}
    if kind == "slab":
        shape = (case["n0"], case["n1"], case["n2"])
        return {"kind": kind, "recon": Recon(shape, **_options(case)), "rho": _lognormal(shape, seed)}
    if kind == "batch":
        recons, poss = [], []
        for n, i in _mocks(case):
            poss.append(_particles(n, 3.125, 1, seed + _STRIDE * (i + 1)))
            recons.append(Recon((n, n, n), box=n * 3.125, precision="mixed", k_max=case["steps"],
                                stream=torch.cuda.Stream()))
        torch.cuda.synchronize()  # the handles' streams read inputs made on this one
        return {"kind": kind, "recons": recons, "pos": poss}
    n, cell = case["n"], case["cell"]
    pos = _particles(n, cell, case.get("order", 1), seed)
    if kind == "adjoint":
        recon = Recon((n, n, n), box=n * cell, checkpoint=1, **_options(case))
        recon.deposit_particles(pos)
        rho = recon.field("density").reshape(n, n, n).requires_grad_()
        grad = torch.randn((n, n, n), generator=_generator(seed + 2), device="cuda", dtype=torch.float64)
        return {"kind": kind, "recon": recon, "rho": rho, "grad": grad}
    return {"kind": kind, "recon": Recon((n, n, n), box=n * cell, **_options(case)), "pos": pos}


def _steps_of(recon, stats):
    """The step lengths taken, and 0 for the steps that a stall left out."""
    return np.pad(stats.alpha, (0, recon.params.k_max - stats.steps))


def run(state):
    kind = state["kind"]
    if kind == "batch":
        for recon, pos in zip(state["recons"], state["pos"]):
            recon.deposit_particles(pos)
        stats = solve_batch(state["recons"])
        return [{"phi": r.field("phi"), "delta_r": r.field("delta_r"), "alpha": _steps_of(r, s)}
                for r, s in zip(state["recons"], stats)]
    recon = state["recon"]
    if kind == "deposit":
        recon.deposit_particles(state["pos"], state["mass"])
        return {"density": recon.field("density")}
    if kind == "adjoint":
        delta_r = reconstruct(recon, state["rho"])
        (grad_rho,) = torch.autograd.grad(delta_r, state["rho"], state["grad"])
        return {"delta_r": delta_r.detach(), "grad_rho": grad_rho}
    if kind == "slab":
        recon.deposit_grid(state["rho"])
    else:
        recon.deposit_particles(state["pos"])
    stats = recon.solve()
    return {"phi": recon.field("phi"), "delta_r": recon.field("delta_r"), "alpha": _steps_of(recon, stats)}


# ---------------------------------------------------- what a pass has to do

def _solve_work(cells, particles, steps, update, fields=2):
    # the catalogue and the outputs once, and per step the state that a step
    # carries on (phi, and per tracer three offsets read and written and its
    # mass read, or the mass per cell read and written) and the linear
    # system's solution, written and read, all in FP64
    state = 16 + (16 if update else 56) + 16
    return {"bytes": 24 * particles + 8 * fields * cells + steps * state * cells,
            # a step's Hessian, determinant, source, smoothing, limiter and
            # advance, and at least four sweeps and residuals
            "flops": steps * cells * 400 + particles * 30}


def work(case):
    kind = case["kind"]
    if kind == "deposit":
        n, count = case["n"], case["np"]
        return {"bytes": count * (32 if case["mass"] else 24) + 8 * n ** 3, "flops": 30 * count}
    if kind == "slab":
        cells = case["n0"] * case["n1"] * case["n2"]
        w = _solve_work(cells, 0, case["steps"], 0)
        return {"bytes": w["bytes"] + 8 * cells, "flops": w["flops"]}
    if kind == "batch":
        ws = [_solve_work(n ** 3, n ** 3, case["steps"], 0) for n, _ in _mocks(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    cells = case["n"] ** 3
    if kind == "adjoint":
        w = _solve_work(cells, 0, case["steps"], 0, fields=4)
        # the step states written on the way and read on the way back, and a
        # backward step's work like a forward one's
        return {"bytes": w["bytes"] + case["steps"] * (80 + 88) * cells, "flops": 2 * w["flops"]}
    return _solve_work(cells, cells, case["steps"], case["update"])


# -------------------------------------------- the same outputs in plain torch

def _cic(shape, x, w):
    """Cloud-in-cell deposit of points x (grid units) with masses w."""
    base = torch.floor(x)
    f = x - base
    base = base.to(torch.int64)
    out = torch.zeros(shape[0] * shape[1] * shape[2], device=x.device, dtype=torch.float64)
    for corner in range(8):
        at, q = 0, w
        for a in range(3):
            d = (corner >> a) & 1
            at = at * shape[a] + torch.remainder(base[:, a] + d, shape[a])
            q = q * (f[:, a] if d else 1.0 - f[:, a])
        out.index_add_(0, at, q)
    return out.reshape(shape)


def _gather(field, x):
    shape = field.shape
    base = torch.floor(x)
    f = x - base
    base = base.to(torch.int64)
    out = torch.zeros(x.shape[0], device=x.device, dtype=torch.float64)
    flat = field.reshape(-1)
    for corner in range(8):
        at, q = 0, 1.0
        for a in range(3):
            d = (corner >> a) & 1
            at = at * shape[a] + torch.remainder(base[:, a] + d, shape[a])
            q = q * (f[:, a] if d else 1.0 - f[:, a])
        out += q * flat[at]
    return out


def _at(f, *steps):
    """f at the neighbour reached by (axis, +-1) steps."""
    for a, s in steps:
        f = torch.roll(f, -s, a)
    return f


def _hessian(f):
    h = {}
    for a in range(3):
        h[a, a] = _at(f, (a, 1)) - 2.0 * f + _at(f, (a, -1))
        for b in range(a + 1, 3):
            h[a, b] = 0.25 * (_at(f, (a, 1), (b, 1)) - _at(f, (a, 1), (b, -1)) - _at(f, (a, -1), (b, 1))
                              + _at(f, (a, -1), (b, -1)))
    return h


def _det(e):
    return (e[0, 0] * (e[1, 1] * e[2, 2] - e[1, 2] ** 2) - e[0, 1] * (e[0, 1] * e[2, 2] - e[1, 2] * e[0, 2])
            + e[0, 2] * (e[0, 1] * e[1, 2] - e[1, 1] * e[0, 2]))


def _min_eig(e):
    """Smallest eigenvalue of symmetric 3 x 3 matrices: the trigonometric
    closed form, then Newton steps on the characteristic polynomial."""
    q = (e[0, 0] + e[1, 1] + e[2, 2]) / 3.0
    p2 = sum((e[a, a] - q) ** 2 for a in range(3)) + 2.0 * (e[0, 1] ** 2 + e[0, 2] ** 2 + e[1, 2] ** 2)
    p = torch.sqrt(p2 / 6.0).clamp_min(1e-300)
    b = {k: (v - q if k[0] == k[1] else v) / p for k, v in e.items()}
    lam = q + 2.0 * p * torch.cos(torch.acos((0.5 * _det(b)).clamp(-1.0, 1.0)) / 3.0 + 2.0 * math.pi / 3.0)
    for _ in range(3):
        c = {k: (v - lam if k[0] == k[1] else v) for k, v in e.items()}
        d = -((c[1, 1] * c[2, 2] - c[1, 2] ** 2) + (c[0, 0] * c[2, 2] - c[0, 2] ** 2)
              + (c[0, 0] * c[1, 1] - c[0, 1] ** 2))
        step = torch.where(d != 0.0, _det(c) / d, torch.zeros_like(d))
        lam = torch.where(step.abs() < 1e-6, lam - step, lam)
    return lam


def _smooth(f):
    for a in range(3):
        f = 0.5 * f + 0.25 * (_at(f, (a, 1)) + _at(f, (a, -1)))
    return f


def _laplacian_inverse(shape):
    sym = 0.0
    for a, n in enumerate(shape):
        k = torch.arange(n // 2 + 1 if a == 2 else n, device="cuda", dtype=torch.float64) * (2.0 * math.pi / n)
        sym = sym + (2.0 - 2.0 * torch.cos(k)).reshape([-1 if b == a else 1 for b in range(3)])
    sym[0, 0, 0] = 1.0
    inv = 1.0 / sym
    inv[0, 0, 0] = 0.0
    return inv


def _elliptic(a, s, u, inv):
    """div(a grad u) = s by conjugate gradients, to 1e-13 of |s|."""
    face = [0.5 * (a + _at(a, (x, 1))) for x in range(3)]
    root = torch.rsqrt(sum(f + _at(f, (x, -1)) for x, f in enumerate(face)) / 6.0)

    def apply(v):  # minus the operator
        out = torch.zeros_like(v)
        for x in range(3):
            flux = face[x] * (_at(v, (x, 1)) - v)
            out -= flux - _at(flux, (x, -1))
        return out

    def precondition(r):
        z = torch.fft.irfftn(torch.fft.rfftn(root * r) * inv, s=a.shape) * root
        return z - z.mean()

    r = -s - apply(u)
    z = precondition(r)
    p, rz, stop = z, (r * z).sum(), 1e-13 * torch.linalg.vector_norm(s)
    for it in range(800):
        ap = apply(p)
        alpha = rz / (p * ap).sum()
        u = u + alpha * p
        r = r - alpha * ap
        if it % 16 == 15 and bool(torch.linalg.vector_norm(r) <= stop):
            break
        z = precondition(r)
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return u


def _literal_change(e, m, v):
    """d_mu(m (e^-1)^{mu nu} d_nu v) in flux form."""
    adj = {(0, 0): e[1, 1] * e[2, 2] - e[1, 2] ** 2, (1, 1): e[0, 0] * e[2, 2] - e[0, 2] ** 2,
           (2, 2): e[0, 0] * e[1, 1] - e[0, 1] ** 2, (0, 1): e[0, 2] * e[1, 2] - e[0, 1] * e[2, 2],
           (0, 2): e[0, 1] * e[1, 2] - e[0, 2] * e[1, 1], (1, 2): e[0, 1] * e[0, 2] - e[0, 0] * e[1, 2]}
    scale = m / _det(e)
    out = torch.zeros_like(m)
    for a in range(3):
        k = adj[a, a] * scale
        flux = 0.5 * (k + _at(k, (a, 1))) * (_at(v, (a, 1)) - v)
        out += flux - _at(flux, (a, -1))
        for b in range(3):
            if b != a:
                g = adj[min(a, b), max(a, b)] * scale * (_at(v, (b, 1)) - _at(v, (b, -1)))
                out += 0.25 * (_at(g, (a, 1)) - _at(g, (a, -1)))
    return out


def _solve(rho, steps, update):
    """The moving-mesh iteration at its default parameters."""
    shape = rho.shape
    xi_m, v_m, a_min, floor, d_max = 0.1, 10.0, 0.01, 0.01, 0.5
    node = torch.stack(torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float64) for n in shape],
                                      indexing="ij"), -1).reshape(-1, 3)
    w = (rho / rho.mean()).reshape(-1)
    off = torch.zeros_like(node)
    phi = torch.zeros(shape, device="cuda", dtype=torch.float64)
    m, u, inv, alphas = w.reshape(shape), torch.zeros_like(phi), _laplacian_inverse(shape), []
    for _ in range(steps):
        if not update:
            m = _cic(shape, node + off, w)
        e = _hessian(phi)
        for a in range(3):
            e[a, a] = e[a, a] + 1.0
        lam = _min_eig(e)
        sigma = 1.0 - m
        t = sigma + 4.0 * (xi_m / lam.clamp_min(1e-12) - 1.0).clamp_min(0.0) ** 2
        t = t - 2.0 * torch.where(_det(e) > v_m, sigma.abs(), torch.zeros_like(m))
        s = _smooth(t) - t.mean()
        if float(torch.sqrt((s * s).mean())) <= 1e-3:
            break
        u = _elliptic(m.clamp_min(a_min), s, u, inv)
        d = _smooth(u)
        grad = [0.5 * (_at(d, (a, 1)) - _at(d, (a, -1))) for a in range(3)]
        most, h, alpha = max(float(g.abs().max()) for g in grad), _hessian(d), 1.0
        while alpha >= 2.0 ** -20:
            c = {k: e[k] + alpha * h[k] - (floor if k[0] == k[1] else 0.0) for k in e}
            good = (c[0, 0] > 0) & (c[0, 0] * c[1, 1] - c[0, 1] ** 2 > 0) & (_det(c) > 0)
            if bool(good.all()) and alpha * most <= d_max:
                break
            alpha *= 0.5
        if alpha < 2.0 ** -20:
            break
        alphas.append(alpha)
        if update:
            m = m + alpha * _literal_change(e, m, d)
        else:
            det = _det(e)
            adj = {(0, 0): e[1, 1] * e[2, 2] - e[1, 2] ** 2, (1, 1): e[0, 0] * e[2, 2] - e[0, 2] ** 2,
                   (2, 2): e[0, 0] * e[1, 1] - e[0, 1] ** 2, (0, 1): e[0, 2] * e[1, 2] - e[0, 1] * e[2, 2],
                   (0, 2): e[0, 1] * e[1, 2] - e[0, 2] * e[1, 1], (1, 2): e[0, 1] * e[0, 2] - e[0, 0] * e[1, 2]}
            x = node + off
            off = off - alpha * torch.stack(
                [_gather(sum(adj[min(a, b), max(a, b)] * grad[b] for b in range(3)) / det, x) for a in range(3)], -1)
        phi = phi + alpha * (d - d.mean())
    lap = sum(_at(phi, (a, 1)) - 2.0 * phi + _at(phi, (a, -1)) for a in range(3))
    return phi, -lap, np.array(alphas + [0.0] * (steps - len(alphas)))


def exact(case, seed):
    kind = case["kind"]
    if kind == "deposit":
        n = case["n"]
        pos, mass = _clustered(n, case["cell"], case["np"], case["mass"], seed)
        return {"density": _cic((n, n, n), pos / case["cell"], torch.ones_like(pos[:, 0]) if mass is None else mass)}
    if kind == "slab":
        shape = (case["n0"], case["n1"], case["n2"])
        phi, delta_r, alpha = _solve(_lognormal(shape, seed), case["steps"], 0)
        return {"phi": phi, "delta_r": delta_r, "alpha": alpha}
    if kind == "batch":
        outs = []
        for n, i in _mocks(case):
            if n > 64:  # the larger ones take too long
                outs.append({"phi": None, "delta_r": None, "alpha": None})
                continue
            x = _particles(n, 3.125, 1, seed + _STRIDE * (i + 1)) / 3.125
            phi, delta_r, alpha = _solve(_cic((n, n, n), x, torch.ones_like(x[:, 0])), case["steps"], 0)
            outs.append({"phi": phi * 3.125 ** 2, "delta_r": delta_r, "alpha": alpha})
        return outs
    n, cell = case["n"], case["cell"]
    if n > 128:  # a solve of these sizes takes too long here
        return None
    x = _particles(n, cell, case.get("order", 1), seed) / cell
    phi, delta_r, alpha = _solve(_cic((n, n, n), x, torch.ones_like(x[:, 0])), case["steps"], case.get("update", 0))
    if kind == "adjoint":  # the gradient has no short plain form
        return {"delta_r": delta_r, "grad_rho": None}
    return {"phi": phi * cell * cell, "delta_r": delta_r, "alpha": alpha}
