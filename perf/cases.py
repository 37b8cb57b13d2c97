"""The workloads the library is timed on, and what they give in 64 bits.

Each case is one pass of a job a user runs through the public entry points: stepping a run
from a snapshot, drawing initial conditions, an ensemble of small runs, the spectra of a mesh,
the halo-proxy bias, the relativistic displacement combination, a gradient through a run, and
the stateless particle operators.  ``listed`` names fixed sizes, ``draw`` others of the same
ranges; ``prepare`` makes the inputs and the handle a program keeps, ``run`` is one pass,
``exact`` the same result from plain FP64 torch.

The estimators of an FP32 context return their numbers in double arrays; they are kept here in
the precision of the field they were measured on (``_as_field``).  Counts are kept as integers.
"""
import functools
import math

import numpy as np
import torch
import torch.utils.checkpoint

import paper_2404_02783_gb300 as pm

DEV = "cuda"
OMEGA_M, OMEGA_B, HUBBLE, N_S, SIGMA8, T_CMB = 0.31, 0.049, 0.67, 0.965, 0.81, 2.7255
C_LIGHT = 2997.92458  # speed of light in units of 100 km/s
BATCH_BOXES = (1000.0, 2000.0, 4000.0)  # the boxes an ensemble cycles through [Mpc/h]


# ------------------------------------------------------------------ the cases
def _run(name, n_part, n_mesh, box, z0, grid, start, steps, mode="newton", gradient="spectral", precision="fp32",
         stepping="integrals"):
    return dict(name=name, kind="run", np=n_part, nmesh=n_mesh, box=box, a0=1.0 / (1.0 + z0), grid=grid, start=start,
                steps=steps, mode=mode, gradient=gradient, precision=precision, stepping=stepping)


def listed():
    return [
        # a quick-look run on a small mesh: launches and latency decide
        _run("run_64_small", 64, 64, 625.0, 50.0, 100, 40, 20),
        # the large simulation: a span of its later steps, resumed from a snapshot
        _run("run_512", 512, 512, 5000.0, 50.0, 100, 60, 5),
        # the relativistic run of the horizon-scale pair: Poisson gauge, mesh finer than the lattice
        _run("run_128_on_256_gr", 128, 256, 4000.0, 100.0, 100, 0, 10, mode="gr"),
        # the paper's own first-order gradient, growth-matched steps
        _run("run_256_fd1", 256, 256, 2500.0, 50.0, 50, 10, 8, gradient="fd1", stepping="growth"),
        # a reference run in double precision
        _run("run_256_fp64", 256, 256, 2000.0, 50.0, 20, 8, 2, precision="fp64"),
        # initial conditions of the large simulation
        dict(name="ic_512", kind="ic", np=512, nmesh=512, box=5000.0, a0=1.0 / 51.0, lpt=1, paired=False, fixed=False),
        # an ensemble of realisations with three box sizes: initial conditions, steps, every P(k)
        dict(name="ensemble_64x64", kind="batch", np=64, nmesh=128, count=64, a0=1.0 / 51.0, grid=50, steps=10,
             mode="newton", bins=24),
        # one snapshot's P(k) and B(k)
        dict(name="spectra_512", kind="spectra", nmesh=512, box=5000.0, bins=64, bk_bins=24, m=128),
        # halo proxy and linear-bias fit of a snapshot
        dict(name="bias_256", kind="bias", nmesh=256, box=2000.0, fraction=0.05, bins=32, terms=2),
        # the relativistic displacement of a 256^3 pair added to a 512^3 run
        dict(name="combine_256_to_512", kind="combine", np=256, ratio=2, box=4000.0),
        # a field-level fit: the gradient of a loss through a whole run
        dict(name="gradient_128", kind="gradient", np=128, nmesh=128, box=2000.0, a0=1.0 / 51.0, steps=50, every=10,
             mode="newton", gradient="spectral"),
        # particle operators on a ragged particle list (halos, a light cone, a cut-out)
        dict(name="points_ragged", kind="points", nmesh=128, points=3000017, precision="fp32"),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def draw(rng):
    kind = rng.choice(("run", "run", "run", "ic", "batch", "spectra", "bias", "combine", "gradient", "points"))
    cell = math.exp(rng.uniform(math.log(6.0), math.log(30.0)))  # Mpc/h
    z0 = rng.uniform(30.0, 100.0)
    if kind == "run":
        fp64 = rng.random() < 0.25
        gr = rng.random() < 0.35
        n = _pow2(rng, 5, 7 if fp64 else 9)
        ratio = rng.choice((1, 1, 2, 4)) if n >= 64 else 1
        steps = rng.randint(1, 3 if n == 512 else 8 if n == 256 else 20)
        grid = rng.randint(40, 120)
        c = _run("", n // ratio, n, round(cell * n, 1), z0, grid, 0 if gr else rng.randint(0, grid // 2), steps,
                 mode="gr" if gr else "newton", gradient="fd1" if rng.random() < 0.3 else "spectral",
                 precision="fp64" if fp64 else "fp32", stepping="growth" if rng.random() < 0.3 else "integrals")
        del c["name"]
        return c
    if kind == "ic":
        n = _pow2(rng, 5, 9)
        return dict(kind=kind, np=n, nmesh=n, box=round(cell * n, 1), a0=1.0 / (1.0 + z0),
                    lpt=2 if n < 512 and rng.random() < 0.5 else 1, paired=rng.random() < 0.5, fixed=rng.random() < 0.5)
    if kind == "batch":
        n = _pow2(rng, 5, 6)
        return dict(kind=kind, np=n, nmesh=2 * n if n == 32 else rng.choice((n, 2 * n)), count=rng.randint(2, 60),
                    a0=1.0 / (1.0 + z0), grid=rng.randint(30, 60), steps=rng.randint(2, 10),
                    mode=rng.choice(("newton", "newton", "gr")), bins=rng.randint(8, 40))
    if kind == "spectra":
        n = _pow2(rng, 6, 9)
        m = min(_pow2(rng, 6, 7), 2 * n)
        return dict(kind=kind, nmesh=n, box=round(cell * n, 1), bins=rng.randint(9, 128),
                    bk_bins=rng.randint(5, min((m - 1) // 3, n // 2 - 1, 29) - 1), m=m)
    if kind == "bias":
        n = _pow2(rng, 6, 8)
        return dict(kind=kind, nmesh=n, box=round(cell * n, 1), fraction=round(rng.uniform(0.01, 0.2), 4),
                    bins=rng.randint(12, 40), terms=rng.randint(1, 3))
    if kind == "combine":
        return dict(kind=kind, np=_pow2(rng, 5, 7), ratio=rng.choice((1, 2, 4)), box=round(1000 * rng.uniform(1, 8), 1))
    if kind == "gradient":
        n = _pow2(rng, 5, 7)
        ratio = rng.choice((1, 1, 2)) if n < 128 else 1
        return dict(kind=kind, np=n, nmesh=n * ratio, box=round(cell * n * ratio, 1), a0=1.0 / (1.0 + z0),
                    steps=rng.randint(5, 40), every=rng.randint(2, 10), mode=rng.choice(("newton", "newton", "gr")),
                    gradient=rng.choice(("spectral", "spectral", "fd1")))
    return dict(kind="points", nmesh=_pow2(rng, 5, 8), points=int(math.exp(rng.uniform(math.log(1e3), math.log(5e6)))),
                precision=rng.choice(("fp32", "fp32", "fp64")))


# ------------------------------------------------------------------ cosmology in 64 bits
_GL = np.polynomial.legendre.leggauss(20)


def _integral(f, lo, hi, panels=64):
    e = np.linspace(lo, hi, panels + 1)
    h = 0.5 * np.diff(e)
    x = (0.5 * (e[1:] + e[:-1]))[:, None] + h[:, None] * _GL[0]
    return float(np.sum(h[:, None] * _GL[1] * f(x)))


def _E(a):
    return np.sqrt(OMEGA_M / a**3 + 1.0 - OMEGA_M)


def _omega_m_a(a):
    return OMEGA_M / a**3 / _E(a)**2


def _growth_integral(a):
    # int_0^a da / (a E)^3 with a = s^2
    return _integral(lambda s: 2.0 * s**4 / (OMEGA_M + (1.0 - OMEGA_M) * s**6)**1.5, 0.0, math.sqrt(a))


def _D(a):
    return float(_E(a) * _growth_integral(a) / (_E(1.0) * _growth_integral(1.0)))


def _f(a):
    return float(-1.5 * _omega_m_a(a) + 1.0 / (a * a * _E(a)**3 * _growth_integral(a)))


def _growth_p(a):
    return float(a * a * _E(a) * _f(a) * _D(a))


def _transfer(k):
    """Eisenstein & Hu (1998), the no-wiggle fit (their Eqs. 26 and 28-31); k in h/Mpc."""
    omh2, obh2, fb = OMEGA_M * HUBBLE**2, OMEGA_B * HUBBLE**2, OMEGA_B / OMEGA_M
    s = 44.5 * math.log(9.83 / omh2) / math.sqrt(1.0 + 10.0 * obh2**0.75)
    alpha = 1.0 - 0.328 * math.log(431.0 * omh2) * fb + 0.38 * math.log(22.3 * omh2) * fb * fb
    gamma = OMEGA_M * HUBBLE * (alpha + (1.0 - alpha) / (1.0 + (0.43 * k * HUBBLE * s)**4))
    q = k * (T_CMB / 2.7)**2 / gamma
    L0 = np.log(2.0 * math.e + 1.8 * q)
    return L0 / (L0 + (14.2 + 731.0 / (1.0 + 62.5 * q)) * q * q)


@functools.lru_cache(maxsize=None)
def _amplitude():
    def f(lnk):
        k = np.exp(lnk)
        x = 8.0 * k
        xs = np.maximum(x, 1e-3)
        w = np.where(x < 1e-3, 1.0 - x * x / 10.0, 3.0 * (np.sin(xs) - xs * np.cos(xs)) / xs**3)
        return k**(3.0 + N_S) * (_transfer(k) * w)**2 / (2.0 * math.pi**2)
    return SIGMA8**2 / _integral(f, math.log(1e-7), math.log(1e3), 20000)


def _power(k):
    return _amplitude() * k**N_S * _transfer(k)**2


class _Steps:
    """Kick and drift factors of the uniform a-grid, and the Poisson-gauge scalars."""

    def __init__(self, a0, a1, grid, stepping):
        self.a = [a0 + ((a1 - a0) * i) / grid for i in range(grid + 1)]
        self.growth = stepping == "growth"

    def half(self, s):
        return 0.5 * (self.a[s] + self.a[s + 1])

    def _kick(self, lo, hi, at):
        if self.growth:
            return (_growth_p(hi) - _growth_p(lo)) / (1.5 * OMEGA_M * _D(at))
        return _integral(lambda a: 1.0 / (a * a * _E(a)), lo, hi)

    def kick(self, s):
        return self._kick(self.a[0] if s == 0 else self.half(s - 1), self.half(s), self.a[s])

    def close(self):
        return self._kick(self.half(len(self.a) - 2), self.a[-1], self.a[-1])

    def drift(self, s):
        lo, hi = self.a[s], self.a[s + 1]
        if self.growth:
            return (_D(hi) - _D(lo)) / _growth_p(self.half(s))
        return _integral(lambda a: 1.0 / (a**3 * _E(a)), lo, hi)


# ------------------------------------------------------------------ meshes and modes
def _modes(n):
    """Signed integer wavenumbers of the half grid (x, y, z), as broadcastable int64 tensors."""
    f = torch.arange(n, device=DEV)
    f = torch.where(f < n // 2, f, f - n)
    return f[:, None, None], f[None, :, None], torch.arange(n // 2 + 1, device=DEV)[None, None, :]


def _n2(n):
    nx, ny, nz = _modes(n)
    return nx * nx + ny * ny + nz * nz


def _not_nyquist(n):
    nx, ny, nz = _modes(n)
    return (nx != -(n // 2)) & (ny != -(n // 2)) & (nz != n // 2)


def _table(n, fn):
    """fn of |n|^2 > 0 on every half-grid mode, 0 on the zero mode (FP64)."""
    v = np.zeros(3 * (n // 2)**2 + 1)
    v[1:] = fn(np.arange(1, len(v), dtype=np.float64))
    return torch.from_numpy(v).to(DEV)[_n2(n)]


def _linear(g, n, box):
    """delta_k (unnormalised transform) of the linear field at a = 1 with unit phases g."""
    kf = 2.0 * math.pi / box
    amp = _table(n, lambda s: n**3 * np.sqrt(_power(kf * np.sqrt(s)) / box**3)).to(g.real.dtype)
    return torch.where(_not_nyquist(n), g * amp, torch.zeros((), dtype=g.dtype, device=DEV))


def _k_axes(n, box):
    """k_j of the three axes, 0 at the Nyquist index."""
    kf = 2.0 * math.pi / box
    return [kf * torch.where(m.abs() == n // 2, torch.zeros_like(m), m).to(torch.float64) for m in _modes(n)]


def _gradient(phi_k, n, box):
    """IFFT[i k_j phi_k] for the three axes."""
    for k in _k_axes(n, box):
        yield torch.fft.irfftn(1j * k.to(phi_k.real.dtype) * phi_k, s=(n, n, n))


def _displacement(delta_k, n, box):
    """First-order displacement Psi of a linear field, three n^3 meshes."""
    inv = _table(n, lambda s: 1.0 / s).to(delta_k.real.dtype) / (2.0 * math.pi / box)**2
    return [p.reshape(-1) for p in _gradient(delta_k * inv, n, box)]


def _white(n, gen, dtype=torch.float32):
    return torch.randn((n, n, n), generator=gen, device=DEV, dtype=dtype)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _lattice(n, axis):
    """Lattice index along an axis of every particle id."""
    i = torch.arange(n**3, device=DEV)
    return (i // n**(2 - axis)) % n


def _particles(n, box, a, a_mom, gen, fp64):
    """A snapshot at scale factor a: lattice particles displaced by a linear field's Zel'dovich
    displacement, momenta of a_mom; ticks (int32) or box fractions, and momenta."""
    psi = _displacement(_linear(torch.fft.rfftn(_white(n, gen)) / n**1.5, n, box), n, box)
    x = torch.empty((3, n**3), dtype=torch.float64 if fp64 else torch.int32, device=DEV)
    p = torch.empty((3, n**3), dtype=torch.float64 if fp64 else torch.float32, device=DEV)
    D, P = _D(a), _growth_p(a_mom)
    for j in range(3):
        d = psi[j].to(torch.float64) * D
        q = _lattice(n, j)
        if fp64:
            v = q.to(torch.float64) / n + d / box
            x[j] = v - torch.floor(v)
        else:
            x[j] = (q * (2**32 // n) + torch.round(d * (2.0**32 / box)).to(torch.int64)).to(torch.int32)
        p[j] = psi[j].to(p.dtype) * P
    return x, p


def _contrast(n, box, gen):
    """A log-normal density contrast mesh with the linear spectrum (FP32)."""
    g = torch.fft.irfftn(_linear(torch.fft.rfftn(_white(n, gen)) / n**1.5, n, box), s=(n, n, n))
    return torch.exp(g - 0.5 * g.var()) - 1.0


def _fractions(x):
    """Box fractions in FP64 of ticks or fractions."""
    return x if x.dtype == torch.float64 else (x.to(torch.int64) & 0xFFFFFFFF).to(torch.float64) * 2.0**-32


# ------------------------------------------------------------------ the particle-mesh step in 64 bits
def _corners(x, n):
    """(linear cell, weight, signs) of the eight cloud-in-cell corners of fractions x [3][count]."""
    s = [v * n - 0.5 for v in x]
    base = [torch.floor(v.detach()) for v in s]
    w1 = [v - b for v, b in zip(s, base)]
    b = [v.to(torch.int64) % n for v in base]
    for c in range(8):
        d = (c >> 2, (c >> 1) & 1, c & 1)
        ix, iy, iz = ((b[j] + d[j]) % n for j in range(3))
        w = [w1[j] if d[j] else 1.0 - w1[j] for j in range(3)]
        yield (ix * n + iy) * n + iz, w, d


def _deposit(x, n, mass):
    rho = torch.zeros(n**3, dtype=torch.float64, device=DEV)
    for idx, w, _ in _corners(x, n):
        rho = rho.index_add(0, idx, mass * w[0] * w[1] * w[2])
    return rho.reshape(n, n, n)


def _gather(fields, x, n):
    out = [0.0] * len(fields)
    for idx, w, _ in _corners(x, n):
        ww = w[0] * w[1] * w[2]
        out = [o + ww * f.reshape(-1)[idx] for o, f in zip(out, fields)]
    return out


def _gather_gradient(phi, x, n, box):
    out, flat = [0.0, 0.0, 0.0], phi.reshape(-1)
    for idx, w, d in _corners(x, n):
        v = flat[idx] * (n / box)
        for j in range(3):
            k, l = (j + 1) % 3, (j + 2) % 3
            out[j] = out[j] + (v if d[j] else -v) * w[k] * w[l]
    return out


def _force(x, c, a, history):
    """-grad phi at the particles; `history` is (Phi_k, a) of the evaluation before, and the new one."""
    n, box = c["nmesh"], c["box"]
    dk = torch.fft.rfftn(_deposit(x, n, (n / c["np"])**3) - 1.0)
    k2 = _table(n, lambda s: s) * (2.0 * math.pi / box)**2
    if c["mode"] == "newton":
        phi = -1.5 * OMEGA_M * dk / torch.where(k2 > 0, k2, torch.inf)
    else:
        H, om = a * float(_E(a)) / C_LIGHT, float(_omega_m_a(a))
        src, den = -1.5 * H * H * om * dk, k2 + 3.0 * H * H + 4.5 * H * H * om
        if history is not None:
            lag = 3.0 * H / (C_LIGHT * _integral(lambda b: 1.0 / (b * b * _E(b)), history[1], a))
            src, den = src + lag * history[0], den + lag
        Phi = torch.where(k2 > 0, src / den, torch.zeros_like(src))
        history = (Phi, a)
        phi = a * C_LIGHT**2 * Phi
    if c["gradient"] == "fd1":
        g = _gather_gradient(torch.fft.irfftn(phi, s=(n, n, n)), x, n, box)
    else:
        g = _gather(list(_gradient(phi, n, box)), x, n)
    return [-v for v in g], history


def _evolve(x, p, c, grid, start, steps, stepping="integrals", checkpoint=False):
    """`steps` kick-drift-kick steps of fractions x and momenta p (lists of three FP64 tensors)."""
    t = _Steps(c["a0"], 1.0, grid, stepping)
    history = None

    def one(a, kick, drift, history, *xp):
        x, p = list(xp[:3]), list(xp[3:])
        g, history = _force(x, c, a, history)
        p = [u + kick * v for u, v in zip(p, g)]
        x = [u + (drift / c["box"]) * v for u, v in zip(x, p)]
        x = [u - torch.floor(u.detach()) for u in x]
        return (history, *x, *p)

    for s in range(start, start + steps):
        args = (t.a[s], t.kick(s), t.drift(s), history, *x, *p)
        got = torch.utils.checkpoint.checkpoint(one, *args, use_reentrant=False) if checkpoint else one(*args)
        history, x, p = got[0], list(got[1:4]), list(got[4:])
    if start + steps == grid:
        g, history = _force(x, c, 1.0, history)
        p = [u + t.close() * v for u, v in zip(p, g)]
    return x, p


def _from_lattice(x, n, box):
    """Displacements from the lattice nodes, minimum image, Mpc/h."""
    d = [x[j] - _lattice(n, j).to(torch.float64) / n for j in range(3)]
    return torch.stack([(v - torch.round(v.detach())) * box for v in d])


# ------------------------------------------------------------------ initial conditions in 64 bits
def _philox(counter, seed):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words: words 0 and 1."""
    mask = 0xFFFFFFFF
    c = [v & mask for v in counter]
    k = [seed & mask, (seed >> 32) & mask]
    for r in range(10):
        if r:
            k = [(k[0] + 0x9E3779B9) & mask, (k[1] + 0xBB67AE85) & mask]
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # low 64 bits
        c = [((p1 >> 32) & mask) ^ c[1] ^ k[0], p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k[1], p0 & mask]
    return c[0], c[1]


def _phases(n, seed):
    """Unit complex Gaussian per wavevector of the half grid, Hermitian on its kz = 0 plane."""
    nx, ny, nz = torch.broadcast_tensors(*_modes(n))
    canonical = (nz > 0) | (ny > 0) | ((ny == 0) & (nx > 0))
    sign = torch.where(canonical, 1, -1)
    r0, r1 = _philox([sign * nx, sign * ny, nz, torch.zeros_like(nz)], int(seed))
    amp = torch.sqrt(-torch.log((r0.to(torch.float64) + 0.5) * 2.0**-32))
    g = torch.polar(amp, (2.0 * math.pi * 2.0**-32) * (r1.to(torch.float64) + 0.5) * sign)
    g[0, 0, 0] = 0.0
    return torch.where(_not_nyquist(n), g, torch.zeros((), dtype=g.dtype, device=DEV))


def _initial(n, box, a, g, lpt=1):
    """Displacements (Mpc/h) and momenta at a of phases g (three FP64 tensors each)."""
    psi = _displacement(_linear(g, n, box), n, box)
    x, p = [_D(a) * v for v in psi], [_growth_p(a) * v for v in psi]
    if lpt == 2:
        d = [[v.reshape(-1) for v in _gradient(torch.fft.rfftn(u.reshape(n, n, n)) * _not_nyquist(n), n, box)] for u in psi]
        src = sum(d[i][i] * d[j][j] - d[i][j]**2 for i, j in ((0, 1), (0, 2), (1, 2)))
        k2 = _table(n, lambda s: s) * (2.0 * math.pi / box)**2
        phi2 = -torch.fft.rfftn(src.reshape(n, n, n)) / torch.where(k2 > 0, k2, torch.inf) * _not_nyquist(n)
        om = float(_omega_m_a(a))
        D2 = -3.0 / 7.0 * _D(a)**2 * om**(-1.0 / 143.0)
        f2 = 2.0 * om**(6.0 / 11.0)
        for j, v in enumerate(_gradient(phi2, n, box)):
            x[j] = x[j] + D2 * v.reshape(-1)
            p[j] = p[j] + a * a * float(_E(a)) * f2 * D2 * v.reshape(-1)
    return x, p


def _place(d, n, box):
    """Box fractions of displaced lattice particles."""
    x = [_lattice(n, j).to(torch.float64) / n + d[j] / box for j in range(3)]
    return [v - torch.floor(v.detach()) for v in x]


# ------------------------------------------------------------------ estimators in 64 bits
def _bin_of(n2, edges):
    e2 = torch.from_numpy(np.asarray(edges, dtype=np.float64)**2).to(DEV)
    v = n2.to(torch.float64)
    b = torch.searchsorted(e2, v, right=True) - 1
    b = torch.where(v == e2[-1], len(edges) - 2, b)
    return torch.where((b >= 0) & (b < len(edges) - 1), b, -1)


def _window(n):
    w = [torch.sinc(m.to(torch.float64) / n)**2 for m in _modes(n)]
    return w[0] * w[1] * w[2]


def _spectrum(f1, f2, box, edges):
    """(k, P, modes) of two meshes' cross spectrum, the cloud-in-cell window divided out."""
    n, nb = f1.shape[0], len(edges) - 1
    d1, d2 = (torch.fft.rfftn(f.to(torch.float64)) / _window(n) for f in (f1, f2))
    n2 = _n2(n)
    b = torch.where((n2 > 0) & (n2 <= (n // 2)**2), _bin_of(n2, edges), -1).reshape(-1)
    w = torch.full((n, n, n // 2 + 1), 2.0, dtype=torch.float64, device=DEV)
    w[:, :, 0] = w[:, :, -1] = 1.0
    w, sel = w.reshape(-1), b >= 0
    sums = [torch.bincount(b[sel], weights=(w * v.reshape(-1))[sel], minlength=nb)
            for v in (torch.ones_like(w), (d1 * d2.conj()).real, torch.sqrt(n2.to(torch.float64)))]
    return 2.0 * math.pi / box * sums[2] / sums[0], box**3 / float(n)**6 * sums[1] / sums[0], sums[0]


def _triangles(field, box, edges, m):
    """(B, counts) of every triangle of bins i <= j <= l by sums over the m^3 grid."""
    n, nb = field.shape[0], len(edges) - 1
    nx, ny, nz = _modes(m)
    h = n // 2
    n2 = _n2(m)
    b = torch.where((n2 > 0) & (n2 <= h * h) & (nx.abs() < h) & (ny.abs() < h) & (nz < h), _bin_of(n2, edges), -1)
    dk = torch.fft.rfftn(field.to(torch.float64)) / _window(n)
    part = dk[(nx % n), (ny % n), nz.clamp(max=h)]
    T, zero = [], torch.zeros((), dtype=part.dtype, device=DEV)
    for q in range(nb):
        T.append([torch.fft.irfftn(torch.where(b == q, v, zero), s=(m, m, m)).reshape(-1) * m**3
                  for v in (part, torch.ones_like(part))])
    sums = []
    for f in (torch.stack([t[0] for t in T]), torch.stack([t[1] for t in T])):
        rows = []
        for i in range(nb):
            s = (f[i] * f[i:]) @ f[i:].T
            rows += [s[j, j:] for j in range(nb - i)]
        sums.append(torch.cat(rows) / float(m)**3)
    cnt = torch.round(sums[1])
    B = box**6 / float(n)**9 * sums[0] / cnt
    return torch.where(cnt > 0, B, torch.nan), cnt


def _log_edges(nbins, n):
    return pm.log_edges(nbins, 1.0, n / 2.0)


def _bk_edges(c):
    return 0.5 + np.arange(c["bk_bins"] + 1.0)


def _k_max(c):
    return 0.4 * c["nmesh"] / 2.0 * 2.0 * math.pi / c["box"]


# ------------------------------------------------------------------ prepare, run
def _config(c, grid=10):
    return pm.make_config(c.get("np", c["nmesh"]), c["nmesh"], c["box"], c.get("a0", 0.02), 1.0, c.get("grid", grid),
                          mode=pm.PM_GR_POISSON if c.get("mode") == "gr" else pm.PM_NEWTON,
                          precision=pm.PM_FP64 if c.get("precision") == "fp64" else pm.PM_FP32_FIXED,
                          n_lo=pm.DEFAULT_N_LO if c.get("mode") == "gr" else 0,
                          gradient=pm.PM_GRAD_FD1 if c.get("gradient") == "fd1" else pm.PM_GRAD_SPECTRAL,
                          stepping=pm.PM_STEP_GROWTH if c.get("stepping") == "growth" else pm.PM_STEP_INTEGRALS)


def _snapshot(c, seed):
    t = _Steps(c["a0"], 1.0, c["grid"], c["stepping"])
    s = c["start"]
    return _particles(c["np"], c["box"], t.a[s], t.half(s - 1) if s else t.a[0], _gen(seed), c["precision"] == "fp64")


def _boxes(c):
    return [BATCH_BOXES[r % 3] for r in range(c["count"])]


def _seeds(c, seed):
    return [1000003 * (int(seed) + 1) + r for r in range(c["count"])]


def _fit_inputs(c, seed):
    """White noise of the current point of a fit, and the density it is compared with."""
    gen = _gen(seed)
    w = _white(c["np"], gen)
    return w, 0.5 * _contrast(c["nmesh"], c["box"], gen)


def _pair(c, seed):
    """Positions of the target run and of the relativistic and Newtonian runs of a pair (ticks)."""
    gen = _gen(seed)
    nt, nc, box = c["np"] * c["ratio"], c["np"], c["box"]
    target = _particles(nt, box, 1.0, 1.0, gen, False)
    newton = _particles(nc, box, 1.0, 1.0, gen, False)
    xi = torch.round(torch.randn((3, nc**3), generator=gen, device=DEV) * (0.7 * 2.0**32 / box)).to(torch.int32)
    return target, (newton[0] + xi, newton[1]), newton


def _points(c, seed):
    """A clustered particle list (two thirds in blobs, the rest uniform) and a smooth mesh to interpolate."""
    gen = _gen(seed)
    count, n, dt = c["points"], c["nmesh"], torch.float64
    x = torch.rand((3, count), generator=gen, device=DEV, dtype=dt)
    blobs = torch.rand((3, max(8, count // 300)), generator=gen, device=DEV, dtype=dt)
    which = torch.randint(0, blobs.shape[1], (count,), generator=gen, device=DEV)
    near = blobs[:, which] + torch.randn((3, count), generator=gen, device=DEV, dtype=dt) * (1.5 / n)
    x = torch.where(torch.arange(count, device=DEV) % 3 == 0, x, near)
    x = x - torch.floor(x)
    if c["precision"] == "fp64":
        return torch.where(x < 1.0, x, torch.zeros_like(x)), _white(n, gen, dt)
    return torch.floor(x * 2.0**32).to(torch.int64).to(torch.int32), _white(n, gen)


def _scratch(nbytes):
    buf = torch.empty(nbytes + 256, dtype=torch.uint8, device=DEV)
    off = (-buf.data_ptr()) % 256
    return buf[off:off + nbytes]


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind == "run":
        s["x"], s["p"] = _snapshot(c, seed)
        s["run"] = pm.PMRun(_config(c))
        pm.pm_autotune_fft(s["run"].ctx)
    elif kind == "ic":
        s["run"], s["seed"] = pm.PMRun(_config(c)), int(seed) + 1
    elif kind == "batch":
        s["batch"], s["seeds"] = pm.PMBatch(_config(dict(c, box=BATCH_BOXES[0])), boxes=_boxes(c)), _seeds(c, seed)
        s["batch"].autotune()
    elif kind == "spectra":
        s["field"], s["run"] = _contrast(c["nmesh"], c["box"], _gen(seed)), pm.PMRun(_config(c))
    elif kind == "bias":
        s["field"], s["run"] = _contrast(c["nmesh"], c["box"], _gen(seed)), pm.PMRun(_config(c))
    elif kind == "combine":
        data = _pair(c, seed)
        s["runs"] = [pm.PMRun(_config(dict(box=c["box"], np=n, nmesh=n))) for n in (c["np"] * c["ratio"], c["np"], c["np"])]
        for r, (x, p) in zip(s["runs"], data):
            pm.pm_set_particles(r.ctx, x, p)
    elif kind == "gradient":
        s["w"], s["target"] = _fit_inputs(c, seed)
        s["run"] = pm.PMRun(_config(c, c["steps"]))
        pm.pm_autotune_fft(s["run"].ctx)
    else:
        s["x"], s["field"] = _points(c, seed)
        s["scratch"] = _scratch(pm.pm_cell_sort_scratch_size(c["points"], c["nmesh"]))
    torch.cuda.synchronize()
    return s


def _as_field(a):
    """An estimator's numbers in the precision of the FP32 field they were measured on."""
    return np.asarray(a, dtype=np.float32)


def _whole(a):
    return np.rint(np.asarray(a)).astype(np.int64)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "run":
        r = state["run"]
        pm.pm_set_state(r.ctx, state["x"], state["p"], c["start"], c["start"] == 0)
        r.step(c["steps"])
        return {"displacement": r.displacement(), "momenta": r.particles()[1]}
    if kind == "ic":
        r = state["run"]
        r.ic(seed=state["seed"], paired=c["paired"], fixed=c["fixed"], lpt_order=c["lpt"])
        return {"displacement": r.displacement(), "momenta": r.particles()[1]}
    if kind == "batch":
        b = state["batch"]
        b.ic(state["seeds"])
        b.step(c["steps"])
        k, p, nm = b.power(_log_edges(c["bins"], c["nmesh"]))
        return {"momenta": torch.stack([b.particles(r)[1] for r in range(c["count"])]), "k": k, "P": _as_field(p),
                "modes": _whole(nm)}
    if kind == "spectra":
        r, f = state["run"], state["field"]
        k, p, nm = r.power(_log_edges(c["bins"], c["nmesh"]), field=f)
        B, nt = r.bispectrum(_bk_edges(c), c["m"], field=f)
        return {"k": k, "P": _as_field(p), "modes": _whole(nm), "B": _as_field(B), "triangles": _whole(nt)}
    if kind == "bias":
        r, f = state["run"], state["field"]
        h = torch.empty_like(f)
        chosen = pm.pm_halo_proxy(r.ctx, h, field=f, fraction=c["fraction"])
        coef, k, ratio, nm = pm.pm_linear_bias(r.ctx, h, f, _log_edges(c["bins"], c["nmesh"]), _k_max(c), c["terms"])
        return {"halos": h, "chosen": chosen, "fit": _as_field(coef), "ratio": _as_field(ratio), "modes": _whole(nm)}
    if kind == "combine":
        target, gr, newton = state["runs"]
        xi = torch.empty((3, target.count), dtype=torch.int32, device=DEV)
        pm.pm_displacement_correction(target.ctx, gr.ctx, newton.ctx, xi)
        return {"xi": xi, "displacement": target.displacement()}
    if kind == "gradient":
        loss, grad = state["run"].loss_grad(state["w"], state["target"], c["every"])
        return {"loss": _as_field(loss), "grad": grad}
    x, f, n, count = state["x"], state["field"], c["nmesh"], c["points"]
    prec = pm.PM_FP64 if c["precision"] == "fp64" else pm.PM_FP32_FIXED
    rho = torch.zeros_like(f)
    pm.pm_cic_deposit(x, count, prec, n, 1.0, rho)
    at = torch.empty(count, dtype=f.dtype, device=DEV)
    pm.pm_cic_interp(f, n, x, count, prec, at)
    keys, order = (torch.empty(count, dtype=torch.int32, device=DEV) for _ in range(2))
    pm.pm_cell_sort(x, count, prec, n, keys, order, state["scratch"])
    return {"density": rho, "interpolated": at, "keys": keys, "order": order}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "run":
        x, p = _snapshot(c, seed)
        x, p = _evolve(list(_fractions(x)), list(p.to(torch.float64)), c, c["grid"], c["start"], c["steps"], c["stepping"])
        return {"displacement": _from_lattice(x, c["np"], c["box"]), "momenta": torch.stack(p)}
    if kind == "ic":
        g = _phases(c["np"], int(seed) + 1)
        if c["fixed"]:
            g = torch.where(g != 0, g / g.abs(), g)
        d, p = _initial(c["np"], c["box"], c["a0"], -g if c["paired"] else g, c["lpt"])
        return {"displacement": torch.stack(d), "momenta": torch.stack(p)}
    if kind == "batch":
        out, edges = [], _log_edges(c["bins"], c["nmesh"])
        for box, sd in zip(_boxes(c), _seeds(c, seed)):
            cc = dict(c, box=box, gradient="spectral")
            d, p = _initial(c["np"], box, c["a0"], _phases(c["np"], sd))
            x, p = _evolve(_place(d, c["np"], box), p, cc, c["grid"], 0, c["steps"])
            rho = _deposit(x, c["nmesh"], (c["nmesh"] / c["np"])**3) - 1.0
            out.append((torch.stack(p), *_spectrum(rho, rho, box, edges)))
        p, k, P, nm = (torch.stack([o[i] for o in out]) for i in range(4))
        return {"momenta": p, "k": k, "P": P, "modes": None}
    if kind == "spectra":
        f = _contrast(c["nmesh"], c["box"], _gen(seed))
        k, p, _ = _spectrum(f, f, c["box"], _log_edges(c["bins"], c["nmesh"]))
        B, _ = _triangles(f, c["box"], _bk_edges(c), c["m"])
        return {"k": k, "P": p, "modes": None, "B": B, "triangles": None}
    if kind == "bias":
        f = _contrast(c["nmesh"], c["box"], _gen(seed))
        n3 = f.numel()
        chosen = math.ceil(c["fraction"] * n3)
        order = torch.sort(f.reshape(-1), descending=True, stable=True).indices[:chosen]
        h = torch.full((n3,), -1.0, dtype=torch.float64, device=DEV)
        h[order] = n3 / chosen - 1.0
        h = h.reshape(f.shape)
        edges = _log_edges(c["bins"], c["nmesh"])
        k, hm, nm = _spectrum(h, f, c["box"], edges)
        ratio = (hm / _spectrum(f, f, c["box"], edges)[1]).cpu().numpy()
        k, nm = k.cpu().numpy(), nm.cpu().numpy()
        a = c.get("a0", 0.02)
        H = a * float(_E(a)) / C_LIGHT
        use = (nm > 0) & (k < _k_max(c))
        A = np.stack([np.ones_like(k), H * H / k**2, k**2], axis=1)[use, :c["terms"]] * np.sqrt(nm[use])[:, None]
        fit = np.linalg.lstsq(A, ratio[use] * np.sqrt(nm[use]), rcond=None)[0]
        return {"halos": h, "chosen": None, "fit": fit, "ratio": ratio, "modes": None}
    if kind == "combine":
        (xt, _), (xg, _), (xn, _) = _pair(c, seed)
        nc, r = c["np"], c["ratio"]
        nt = nc * r
        xi = (xg - xn).to(torch.int64).reshape(3, nc, nc, nc)  # int32 difference: the minimum image
        it = torch.arange(nt, device=DEV)
        out = torch.empty((3, nt**3), dtype=torch.float64, device=DEV)
        for j in range(3):
            v = xi[j].to(torch.float64)
            for ax in range(3):
                lo, hi = v.index_select(ax, it // r), v.index_select(ax, (it // r + 1) % nc)
                w = (it % r).to(torch.float64).reshape([-1 if q == ax else 1 for q in range(3)]) / r
                v = lo * (1.0 - w) + hi * w
            moved = (xt[j].to(torch.int64) & 0xFFFFFFFF) + torch.round(v).to(torch.int64).reshape(-1) \
                - _lattice(nt, j) * (2**32 // nt)
            out[j] = moved.to(torch.int32).to(torch.float64) * (c["box"] / 2.0**32)
        return {"xi": None, "displacement": out}
    if kind == "gradient":
        w, target = _fit_inputs(c, seed)
        w = w.to(torch.float64).requires_grad_()
        g = torch.fft.rfftn(w) / float(c["np"])**1.5
        d, p = _initial(c["np"], c["box"], c["a0"], g)
        x, _ = _evolve(_place(d, c["np"], c["box"]), p, c, c["steps"], 0, c["steps"], checkpoint=True)
        rho = _deposit(x, c["nmesh"], (c["nmesh"] / c["np"])**3) - 1.0
        loss = ((rho - target.to(torch.float64))**2).mean()
        return {"loss": loss.detach(), "grad": torch.autograd.grad(loss, w)[0]}
    x, f = _points(c, seed)
    v = list(_fractions(x))
    at = _gather([f.to(torch.float64)], v, c["nmesh"])[0]
    return {"density": _deposit(v, c["nmesh"], 1.0), "interpolated": at, "keys": None, "order": None}


# ------------------------------------------------------------------ work
def _fft_flops(n):
    """Real-to-complex transform of an n^3 mesh."""
    return 2.5 * n**3 * 3 * math.log2(n)


def work(case):
    """Bytes and operations of one pass that the path cannot do without.  A step reads the positions
    and momenta, deposits, transforms, and writes both back with the force meshes gathered once:
    60 B a particle and 40 B a cell in FP32 (24 B a cell with the one-mesh first-order gradient; a
    Poisson-gauge step also reads and writes its potential history)."""
    c, kind = case, case["kind"]
    wide = 2 if c.get("precision") == "fp64" else 1
    n3, p3 = c["nmesh"]**3 if "nmesh" in c else 0, c.get("np", 0)**3
    transforms = 2 if c.get("gradient") == "fd1" else 4
    cell = (24 if c.get("gradient") == "fd1" else 40) + (8 if c.get("mode") == "gr" else 0)
    step = wide * (60 * p3 + cell * n3)
    flops = transforms * _fft_flops(c["nmesh"]) + 200 * p3 if n3 else 0.0
    if kind == "run":
        evals = c["steps"] + (1 if c["start"] + c["steps"] == c["grid"] else 0)
        return {"bytes": evals * step + wide * 72 * p3, "flops": evals * flops}
    if kind == "ic":
        chains = 1 if c["lpt"] == 1 else 5
        return {"bytes": p3 * (24 + 24), "flops": chains * 3 * _fft_flops(c["np"]) + 100 * p3}
    if kind == "batch":
        one = c["steps"] * step + 24 * p3 + 4 * n3
        return {"bytes": c["count"] * (one + 24 * p3), "flops": c["count"] * (c["steps"] + 1) * flops}
    if kind == "spectra":
        nt = c["bk_bins"] * (c["bk_bins"] + 1) * (c["bk_bins"] + 2) // 6
        return {"bytes": 2 * 4 * n3, "flops": 2 * _fft_flops(c["nmesh"]) + c["bk_bins"] * _fft_flops(c["m"]) + 3.0 * nt * c["m"]**3}
    if kind == "bias":
        return {"bytes": 4 * n3 * 5, "flops": 2 * _fft_flops(c["nmesh"])}
    if kind == "combine":
        t3 = p3 * c["ratio"]**3
        return {"bytes": 24 * p3 + (24 + 12 + 24) * t3, "flops": 60.0 * t3}
    if kind == "gradient":
        # the run, and a reverse sweep that passes the same state and its cotangents once a step
        return {"bytes": c["steps"] * (step + 2 * step), "flops": 3.0 * c["steps"] * flops}
    e = 4 * wide
    return {"bytes": c["points"] * (3 * 3 * e + e + 8) + 3 * e * n3, "flops": 80.0 * c["points"]}
