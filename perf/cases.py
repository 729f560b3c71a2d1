"""Performance cases of the library: what its users have it do, over the sizes that they run.

Each case is one pass through public entry points of ``paper_2405_12913_gb300.hrt``: the PM force (deposit and
Poisson solve) and its transpose, the particle update with the next deposit, the ray step by either kick operator and
its transpose, the convergence power spectrum, and whole reverse co-evolution runs.  Sizes are those of the
workloads in ``configs.py`` and of the tests, with FFT-friendly sides in between.

Inputs are drawn with torch on the GPU from the seed alone: Zel'dovich-like displacements and potential gradients of a
Gaussian field with the power law x BBKS spectrum normalised to sigma8 = 0.8, pixel-grid ray angles.  ``exact`` states
every case in 64 bits with torch, without this package.
"""
import math

import numpy as np
import torch

from paper_2405_12913_gb300 import hrt

OMEGA_M, HUBBLE, N_S, SIGMA8 = 0.3, 0.7, 0.96, 0.8
C_LIGHT = 2997.92458
DECONV = 4.0
A_MID = 2.0 / 3.0  # scale factor of the ray and solve cases (the middle of a reverse run)


def listed():
    return [
        # smallest force: a ragged, non power-of-two mesh of a quick look or a test run; launch latency counts
        dict(name="force_60", kind="force", n=60, box=120.0, ray=False),
        # force of the 256^3 runs with a learned factor on the two ray fields (five fields out of one density)
        dict(name="force_256_ray", kind="force", n=256, box=256.0, ray=True),
        # the mesh between 512^3 and 1024^3 of the resolution ladder: not a power of two
        dict(name="force_768", kind="force", n=768, box=256.0, ray=False),
        # the full-size force: 512^3 particles on 1024^3 cells
        dict(name="force_1024", kind="force", n=1024, box=1000.0, ray=False),
        # backward of the solve at the size of the gradient workload
        dict(name="force_adjoint_256", kind="force_adjoint", n=256, box=256.0),
        # kick, drift and next deposit of 256^3 caller-owned particles on 512^3 cells
        dict(name="kick_deposit_256p", kind="kick", n_side=256, n=512, box=500.0),
        # one step of 2048^2 image rays through the 1024^3 fields with the map readout
        dict(name="ray_step_2048", kind="ray", n=1024, box=1000.0, n_pix=2048, fov=10.0, da=1.0 / 96.0),
        # backward of the ray step of the gradient workload
        dict(name="ray_adjoint_512", kind="ray_adjoint", n=256, box=256.0, n_pix=512, fov=3.5, da=1.0 / 32.0),
        # the ray-mesh kick operator at half the full side
        dict(name="ray_mesh_1024", kind="ray_mesh", n=512, box=500.0, n_pix=1024, fov=10.0, da=1.0 / 96.0),
        # analysis: convergence power spectrum of a full-size map
        dict(name="power_2048", kind="power", m=2048, fov=10.0),
        # a whole reverse run of the 128^3 / 256^3 / 512^2 workload (particles and rays, 16 steps, kappa map)
        dict(name="reverse_256", kind="reverse", n_side=128, n=256, box=256.0, n_pix=512, fov=3.5, steps=16, da=1.0 / 32.0),
        # the start of a full-size reverse run: 512^3 particles, 1024^3 cells, 2048^2 rays
        dict(name="reverse_1024", kind="reverse", n_side=512, n=1024, box=1000.0, n_pix=2048, fov=10.0, steps=8,
             da=1.0 / 96.0),
    ]


def _smooth_sides(lo, hi):
    return [n for n in range(lo, hi + 1, 2) if _is_smooth(n)]


def _is_smooth(n):
    for p in (2, 3, 5, 7):
        while n % p == 0:
            n //= p
    return n == 1


def _log_pick(rng, values):
    """One of the ascending values, spread evenly over their logarithm."""
    x = math.exp(rng.uniform(math.log(values[0]), math.log(values[-1])))
    return min(values, key=lambda v: abs(math.log(v / x)))


def draw(rng):
    kind = rng.choice(["force", "force", "force", "force_adjoint", "kick", "kick", "ray", "ray_adjoint", "ray_mesh",
                       "power", "reverse", "reverse"])
    cell = round(rng.uniform(0.5, 2.0), 3)
    if kind == "force":
        n = _log_pick(rng, _smooth_sides(48, 1024))
        return dict(kind=kind, n=n, box=n * cell, ray=rng.random() < 0.3 and n <= 512)
    if kind == "force_adjoint":
        n = _log_pick(rng, _smooth_sides(32, 512))
        return dict(kind=kind, n=n, box=n * cell)
    if kind == "kick":
        p = int(round(math.exp(rng.uniform(math.log(16), math.log(400)))))  # odd sides among them
        return dict(kind=kind, n_side=p, n=2 * p, box=2 * p * cell)
    if kind in ("ray", "ray_adjoint"):
        n = _log_pick(rng, _smooth_sides(32, 1024 if kind == "ray" else 512))
        m = int(round(math.exp(rng.uniform(math.log(60), math.log(2048 if kind == "ray" else 1024)))))
        return dict(kind=kind, n=n, box=n * cell, n_pix=m, fov=round(rng.uniform(2.0, 10.0), 2),
                    da=1.0 / rng.randint(32, 96))
    if kind == "ray_mesh":
        n = _log_pick(rng, _smooth_sides(64, 512))
        return dict(kind=kind, n=n, box=n * cell, n_pix=rng.randint(128, 1024), fov=round(rng.uniform(3.0, 10.0), 2),
                    da=1.0 / rng.randint(32, 96))
    if kind == "power":
        return dict(kind=kind, m=2 * int(round(math.exp(rng.uniform(math.log(30), math.log(1024))))),
                    fov=round(rng.uniform(2.0, 10.0), 2))
    p = _log_pick(rng, [v for v in range(10, 257) if _is_smooth(v)])
    return dict(kind="reverse", n_side=p, n=2 * p, box=2 * p * cell, n_pix=rng.randint(60, 1024),
                fov=round(rng.uniform(2.0, 10.0), 2), steps=rng.randint(2, 8), da=1.0 / rng.randint(32, 96))


# ------------------------------------------------------------------------------------------------ background (64 bits)
_GX, _GW = np.polynomial.legendre.leggauss(64)


def _integral(f, a, b):
    x = 0.5 * (b - a) * _GX + 0.5 * (a + b)
    return 0.5 * (b - a) * float(np.dot(_GW, f(x)))


def _g(x):
    return OMEGA_M + (1.0 - OMEGA_M) * x ** 3  # a^3 E^2


def _chi(a):
    return C_LIGHT * _integral(lambda x: x ** -0.5 * _g(x) ** -0.5, a, 1.0)


def _a_of_chi(chi):
    a = 1.0
    for _ in range(60):
        step = (_chi(a) - chi) / (-C_LIGHT * a ** -0.5 * _g(a) ** -0.5)
        a = min(1.5, max(1e-3, a - step))
        if abs(step) < 1e-15:
            break
    return a


def _growth(a):
    i = _integral(lambda t: 2.0 * a ** 2.5 * t ** 4 * _g(a * t * t) ** -1.5, 0.0, 1.0)
    i1 = _integral(lambda t: 2.0 * t ** 4 * _g(t * t) ** -1.5, 0.0, 1.0)
    return math.sqrt(_g(a) / a ** 3) * i / i1


def _kick_time(a, b):
    return _integral(lambda x: x ** 0.5 * _g(x) ** -0.5, a, b)


def _drift_time(a, b):
    return _integral(lambda x: x ** -1.5 * _g(x) ** -0.5, a, b)


def _power_shape(k):
    q = k / (OMEGA_M * HUBBLE)
    t = np.log1p(2.34 * q) / (2.34 * q) * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
    return k ** N_S * t * t


def _power_amplitude():
    lnk = np.linspace(math.log(1e-5), math.log(1e2), 20001)
    k = np.exp(lnk)
    x = 8.0 * k
    w = 3.0 * (np.sin(x) - x * np.cos(x)) / x ** 3
    y = k ** 3 * _power_shape(k) * w * w / (2.0 * math.pi ** 2)
    return SIGMA8 ** 2 / float(np.sum(0.5 * (y[1:] + y[:-1]) * np.diff(lnk)))


# ------------------------------------------------------------------------------------------------ inputs
def _freq(n, box, dtype):
    kf = 2.0 * math.pi / box
    f = torch.fft.fftfreq(n, d=1.0 / n, device="cuda").round().to(dtype) * kf
    return f, torch.arange(n // 2 + 1, device="cuda").to(dtype) * kf


def _zeldovich(seed, n, box, smooth, comps=3):
    """Displacement components (comps, n, n, n) in float32 of a Gaussian field at a = 1, smoothed over `smooth`."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.fft.rfftn(torch.randn(n, n, n, generator=g, device="cuda"))
    kx, kz = _freq(n, box, torch.float32)
    k_top = math.sqrt(3.0) * math.pi * n / box * 1.01
    table = np.linspace(0.0, k_top, 8192)
    amp = np.zeros_like(table)
    amp[1:] = np.sqrt(_power_amplitude() * _power_shape(table[1:]) * (n / box) ** 3) / table[1:] ** 2
    amp[1:] *= np.exp(-0.5 * (table[1:] * smooth) ** 2)
    amp = torch.tensor(amp, dtype=torch.float32, device="cuda")
    slab = max(1, (1 << 26) // (n * n))
    for i in range(0, n, slab):
        kk = torch.sqrt(kx[i:i + slab, None, None] ** 2 + kx[None, :, None] ** 2 + kz[None, None, :] ** 2)
        t = kk * (8191 / k_top)
        j = t.to(torch.int64).clamp_(max=8190)
        w[i:i + slab] *= amp[j] + (amp[j + 1] - amp[j]) * (t - j)
    w[0, 0, 0] = 0
    out = torch.empty(comps, n, n, n, device="cuda")
    for c in range(comps):
        d = kz.clone() if c == 2 else kx.clone()
        if n % 2 == 0:
            d[n // 2] = 0.0
        shape = [1, 1, 1]
        shape[c] = -1
        out[c] = torch.fft.irfftn(w * (1j * d.view(shape)), s=(n, n, n))
    return out


def _particles(seed, n_side, box):
    disp = _zeldovich(seed, n_side, box, max(2.0, box / n_side)).reshape(3, -1)
    return disp, disp * 0.5133  # p = a^2 E f Psi at a = 1


def _gradients(seed, n, box, comps=2):
    """d_j phi on the mesh: minus (3/2) Omega_m / a times the displacement field, smoothed over a cell."""
    return _zeldovich(seed, n, box, 1.0 * box / n, comps).mul_(-1.5 * OMEGA_M / A_MID)


def _pixels(m, fov):
    d = fov * math.pi / 180.0 / m
    c = (torch.arange(m, dtype=torch.float64, device="cuda") + 0.5 - 0.5 * m) * d
    ty, tx = torch.meshgrid(c, c, indexing="ij")
    return torch.stack([tx.reshape(-1), ty.reshape(-1)], 1).contiguous()


def _table(n, box):
    """A learned-like factor of the ray fields: smooth, above 1 at high |k|, up to 2 pi / cell."""
    k_max = 2.0 * math.pi * n / box
    x = torch.linspace(0.0, 1.0, 512, device="cuda")
    return (1.0 + 0.6 * x * x / (0.05 + x * x)).float().contiguous(), k_max


def _observer(box):
    return (0.5 * box, 0.5 * box, 0.0)


def _shell(case):
    return _chi(A_MID), _chi(A_MID - case["da"])


def _mu(case):
    return case["fov"] * math.pi / 180.0 / case["n_pix"]


IOTA, P_MIN = 0.5, 256.0


class State:
    def close(self):
        for name in ("pm", "rm", "ctx"):
            if getattr(self, name, None) is not None:
                getattr(self, name).close()

    def __del__(self):
        self.close()


def prepare(case, seed):
    s = State()
    s.case, kind = dict(case), case["kind"]
    box = case.get("box")
    if kind in ("force", "force_adjoint"):
        n = case["n"]
        s.pm = hrt.PM(n, box, 2 if case.get("ray") else 0)
        s.pref = 1.5 * OMEGA_M / A_MID
        s.f = hrt.make_filter(DECONV, box / n)
        if kind == "force_adjoint":
            g = torch.Generator(device="cuda").manual_seed(seed)
            s.bar0 = torch.randn(3, n, n, n, generator=g, device="cuda")
            s.bar, s.rho_bar = torch.empty_like(s.bar0), torch.empty(n, n, n, device="cuda")
            return s
        s.disp, _ = _particles(seed, n // 2, box)
        s.rho = torch.empty(n, n, n, device="cuda")
        s.grad = torch.empty(3, n, n, n, device="cuda")
        if case["ray"]:
            s.table, kmax = _table(n, box)
            s.f_ray = hrt.make_filter(DECONV, box / n, s.table, kmax)
            s.ray_grad = torch.empty(2, n, n, n, device="cuda")
    elif kind == "kick":
        s.disp, s.mom = _particles(seed, case["n_side"], box)
        s.grad = _gradients(seed + 1, case["n"], box, 3)
        s.rho = torch.empty(case["n"], case["n"], case["n"], device="cuda")
        s.kick, s.drift, s.sign = _kick_time(1.0, 1.0 - 1.0 / 64), _drift_time(1.0, 1.0 - 1.0 / 64), 1.0
    elif kind in ("ray", "ray_adjoint", "ray_mesh"):
        n, m = case["n"], case["n_pix"]
        s.grad = _gradients(seed, n, box)
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        jitter = torch.rand(m * m, 2, generator=g, device="cuda", dtype=torch.float64) - 0.5
        s.theta0 = _pixels(m, case["fov"]) + jitter * (0.5 * _mu(case))
        s.geom = hrt.make_geom(n, box, _observer(box), 1.0, image_width=m)
        s.chi = _shell(case)
        s.rays = hrt.RayState(m * m)
        if kind == "ray_adjoint":
            hrt.hrt_rays_init(s.rays, s.theta0)
            s.bar0 = [torch.randn(x.shape, generator=g, device="cuda").to(x.dtype)
                      for x in (s.rays.theta, s.rays.eta, s.rays.A, s.rays.B)]
            s.bar, s.grad_bar = hrt.RayState(m * m), torch.empty_like(s.grad)
            s.node_bar = torch.empty(3, hrt.MAX_RAY_NODES, dtype=torch.float64, device="cuda")
            s.drift_bar = torch.empty(1, dtype=torch.float64, device="cuda")
        else:
            s.maps = torch.empty(4, m * m, device="cuda")
        if kind == "ray_mesh":
            s.rm = hrt.RayMesh(hrt.make_raymesh_config(IOTA, P_MIN, _mu(case), m))
    elif kind == "power":
        s.kappa = _map(case, seed)
    else:
        s.disp, s.mom = _particles(seed, case["n_side"], box)
        s.theta0 = _pixels(case["n_pix"], case["fov"])
        s.ctx = hrt.Context(hrt.make_config(case["n"], box, case["n_side"], OMEGA_M, HUBBLE, N_S, SIGMA8, DECONV, 1.0, 1.0,
                                            _observer(box), n_sources=1))
    return s


def _map(case, seed):
    """A Gaussian convergence map with a falling spectrum, rms 0.02."""
    m = case["m"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.fft.rfft2(torch.randn(m, m, generator=g, device="cuda"))
    f, fz = _freq(m, 2.0 * math.pi, torch.float32)
    k2 = f[:, None] ** 2 + fz[None, :] ** 2
    x = torch.fft.irfft2(w * (1.0 + k2) ** -0.45, s=(m, m))
    return (x * (0.02 / x.std())).contiguous().reshape(-1)


def _power_args(case):
    m = case["m"]
    dtheta = case["fov"] * math.pi / 180.0 / m
    return m, dtheta, 20, 2.0 * math.pi / (m * dtheta), math.pi / dtheta


def run(s):
    c, kind = s.case, s.case["kind"]
    if kind == "force":
        hrt.hrt_cic_scatter(s.disp, c["n"] // 2, c["n"], c["box"], s.rho)
        if c["ray"]:
            s.pm.solve(s.rho, s.pref, s.f, s.grad, s.f_ray, s.ray_grad)
            return [s.grad, s.ray_grad]
        s.pm.solve(s.rho, s.pref, s.f, s.grad)
        return [s.grad]
    if kind == "force_adjoint":
        s.bar.copy_(s.bar0)  # the call destroys the cotangents it is given
        s.pm.solve_adjoint(s.bar, s.pref, s.f, s.rho_bar)
        return [s.rho_bar]
    if kind == "kick":  # forward and backward in turn: the particles stay where they are in earnest
        hrt.hrt_particle_kick_drift_deposit(s.grad, c["n"], c["box"], c["n_side"], s.disp, s.mom, s.sign * s.kick,
                                            s.sign * s.drift, s.rho)
        s.sign = -s.sign
        return [s.disp, s.mom, s.rho]
    if kind == "ray":
        hrt.hrt_rays_init(s.rays, s.theta0)
        hrt.hrt_ray_step(s.rays, s.grad[0], s.grad[1], s.geom, s.chi[0], s.chi[1], A_MID, OMEGA_M, s.maps)
        return [s.rays.theta, s.rays.eta, s.rays.A, s.rays.B, s.maps]
    if kind == "ray_mesh":
        hrt.hrt_rays_init(s.rays, s.theta0)
        s.rm.hrt_raymesh_ray_step(s.rays, s.grad[0], s.grad[1], s.geom, s.chi[0], s.chi[1], A_MID, OMEGA_M, s.maps)
        return [s.rays.theta, s.rays.eta, s.rays.A, s.rays.B, s.maps]
    if kind == "ray_adjoint":
        for x, y in zip((s.bar.theta, s.bar.eta, s.bar.A, s.bar.B), s.bar0):
            x.copy_(y)
        for x in (s.grad_bar, s.node_bar, s.drift_bar):
            x.zero_()
        hrt.hrt_ray_step_adjoint(s.rays, s.grad[0], s.grad[1], s.geom, s.chi[0], s.chi[1], A_MID, OMEGA_M, s.bar,
                                 s.grad_bar[0], s.grad_bar[1], s.node_bar, s.drift_bar)
        return [s.bar.theta, s.bar.eta, s.bar.A, s.bar.B, s.grad_bar, s.node_bar, s.drift_bar]
    if kind == "power":
        return list(hrt.hrt_kappa_power(s.kappa, *_power_args(c)))
    s.ctx.hrt_init_particles(s.disp, s.mom, 1.0)
    s.ctx.hrt_init_rays(s.theta0)
    for i in range(c["steps"]):
        s.ctx.hrt_step(1.0 - (i + 1) * c["da"], 0 if i + 1 == c["steps"] else -1)
    disp, mom, _, _ = s.ctx.hrt_read_particles()
    theta, eta, _, _ = s.ctx.hrt_read_rays()
    s.ctx.hrt_read_maps(0)
    # A, B and the maps are read but not returned: the derivative of the interpolant jumps where a line-of-sight node
    # crosses a cell face, and over a whole run the order of the deposit's atomics decides a few such crossings, so
    # that they differ by up to 1e-2 in single rays from one run to the next.  The ray cases return them.
    return [disp, mom, theta, eta]


# ------------------------------------------------------------------------------------------------ work
def _fft_flops(n):
    return 2.5 * n ** 3 * math.log2(float(n) ** 3)


def work(case):
    kind = case["kind"]
    if kind == "power":
        m = case["m"]
        return {"bytes": 4.0 * m * m, "flops": 5.0 * m * m * math.log2(m)}
    n = case["n"]
    cells = float(n) ** 3
    rays = float(case.get("n_pix", 0)) ** 2
    ray_io = rays * (16 + 48 + 16)  # initial angles in; state and maps out
    if kind in ("ray", "ray_adjoint", "ray_mesh"):
        chi = _shell(case)
        side = min(case["box"], 2.0 * math.tan(0.5 * math.radians(case["fov"])) * chi[1]) * n / case["box"]
        planes = min(float(n), (chi[1] - chi[0]) * n / case["box"] + 1)
        slab = 8.0 * side * side * planes
        nodes = rays * planes
        if kind == "ray_adjoint":
            return {"bytes": rays * (48 + 2 * 48) + slab + 8.0 * cells, "flops": nodes * 400}
        if kind == "ray_mesh":
            return {"bytes": ray_io + slab, "flops": 30.0 * side * side * planes + rays * 100}
        return {"bytes": ray_io + slab, "flops": nodes * 90}
    if kind == "force":
        fields = 5 if case["ray"] else 3
        return {"bytes": 12.0 * (n // 2) ** 3 + 4.0 * fields * cells, "flops": (1 + fields) * _fft_flops(n)}
    if kind == "force_adjoint":
        return {"bytes": 16.0 * cells, "flops": 4 * _fft_flops(n)}
    np_ = float(case["n_side"]) ** 3
    if kind == "kick":
        return {"bytes": 48.0 * np_ + 16.0 * cells, "flops": 150.0 * np_}
    steps = case["steps"]  # the particles and rays go in and out once; the fields of every force are read by both
    return {"bytes": 48.0 * np_ + ray_io + steps * (48.0 * np_ + 28.0 * cells + 96.0 * rays),
            "flops": (steps + 1) * 4 * _fft_flops(n) + steps * 150.0 * np_}


# ------------------------------------------------------------------------------------------------ 64 bits
def _corners(u, n):
    i0 = torch.floor(u)
    return i0.to(torch.int64) % n, u - i0


def _positions(disp, n_side, box, lo, hi):
    p = torch.arange(lo, hi, device="cuda")
    q = torch.stack([p // (n_side * n_side), (p // n_side) % n_side, p % n_side]).double() * (box / n_side)
    return q + disp[:, lo:hi].double()


def _cic(disp, n_side, n, box, chunk=1 << 24):
    rho = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    total = n_side ** 3
    for lo in range(0, total, chunk):
        i0, f = _corners(torch.remainder(_positions(disp, n_side, box, lo, min(total, lo + chunk)), box) * (n / box), n)
        for corner in range(8):
            w, idx = (n ** 3 / total), 0
            for a in range(3):
                up = (corner >> a) & 1
                w = w * (f[a] if up else 1.0 - f[a])
                idx = idx * n + (i0[a] + up) % n
            rho.index_add_(0, idx, w)
    return rho.view(n, n, n)


def _multiplier(n, box, pref, smooth, table=None, k_max=0.0):
    """G(k) W(k) [g(|k|)] on x-slabs of the half spectrum: a function of the slab."""
    kx, kz = _freq(n, box, torch.float64)

    def sinc(k):
        x = 0.5 * k * box / n
        return torch.where(x == 0, torch.ones_like(x), torch.sin(x) / torch.where(x == 0, torch.ones_like(x), x))

    def slab(lo, hi):
        ks = kx[lo:hi, None, None], kx[None, :, None], kz[None, None, :]
        k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
        m = torch.where(k2 > 0, -pref / torch.where(k2 > 0, k2, torch.ones_like(k2)), torch.zeros_like(k2))
        m = m * (sinc(ks[0]) * sinc(ks[1]) * sinc(ks[2])) ** -DECONV * torch.exp(-0.5 * k2 * smooth * smooth)
        if table is not None:
            t = torch.sqrt(k2) * ((table.numel() - 1) / k_max)
            j = t.to(torch.int64).clamp(max=table.numel() - 2)
            g = table.double()
            m = m * torch.where(t < table.numel() - 1, g[j] + (g[j + 1] - g[j]) * (t - j), torch.ones_like(t))
        return m

    return slab


def _derivative(n, box, c):
    kx, kz = _freq(n, box, torch.float64)
    d = (kz if c == 2 else kx).clone()
    d[n // 2] = 0.0
    shape = [1, 1, 1]
    shape[c] = -1
    return d.view(shape)


def _solve(rho, box, pref, smooth, comps=3, table=None, k_max=0.0):
    n = rho.shape[0]
    phi = torch.fft.rfftn(rho)
    slab = _multiplier(n, box, pref, smooth, table, k_max)
    step = max(1, (1 << 26) // (n * n))
    for i in range(0, n, step):
        phi[i:i + step] *= slab(i, i + step)
    return [torch.fft.irfftn(phi * (1j * _derivative(n, box, c)), s=(n, n, n)) for c in range(comps)]


def _kick_drift(disp, mom, grads, n_side, n, box, kick, drift, chunk=1 << 24):
    total = n_side ** 3
    flat = [g.reshape(-1) for g in grads]
    for lo in range(0, total, chunk):
        hi = min(total, lo + chunk)
        i0, f = _corners(torch.remainder(_positions(disp, n_side, box, lo, hi), box) * (n / box), n)
        for corner in range(8):
            w, idx = 1.0, 0
            for a in range(3):
                up = (corner >> a) & 1
                w = w * (f[a] if up else 1.0 - f[a])
                idx = idx * n + (i0[a] + up) % n
            for a in range(3):
                mom[a, lo:hi] -= kick * w * flat[a][idx]
        disp[:, lo:hi] += drift * mom[:, lo:hi]


def _nodes(chi_a, chi_b, cell, a_ref):
    count = max(1, math.ceil(abs(chi_b - chi_a) / cell))
    h = (chi_b - chi_a) / count
    out = []
    for j in range(count):
        chi = chi_a + (j + 0.5) * h
        a = _a_of_chi(chi)
        out.append((chi, -(2.0 / C_LIGHT) * h * chi * _growth(a) / _growth(a_ref) * a_ref / a))
    return out


def _node_gather(gx, gy, theta, chi, box):
    """Trilinear (d_x phi, d_y phi) and its transverse derivative at the rays' points at distance chi."""
    n = gx.shape[0]
    o = _observer(box)
    ix, fx = _corners(torch.remainder(o[0] + chi * theta[:, 0], box) * (n / box), n)
    iy, fy = _corners(torch.remainder(o[1] + chi * theta[:, 1], box) * (n / box), n)
    uz = ((o[2] + chi) % box) * (n / box)
    iz, fz = int(math.floor(uz)) % n, uz - math.floor(uz)
    ix1, iy1, val, der = (ix + 1) % n, (iy + 1) % n, [], []
    inv = n / box
    for g in (gx, gy):
        flat = (g[:, :, iz] * (1.0 - fz) + g[:, :, (iz + 1) % n] * fz).reshape(-1).double()
        v00, v01, v10, v11 = flat[ix * n + iy], flat[ix * n + iy1], flat[ix1 * n + iy], flat[ix1 * n + iy1]
        low, high = v00 + (v01 - v00) * fy, v10 + (v11 - v10) * fy
        val.append(low + (high - low) * fx)
        der.append(torch.stack([(high - low) * inv, ((v01 - v00) * (1.0 - fx) + (v11 - v10) * fx) * inv], 1))
    return torch.stack(val, 1), torch.stack(der, 1)


def _half_kick(theta, gx, gy, chi_a, chi_b, box, a_ref):
    kick = torch.zeros_like(theta)
    jac = theta.new_zeros(theta.shape[0], 2, 2)
    for chi, c in _nodes(chi_a, chi_b, box / gx.shape[0], a_ref):
        val, der = _node_gather(gx, gy, theta, chi, box)
        kick = kick + c * val
        jac = jac + (c * chi) * der
    return kick, jac


def _init_rays(theta0):
    r = theta0.shape[0]
    eye = torch.eye(2, dtype=torch.float64, device="cuda").expand(r, 2, 2).clone()
    return theta0.clone(), torch.zeros(r, 2, dtype=torch.float64, device="cuda"), eye, torch.zeros_like(eye)


def _ray_step(state, chi_a, chi_b, half):
    theta, eta, A, B = state
    mid = 0.5 * (chi_a + chi_b)
    kick, jac = half(theta, chi_a, mid)
    eta, B = eta + kick, B + jac @ A
    d = (chi_b - chi_a) / (C_LIGHT * mid * mid)
    theta, A = theta + d * eta, A + d * B
    kick, jac = half(theta, mid, chi_b)
    return theta, eta + kick, A, B + jac @ A


def _maps(A):
    c1, c2 = 0.5 * (A[:, 0, 0] + A[:, 1, 1]), 0.5 * (A[:, 0, 1] - A[:, 1, 0])
    c3, c4 = 0.5 * (A[:, 1, 1] - A[:, 0, 0]), 0.5 * (A[:, 0, 1] + A[:, 1, 0])
    w = c2 / c1
    return torch.stack([1.0 - c1, c3 + c4 * w, c3 * w - c4, w])


def _rays_out(state):
    theta, eta, A, B = state
    return [theta, eta, A.reshape(-1, 4), B.reshape(-1, 4), _maps(A)]


def _mesh_kick(gx, gy, box, chi_a, chi_b, mu, m_pix, a_ref):
    """The filtered ray mesh (2, N, N) of a half shell and its spacing: CIC projection of the node planes."""
    n = gx.shape[0]
    cell, o = box / n, _observer(box)
    lam = max(2.0 * cell / (chi_a + chi_b), mu)
    x2d = IOTA * lam
    need = math.ceil(m_pix * mu / x2d + P_MIN / IOTA)
    side = 1 << max(0, need - 1).bit_length()
    mesh = torch.zeros(2, side * side, dtype=torch.float64, device="cuda")
    lo, hi = min(chi_a, chi_b), max(chi_a, chi_b)
    node = torch.arange(n, dtype=torch.float64, device="cuda") * cell
    for kz in range(math.ceil((o[2] + lo) / cell) - 1, math.ceil((o[2] + hi) / cell) + 1):
        chi = kz * cell - o[2]
        if not (lo <= chi < hi and chi > 0):
            continue
        a = _a_of_chi(chi)
        w = -(2.0 / C_LIGHT) * chi * _growth(a) / _growth(a_ref) * a_ref / a * math.copysign(1.0, chi_b - chi_a)
        w *= cell ** 3 / (chi * x2d) ** 2
        plane = [gx[:, :, kz % n].double() * w, gy[:, :, kz % n].double() * w]
        reach = (0.5 * side * x2d + x2d) * chi + cell
        axis = []
        for d in range(2):
            first, last = math.floor((o[d] - reach) / box), math.floor((o[d] + reach) / box)
            u = torch.cat([(node + i * box - o[d]) / chi / x2d + side // 2 for i in range(first, last + 1)])
            who = torch.arange(n, device="cuda").repeat(last - first + 1)
            ok = (u > -1) & (u < side)
            axis.append((u[ok], who[ok]))
        (ux, wx), (uy, wy) = axis
        jx, jy = torch.floor(ux), torch.floor(uy)
        for dx in (0, 1):
            for dy in (0, 1):
                tx, ty = (jx + dx).long(), (jy + dy).long()
                fx = (ux - jx if dx else 1.0 - (ux - jx)) * ((tx >= 0) & (tx < side))
                fy = (uy - jy if dy else 1.0 - (uy - jy)) * ((ty >= 0) & (ty < side))
                idx = (tx.clamp(0, side - 1)[:, None] * side + ty.clamp(0, side - 1)[None, :]).reshape(-1)
                weight = fx[:, None] * fy[None, :]
                for c in range(2):
                    mesh[c].index_add_(0, idx, (weight * plane[c][wx][:, wy]).reshape(-1))
    k = 2.0 * math.pi * torch.fft.fftfreq(side, d=x2d, dtype=torch.float64, device="cuda")
    s = torch.special.sinc(k * (x2d / (2.0 * math.pi))) ** -4 * torch.exp(-0.5 * k * k * lam * lam)
    return torch.fft.ifft2(torch.fft.fft2(mesh.view(2, side, side)) * (s[:, None] * s[None, :])).real, x2d


def _mesh_gather(mesh, x2d, theta):
    side = mesh.shape[1]
    u = theta / x2d + side // 2
    j = torch.floor(u)
    f = u - j
    val, der = torch.zeros_like(theta), theta.new_zeros(theta.shape[0], 2, 2)
    for dx in (0, 1):
        for dy in (0, 1):
            jx, jy = (j[:, 0] + dx).long(), (j[:, 1] + dy).long()
            ok = (jx >= 0) & (jx < side) & (jy >= 0) & (jy < side)
            wx, wy = (f[:, 0] if dx else 1.0 - f[:, 0]), (f[:, 1] if dy else 1.0 - f[:, 1])
            for c in range(2):
                v = mesh[c][jx.clamp(0, side - 1), jy.clamp(0, side - 1)] * ok
                val[:, c] += wx * wy * v
                der[:, c, 0] += (2 * dx - 1) / x2d * wy * v
                der[:, c, 1] += (2 * dy - 1) / x2d * wx * v
    return val, der


def _exact_power(case, seed):
    m, dtheta, bins, lo, hi = _power_args(case)
    p = torch.fft.fft2(_map(case, seed).view(m, m).double()).abs().cpu().numpy() ** 2 * dtheta ** 4 / (m * dtheta) ** 2
    f = np.fft.fftfreq(m, d=1.0 / m).round()
    ell = 2.0 * math.pi * np.sqrt(f[:, None] ** 2 + f[None, :] ** 2) / (m * dtheta)
    with np.errstate(divide="ignore"):
        b = np.floor(bins * np.log(ell / lo) / math.log(hi / lo) + 1e-9)
    ok = (ell > 0) & (b >= 0) & (b < bins)
    b = b[ok].astype(np.int64)
    count = np.bincount(b, minlength=bins)
    some = np.maximum(count, 1)
    return [np.bincount(b, ell[ok], bins) / some, np.bincount(b, p[ok], bins) / some, None]


def _exact_ray_adjoint(case, seed):
    s = prepare(case, seed)
    n, box = case["n"], case["box"]
    # leaves: the ray state, the fields, and the node table as the step's coefficients
    state = [x.requires_grad_() for x in _init_rays(s.theta0)]
    fields = s.grad.double().requires_grad_()
    chi_a, chi_b = s.chi
    mid = 0.5 * (chi_a + chi_b)
    coef = [_nodes(a, b, box / n, A_MID) for a, b in ((chi_a, mid), (mid, chi_b))]
    split, nodes = len(coef[0]), coef[0] + coef[1]
    chis = [c[0] for c in nodes]
    cw = torch.tensor([c[1] for c in nodes], dtype=torch.float64, device="cuda")
    cwr = torch.tensor([c[1] * c[0] * n / box for c in nodes], dtype=torch.float64, device="cuda")
    drift = torch.tensor((chi_b - chi_a) / (C_LIGHT * mid * mid), dtype=torch.float64, device="cuda")
    cw.requires_grad_()
    cwr.requires_grad_()
    drift.requires_grad_()

    bars = [b.double().view_as(x) for b, x in zip(s.bar0, state)]
    # the step by hand, so that one node's graph lives at a time: a forward pass, then the reverse pass node by node
    with torch.no_grad():
        theta, eta, A, B = (x.detach() for x in state)
        halves = []
        for h in (0, 1):
            lo, hi = (0, split) if h == 0 else (split, len(nodes))
            kick, jac = torch.zeros_like(theta), torch.zeros_like(A)
            for j in range(lo, hi):
                val, der = _node_gather(fields[0], fields[1], theta, chis[j], box)
                kick += cw[j] * val
                jac += cwr[j] * der * (box / n)
            halves.append((theta, A, jac, lo, hi))
            eta, B = eta + kick, B + jac @ A
            if h == 0:
                eta1, B1 = eta, B
                theta, A = theta + drift * eta, A + drift * B
    tb, eb, Ab, Bb = bars
    out = dict(fields=torch.zeros_like(fields), cw=torch.zeros_like(cw), cwr=torch.zeros_like(cwr),
               chi=torch.zeros_like(cw))

    def back(h, tb, eb, Ab, Bb):
        theta, A, jac, lo, hi = halves[h]
        Jb = Bb @ A.transpose(1, 2)
        Ab = Ab + jac.transpose(1, 2) @ Bb
        for j in range(lo, hi):
            th = theta.clone().requires_grad_()
            ch = torch.tensor(chis[j], dtype=torch.float64, device="cuda")
            z = int(math.floor(((chis[j] % box)) * (n / box))) % n
            local = [fields[c][:, :, [z, (z + 1) % n]].detach().clone().requires_grad_() for c in (0, 1)]
            with torch.enable_grad():
                chl = ch.requires_grad_()
                val, der = _gather_two(local, th, chl, box, n)
                loss = cw[j].detach() * (eb * val).sum() + cwr[j].detach() * (box / n) * (Jb * der).sum()
                parts = torch.autograd.grad(loss, [th, local[0], local[1], chl])
            with torch.no_grad():
                tb = tb + parts[0]
                for c in (0, 1):
                    out["fields"][c][:, :, z] += parts[1 + c][:, :, 0]
                    out["fields"][c][:, :, (z + 1) % n] += parts[1 + c][:, :, 1]
                out["chi"][j] = parts[3]
                out["cw"][j] = (eb * val).sum()
                out["cwr"][j] = (box / n) * (Jb * der).sum()
        return tb, eb, Ab, Bb

    with torch.no_grad():
        tb, eb, Ab, Bb = back(1, tb, eb, Ab, Bb)
        drift_bar = (tb * eta1).sum() + (Ab * B1).sum()
        d = drift.detach()
        eb, Bb = eb + d * tb, Bb + d * Ab
        tb, eb, Ab, Bb = back(0, tb, eb, Ab, Bb)
    node = torch.zeros(3, hrt.MAX_RAY_NODES, dtype=torch.float64, device="cuda")
    k = len(nodes)
    node[0, :k], node[1, :k] = out["cw"], out["cwr"]
    return [tb, eb, Ab.reshape(-1, 4), Bb.reshape(-1, 4), out["fields"], None, drift_bar.reshape(1)]


def _gather_two(planes, theta, chi, box, n):
    """_node_gather on the two z-planes that hold the node, differentiable in theta, chi and the planes."""
    o = _observer(box)
    ux = torch.remainder(o[0] + chi * theta[:, 0], box) * (n / box)
    uy = torch.remainder(o[1] + chi * theta[:, 1], box) * (n / box)
    uz = torch.remainder(o[2] + chi, box) * (n / box)
    ix, iy = torch.floor(ux.detach()), torch.floor(uy.detach())
    fx, fy, fz = ux - ix, uy - iy, uz - torch.floor(uz.detach())
    ix, iy = ix.long() % n, iy.long() % n
    ix1, iy1, val, der = (ix + 1) % n, (iy + 1) % n, [], []
    for p in planes:
        flat = (p[:, :, 0] * (1.0 - fz) + p[:, :, 1] * fz).reshape(-1)
        v00, v01, v10, v11 = flat[ix * n + iy], flat[ix * n + iy1], flat[ix1 * n + iy], flat[ix1 * n + iy1]
        low, high = v00 + (v01 - v00) * fy, v10 + (v11 - v10) * fy
        val.append(low + (high - low) * fx)
        der.append(torch.stack([(high - low) * (n / box), ((v01 - v00) * (1.0 - fx) + (v11 - v10) * fx) * (n / box)], 1))
    return torch.stack(val, 1), torch.stack(der, 1)


def exact(case, seed):
    kind, box = case["kind"], case.get("box")
    if kind == "power":
        return _exact_power(case, seed)
    if kind == "ray_adjoint":
        return _exact_ray_adjoint(case, seed)
    n = case["n"]
    pref = 1.5 * OMEGA_M / A_MID
    if kind == "force":
        disp, _ = _particles(seed, n // 2, box)
        rho = _cic(disp, n // 2, n, box)
        out = [torch.stack(_solve(rho, box, pref, box / n))]
        if case["ray"]:
            table, k_max = _table(n, box)
            out.append(torch.stack(_solve(rho, box, pref, box / n, 2, table, k_max)))
        return out
    if kind == "force_adjoint":
        g = torch.Generator(device="cuda").manual_seed(seed)
        bar = torch.randn(3, n, n, n, generator=g, device="cuda")
        total = 0
        slab = _multiplier(n, box, pref, box / n)(0, n)
        for c in range(3):
            total = total + torch.fft.rfftn(bar[c].double()) * (-1j * _derivative(n, box, c)) * slab
        return [torch.fft.irfftn(total, s=(n, n, n))]
    if kind == "kick":
        n_side = case["n_side"]
        disp, mom = (x.double() for x in _particles(seed, n_side, box))
        grad = _gradients(seed + 1, n, box, 3).double()
        _kick_drift(disp, mom, grad, n_side, n, box, _kick_time(1.0, 1.0 - 1.0 / 64), _drift_time(1.0, 1.0 - 1.0 / 64))
        return [disp, mom, _cic(disp, n_side, n, box)]
    if kind in ("ray", "ray_mesh"):
        s = prepare(case, seed)
        if kind == "ray":
            def half(theta, a, b):
                return _half_kick(theta, s.grad[0], s.grad[1], a, b, box, A_MID)
        else:
            def half(theta, a, b):
                return _mesh_gather(*_mesh_kick(s.grad[0], s.grad[1], box, a, b, _mu(case), case["n_pix"], A_MID), theta)
        return _rays_out(_ray_step(_init_rays(s.theta0), *s.chi, half))
    n_side = case["n_side"]
    disp, mom = (x.double() for x in _particles(seed, n_side, box))
    rays = _init_rays(_pixels(case["n_pix"], case["fov"]))
    a, a_mom = 1.0, 1.0
    for i in range(case["steps"]):
        grads = _solve(_cic(disp, n_side, n, box), box, 1.5 * OMEGA_M / a, box / n)
        a_next = 1.0 - (i + 1) * case["da"]
        rays = _ray_step(rays, _chi(a), _chi(a_next), lambda t, p, q: _half_kick(t, grads[0], grads[1], p, q, box, a))
        mid = 0.5 * (a + a_next)
        _kick_drift(disp, mom, grads, n_side, n, box, _kick_time(a_mom, mid), _drift_time(a, a_next))
        a, a_mom = a_next, mid
    return [disp, mom, rays[0], rays[1]]
