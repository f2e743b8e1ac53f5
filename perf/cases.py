"""The work a user of the channel solver has it do, as cases that can be timed and checked.

Sizes and physical parameters are those of the workloads in ``paper_2406_01322_gb300/inputs.py``
(tiny, medium and large channel, uneven ensemble, adjoint channel) and ragged {2,3}-smooth sizes
of the same range.  Each case goes through the public entry points of the binding:

kind        one pass
step        ``Grid.step(n)`` on a running channel, then its spectral state
run         a whole short simulation: ``set_fields``, ``step(n)``, ``get_fields``
ensemble    ``Ensemble.step(n)`` of uneven channels, then every member's spectral state
gradient    ``objective_after`` and its backward pass (J and the four gradients)
lines       ``Grid.chebyshev_lines`` there and back on a stack of fields
transform   ``Grid.transform_forward`` and ``Grid.transform_backward`` of one field
noalloc     ``transform_forward_noalloc``
monitor     ``Grid.diagnostics`` and ``Grid.get_fields`` between steps

Results of mixed-precision channels come back in float32, the precision that their transforms
carry and that a program stores them in; everything else in float64.
"""
import math

import numpy as np
import torch

from paper_2406_01322_gb300 import binding

DEV = "cuda:0"
FP64, MIXED, DFLOAT = binding.PREC_FP64, binding.PREC_MIXED, binding.PREC_DFLOAT
LX, LY = 4.0 * math.pi, 2.0 * math.pi


def listed():
    return [
        # a caller that may not allocate transforms one small field: launches and latency only
        dict(name="noalloc_32", kind="noalloc", nx=32, ny=32, nz=33),
        # the tiny channel, run whole as in a parameter scan: every kernel is far below a wave
        dict(name="run_32_fp64", kind="run", nx=32, ny=32, nz=33, precision=FP64, tc=False,
             steps=10, drops=1, re_tau=150.0, ch=0.05, dt=1e-4),
        # the medium channel in float64 with the default settings
        dict(name="step_128_fp64", kind="step", nx=128, ny=128, nz=129, precision=FP64, tc=False,
             steps=4, drops=8, re_tau=150.0, ch=0.02, dt=5e-5),
        # the same with the tensor-core Chebyshev transform, the faster method on this grid
        dict(name="step_128_fp64_tc", kind="step", nx=128, ny=128, nz=129, precision=FP64, tc=True,
             steps=4, drops=8, re_tau=150.0, ch=0.02, dt=5e-5),
        # the large production channel: mixed precision, tensor-core Chebyshev transform
        dict(name="step_512_mixed_tc", kind="step", nx=512, ny=256, nz=257, precision=MIXED,
             tc=True, steps=2, drops=64, re_tau=300.0, ch=0.01, dt=2e-5),
        # double-float x/y work on a grid whose lengths are no powers of two
        dict(name="step_192_dfloat_tc", kind="step", nx=192, ny=144, nz=193, precision=DFLOAT,
             tc=True, steps=2, drops=8, re_tau=150.0, ch=0.02, dt=5e-5),
        # ragged mixed channel (2 3^4 in x and z) with the default Chebyshev method
        dict(name="step_162_mixed", kind="step", nx=162, ny=108, nz=163, precision=MIXED, tc=False,
             steps=4, drops=8, re_tau=150.0, ch=0.02, dt=5e-5),
        # uneven ensemble of small channels advanced together
        dict(name="ensemble_16_mixed_tc", kind="ensemble", members=16, precision=MIXED, tc=True,
             steps=2, re_tau=150.0, ch=0.03, dt=5e-5),
        # sensitivity of the final state: forward run with checkpoints, reverse sweep
        dict(name="gradient_128", kind="gradient", nx=128, ny=128, nz=129, precision=FP64,
             tc=False, steps=4, every=2, drops=4, re_tau=150.0, ch=0.02, dt=5e-5),
        # Chebyshev transforms of a stack of fields for post-processing
        dict(name="lines_128_tc", kind="lines", nx=128, ny=64, nz=129, precision=FP64, tc=True,
             fields=5),
        # analysis transform of one physical field and back
        dict(name="transform_256", kind="transform", nx=256, ny=128, nz=129, precision=FP64,
             tc=False),
        # what a run looks at between its steps: diagnostics and a snapshot
        dict(name="monitor_192", kind="monitor", nx=192, ny=192, nz=97, precision=FP64, tc=False,
             drops=8, re_tau=150.0, ch=0.02, dt=5e-5),
    ]


# {2,3}-smooth sizes: even lengths whose halves are smooth, and wall-normal degrees
EVEN = sorted({2 ** a * 3 ** b for a in range(1, 10) for b in range(0, 5)
               if 24 <= 2 ** a * 3 ** b <= 512})
DEGREES = sorted({2 ** a * 3 ** b for a in range(1, 9) for b in range(0, 5)
                  if 16 <= 2 ** a * 3 ** b <= 256})
# points x steps of a pass that stay within the cost of the largest listed case
COST = {FP64: 5.5e6, MIXED: 2.2e7, DFLOAT: 9e6}


def _near(sizes, lo, hi, rng):
    """A size drawn evenly over the logarithm of the range."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((s for s in sizes if lo <= s <= hi), key=lambda s: (abs(math.log(s / want)), s))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "run", "ensemble", "gradient", "lines",
                       "transform", "noalloc", "monitor"])
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(3, 20), precision=rng.choice([MIXED, FP64]),
                    tc=rng.random() < 0.6, steps=rng.randint(1, 2), re_tau=150.0, ch=0.03, dt=5e-5,
                    which=rng.randint(0, 1 << 20))
    big = {"step": 512, "run": 96, "gradient": 192, "lines": 256, "transform": 384,
           "noalloc": 96, "monitor": 256}[kind]
    nx, ny = _near(EVEN, 24, big, rng), _near(EVEN, 24, min(big, 256), rng)
    nz = _near(DEGREES, 16, min(256, max(64, big)), rng) + 1
    precision = rng.choice([FP64, MIXED, DFLOAT]) if kind in ("step", "run") else FP64
    tc = kind in ("step", "lines") and rng.random() < 0.6
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, tc=tc)
    if kind == "lines":
        c["fields"] = rng.randint(1, 7)
        while c["nx"] * c["ny"] * nz * c["fields"] > 5e7:
            c["nx"] = _near(EVEN, 24, c["nx"] // 2, rng)
    if kind in ("transform", "monitor", "noalloc"):
        while c["nx"] * c["ny"] * nz > (1.5e6 if kind == "noalloc" else 1e7):
            c["nx"] = _near(EVEN, 24, max(24, c["nx"] // 2), rng)
    if kind in ("noalloc", "lines", "transform"):
        return c
    c.update(drops=rng.randint(1, 16), re_tau=rng.choice([150.0, 300.0]), ch=0.02, dt=5e-5)
    if kind == "gradient":
        c.update(steps=rng.randint(1, 4), every=rng.randint(1, 3))
        while c["nx"] * c["ny"] * nz * c["steps"] > 4e6 and c["nx"] > 24:
            c["nx"] = _near(EVEN, 24, max(24, c["nx"] // 2), rng)
    elif kind in ("step", "run"):
        c["steps"] = rng.randint(1, 4) if kind == "step" else rng.randint(2, 10)
        while c["nx"] * c["ny"] * nz > COST[precision] and c["nx"] > 24:
            c["nx"] = _near(EVEN, 24, max(24, c["nx"] // 2), rng)
        c["steps"] = max(1, min(c["steps"], int(COST[precision] / (c["nx"] * c["ny"] * nz))))
    return c


def members(case):
    """Sizes of an ensemble's members, as the uneven ensemble workload draws them."""
    rng = np.random.Generator(np.random.PCG64(4 + case.get("which", 0)))
    return [dict(nx=int(rng.choice([64, 96, 128])), ny=int(rng.choice([64, 128])),
                 nz=int(rng.choice([65, 97, 129]))) for _ in range(case["members"])]


def fields(nx, ny, nz, re_tau, ch, drops, seed):
    """(u, v, w, phi) on the GPU: the laminar profile with a divergence-free no-slip perturbation of
    32 seeded Fourier modes (1 <= |mode| <= 8, energy falling with the wavenumber, of the size of
    the friction velocity), and seeded spherical drops with the equilibrium tanh profile."""
    rng = np.random.Generator(np.random.PCG64(seed))
    f64 = dict(dtype=torch.float64, device=DEV)
    x = torch.arange(nx, **f64) * (LX / nx)
    y = torch.arange(ny, **f64) * (LY / ny)
    z = torch.cos(torch.arange(nz, **f64) * (math.pi / (nz - 1)))
    f, df, g = (1 - z * z) ** 2, -4 * z * (1 - z * z), 1 - z * z
    u, v, w = (torch.zeros((nz, ny, nx), **f64) for _ in range(3))

    def add(out, coef, prof, ex, ey):
        plane = torch.real(coef * ey[:, None] * ex[None, :])
        out += prof[:, None, None] * plane[None]

    for _ in range(32):
        mx, my = int(rng.integers(0, 9)), int(rng.integers(-8, 9))
        if mx == 0 and my == 0:
            mx = 1
        kx, ky = 2 * math.pi * mx / LX, 2 * math.pi * my / LY
        k2 = kx * kx + ky * ky
        amp = 0.5 / (1.0 + k2)
        a = amp * complex(rng.uniform(-1, 1), rng.uniform(-1, 1))
        b = amp * complex(rng.uniform(-1, 1), rng.uniform(-1, 1))
        ex, ey = torch.exp(1j * kx * x), torch.exp(1j * ky * y)
        add(w, a, f, ex, ey)
        add(u, 1j * kx / k2 * a, df, ex, ey)
        add(v, 1j * ky / k2 * a, df, ex, ey)
        add(u, 1j * ky / math.sqrt(k2) * b, g, ex, ey)
        add(v, -1j * kx / math.sqrt(k2) * b, g, ex, ey)
    u += (0.5 * re_tau * (1 - z * z))[:, None, None]
    radius = 0.4 if drops == 1 else 0.3 if drops <= 16 else 0.2
    d2 = torch.full((nz, ny, nx), 1e30, **f64)
    for _ in range(drops):
        cx, cy = rng.uniform(0, LX), rng.uniform(0, LY)
        cz = rng.uniform(-0.9 + radius, 0.9 - radius)
        rx = torch.remainder(x - cx + LX / 2, LX) - LX / 2
        ry = torch.remainder(y - cy + LY / 2, LY) - LY / 2
        d2 = torch.minimum(d2, (z - cz)[:, None, None] ** 2 + ry[None, :, None] ** 2
                           + rx[None, None, :] ** 2)
    phi = torch.tanh((radius - torch.sqrt(d2)) / (math.sqrt(2.0) * ch))
    return u, v, w, phi


def _physics(case):
    return dict(re_tau=case["re_tau"], we=1.0, ch=case["ch"], pe=1.0 / case["ch"], dt=case["dt"])


def _fields(case, seed):
    return fields(case["nx"], case["ny"], case["nz"], case["re_tau"], case["ch"], case["drops"],
                  seed)


def _member_fields(case, seed):
    return [fields(m["nx"], m["ny"], m["nz"], case["re_tau"], case["ch"], 1, 1000 * seed + i)
            for i, m in enumerate(members(case))]


def _field(case, seed):
    """One smooth physical field with broadband noise, as a snapshot has."""
    u = fields(case["nx"], case["ny"], case["nz"], 150.0, 0.02, 4, seed)[3]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return u + 1e-3 * torch.randn(u.shape, dtype=torch.float64, device=DEV, generator=gen)


def _lines(case, seed):
    """Stacks of complex z lines, sizes falling with the wavenumber, as the step's fields have."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    shape = (case["fields"], case["nx"] // 2, case["ny"], case["nz"])
    r = torch.randn(shape + (2,), dtype=torch.float64, device=DEV, generator=gen)
    m = torch.arange(shape[1], dtype=torch.float64, device=DEV)[:, None]
    j = torch.arange(shape[2], dtype=torch.float64, device=DEV)[None, :]
    size = 1.0 / (1.0 + m * m + torch.minimum(j, shape[2] - j) ** 2)
    return torch.view_as_complex(r) * size[None, :, :, None]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "noalloc":
        spec = torch.empty((case["nx"] // 2, case["ny"], case["nz"]), dtype=torch.complex128,
                           device=DEV)
        return dict(kind=kind, f=_field(case, seed), spec=spec)
    if kind == "ensemble":
        e = binding.Ensemble([dict(m, **_physics(case)) for m in members(case)],
                             precision=case["precision"])
        if case["tc"]:
            e.set_chebyshev(binding.CHEB_TC)
        for g, f in zip(e.grids, _member_fields(case, seed)):
            g.set_fields(*f)
        return dict(kind=kind, e=e, steps=case["steps"], mixed=case["precision"] == MIXED)
    phys = _physics(case) if "dt" in case else {}
    g = binding.Grid(case["nx"], case["ny"], case["nz"], precision=case["precision"], **phys)
    if case["tc"]:
        g.set_chebyshev(binding.CHEB_TC)
    s = dict(kind=kind, g=g, steps=case.get("steps", 0), mixed=case["precision"] == MIXED)
    if kind == "lines":
        s["x"] = _lines(case, seed)
    elif kind == "transform":
        s["f"] = _field(case, seed)
    elif kind in ("step", "monitor"):
        g.set_fields(*_fields(case, seed))
    else:
        s["f"] = _fields(case, seed)
        s["every"] = case.get("every", 0)
    return s


def _stored(s, tensors):
    """Results as the program keeps them: float32 (complex64) from a mixed-precision channel."""
    if not s["mixed"]:
        return list(tensors)
    return [t.to(torch.complex64 if t.is_complex() else torch.float32) for t in tensors]


def run(s):
    kind = s["kind"]
    if kind == "noalloc":
        return binding.transform_forward_noalloc(s["f"], s["spec"])
    if kind == "ensemble":
        s["e"].step(s["steps"])
        return [t for g in s["e"].grids for t in _stored(s, g.get_spectral())]
    g = s["g"]
    if kind == "step":
        g.step(s["steps"])
        return _stored(s, g.get_spectral())
    if kind == "run":
        g.set_fields(*s["f"])
        g.step(s["steps"])
        return _stored(s, g.get_fields())
    if kind == "gradient":
        leaves = [t.detach().requires_grad_() for t in s["f"]]
        J = binding.objective_after(g, *leaves, s["steps"], checkpoint_every=s["every"])
        J.backward()
        return [J.detach()] + [t.grad for t in leaves]
    if kind == "lines":
        a = g.chebyshev_lines(s["x"], 0)
        return [a, g.chebyshev_lines(a, 1)]
    if kind == "transform":
        a = g.transform_forward(s["f"])
        return [a, g.transform_backward(a)]
    return [g.diagnostics()] + list(g.get_fields())


# ---- what a pass cannot do without ------------------------------------------------------------
def _fft(n):
    return 5.0 * n * math.log2(n)


def _step_work(nx, ny, nz):
    """One time step: the state and its history in and out (float64 complex, three fields each);
    the padded transforms, the products, the assembly and the wall-normal solves."""
    mx, px, py, n = nx // 2, 3 * nx // 2, 3 * ny // 2, nz - 1
    modes = float(mx * ny * nz)
    flops = (12 * mx * ny * _fft(n) + 13 * mx * nz * _fft(py) + 8 * py * nz * _fft(px)
             + 45.0 * px * py * nz + 280.0 * modes)
    return 12 * 16 * modes, flops


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        w = [_step_work(m["nx"], m["ny"], m["nz"]) for m in members(case)]
        return dict(bytes=case["steps"] * sum(b for b, _ in w),
                    flops=case["steps"] * sum(f for _, f in w))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n, mx = float(nx * ny * nz), nx // 2
    one = mx * ny * _fft(nz - 1) + mx * nz * _fft(ny) + 0.5 * ny * nz * _fft(nx)   # one transform
    if kind == "lines":
        lines = case["fields"] * mx * ny
        return dict(bytes=2 * 2 * 16.0 * lines * nz, flops=2 * lines * _fft(nz - 1))
    if kind in ("noalloc", "transform"):
        k = 1 if kind == "noalloc" else 2
        return dict(bytes=k * 16 * n, flops=k * one)
    if kind == "monitor":
        return dict(bytes=24 * n + 32 * n, flops=11 * one + 40 * n)
    b, f = _step_work(nx, ny, nz)
    steps = case["steps"]
    if kind == "step":
        return dict(bytes=steps * b, flops=steps * f)
    if kind == "run":
        return dict(bytes=steps * b + 64 * n, flops=steps * f + 8 * one)
    # gradient: the forward run, its recomputation and a reverse sweep of twice the work
    return dict(bytes=4 * steps * b + 64 * n, flops=4 * steps * f + 8 * one)


# ---- the same results in plain float64 torch ----------------------------------------------------
class _Channel:
    """The discrete step in plain torch: dense Chebyshev matrices, torch.fft, dense tau solves in
    the Gottlieb-Orszag form.  State arrays are (nx / 2, ny, nz) coefficients."""

    def __init__(self, nx, ny, nz, re_tau, we, ch, pe, dt, gx=1.0):
        f64 = dict(dtype=torch.float64, device=DEV)
        self.nx, self.ny, self.nz, self.N = nx, ny, nz, nz - 1
        self.re, self.ch, self.pe, self.dt, self.gx = re_tau, ch, pe, dt, gx
        self.beta, self.lam = 2 * re_tau / dt, math.sqrt(pe / (ch * ch * dt))
        self.shat, self.kappa = 2 * self.lam * ch * ch, 3 / math.sqrt(8.0) * ch / we
        N, mx = self.N, nx // 2
        n = np.arange(N + 1)
        ang = np.cos(np.pi * ((np.outer(n, n)) % (2 * N)) / N)
        cb = np.where((n == 0) | (n == N), 2.0, 1.0)
        self.B = torch.tensor(ang, **f64)                                      # a -> samples
        self.F = torch.tensor(2.0 / N * ang / cb[:, None] / cb[None, :], **f64)
        D = np.zeros((N + 1, N + 1))
        G = np.zeros((N + 1, N + 1))
        for i in range(N + 1):
            D[i, i + 1::2] = 2.0 * n[i + 1::2] / (2.0 if i == 0 else 1.0)
            if i >= 2:
                G[i, i - 2] = (2.0 if i == 2 else 1.0) / (4.0 * i * (i - 1))
                if i <= N - 2:
                    G[i, i] = -1.0 / (2.0 * (i * i - 1.0))
                if i + 2 <= N - 2:
                    G[i, i + 2] = 1.0 / (4.0 * i * (i + 1))
        self.D, self.G = torch.tensor(D, **f64), torch.tensor(G, **f64)
        sg = (-1.0) ** n
        self.dirichlet = torch.tensor(np.stack([np.ones(N + 1), sg]), **f64)
        self.neumann = torch.tensor(np.stack([1.0 * n * n, -sg * n * n]), **f64)
        j = np.arange(ny)
        my = np.where(j < ny // 2, j, j - ny)
        self.kx = torch.tensor(2 * np.pi * np.arange(mx) / LX, **f64)[:, None, None]
        self.ky = torch.tensor(2 * np.pi * my / LY, **f64)[None, :, None]
        self.k2 = self.kx ** 2 + self.ky ** 2
        keep = torch.ones((mx, ny, 1), **f64)
        keep[:, ny // 2] = 0.0
        self.keep = keep
        mean = torch.zeros((mx, ny, 1), **f64)
        mean[0, 0] = 1.0
        self.mean = mean

    def forward(self, f):
        """Physical (nz, py, px) samples -> coefficients of the kept modes."""
        nz, py, px = f.shape
        c = torch.fft.fft(torch.fft.rfft(f, dim=2)[..., :self.nx // 2], dim=1) / (px * py)
        h = self.ny // 2
        c = torch.cat([c[:, :h], torch.zeros_like(c[:, :1]), c[:, py - h + 1:]], dim=1)
        return self.along_z(self.F, c.permute(2, 1, 0))

    def backward(self, a, padded=False):
        k = 3 if padded else 2
        py, px, h = k * self.ny // 2, k * self.nx // 2, self.ny // 2
        a = self.along_z(self.B, a)
        gap = torch.zeros((a.shape[0], py - 2 * h + 1, a.shape[2]), dtype=a.dtype, device=DEV)
        a = torch.cat([a[:, :h], gap, a[:, h + 1:]], dim=1)
        c = torch.fft.ifft(a, dim=1) * py
        first = c[:1].real.to(c.dtype)
        c = torch.cat([first, c[1:]], dim=0).permute(2, 1, 0)
        return torch.fft.irfft(c, n=px, dim=2) * px

    @staticmethod
    def along_z(M, a):
        return torch.complex(a.real @ M.T, a.imag @ M.T)

    def dz(self, a):
        return self.along_z(self.D, a)

    def set_fields(self, u, v, w, phi):
        uh, vh, wh, ph = (self.forward(f) for f in (u, v, w, phi))
        om = 1j * self.kx * vh - 1j * self.ky * uh
        flow = torch.complex(uh.real, vh.real)
        om = om * (1 - self.mean) + flow * self.mean
        return om, wh * (1 - self.mean), ph

    def velocity(self, om, w):
        dw, safe = self.dz(w), self.k2 + self.mean
        u = (1j * self.kx * dw + 1j * self.ky * om) / safe
        v = (1j * self.ky * dw - 1j * self.kx * om) / safe
        real, imag = om.real.to(om.dtype), om.imag.to(om.dtype)
        return u * (1 - self.mean) + real * self.mean, v * (1 - self.mean) + imag * self.mean

    def get_fields(self, s):
        u, v = self.velocity(s[0], s[1])
        return [self.backward(a) for a in (u, v, s[1], s[2])]

    def terms(self, om, w, ph):
        u, v = self.velocity(om, w)
        ikx, iky, k2 = 1j * self.kx, 1j * self.ky, self.k2
        U, V, W, f, fx, fy, fz = (self.backward(a, True)
                                  for a in (u, v, w, ph, ikx * ph, iky * ph, self.dz(ph)))
        k, fwd = self.kappa, self.forward
        sxx, syy = fwd(W * W - U * U + k * (fz * fz - fx * fx)), fwd(W * W - V * V + k * (fz * fz - fy * fy))
        sxy, sxz, syz = (fwd(-(a * b + k * c * d)) for a, b, c, d in
                         ((U, V, fx, fy), (U, W, fx, fz), (V, W, fy, fz)))
        p3, fu, fv, fw = (fwd(f * q) for q in (f * f, U, V, W))
        sx = ikx * sxx + iky * sxy + self.dz(sxz)
        sy = ikx * sxy + iky * syy + self.dz(syz)
        sz = ikx * sxz + iky * syz
        e0 = torch.zeros(self.nz, dtype=torch.float64, device=DEV)
        e0[0] = self.gx
        h_om = (ikx * sy - iky * sx) * (1 - self.mean) + torch.complex(sx.real + e0, sy.real) * self.mean
        h_w = (-k2 * sz - self.dz(ikx * sx + iky * sy)) * (1 - self.mean)
        g = p3 - (1 + self.shat) * ph
        s_phi = -(ikx * fu + iky * fv + self.dz(fw)) + (self.dz(self.dz(g)) - k2 * g) / self.pe
        return h_om, h_w, s_phi

    def solve(self, shift, rhs, rows, walls=None):
        """(D^2 - k^2 - shift) a = rhs with the two wall rows (homogeneous unless `walls` gives the
        wall values and no rhs), chunk by chunk of kx; rhs: list of complex arrays."""
        out, h = [], self.ny // 2
        step = max(1, int(1e9 / ((h + 1) * self.nz ** 2 * 8)))
        eye = torch.eye(self.nz, dtype=torch.float64, device=DEV)
        for m0 in range(0, self.nx // 2, step):
            k2 = self.k2[m0:m0 + step, :h + 1, 0]
            M = eye - (k2 + shift)[..., None, None] * self.G
            M = torch.cat([rows.expand(M.shape[:-2] + rows.shape), M[..., 2:, :]], dim=-2)
            if rhs is None:
                b = torch.zeros(k2.shape + (self.nz, 2), dtype=torch.float64, device=DEV)
                b[..., 0, 0] = 1.0
                b[..., 1, 1] = 1.0
                out.append(torch.linalg.solve(M, b))
                continue
            cols = []
            for r in rhs:
                r = self.along_z(self.G, r[m0:m0 + step])
                low = torch.cat([torch.zeros_like(r[..., :2]), r[..., 2:]], dim=-1)
                up = torch.cat([low[:, :1], low[:, h:].flip(1)], dim=1)      # the modes -my
                for q in (low[:, :h + 1], up):
                    cols += [q.real, q.imag]
            x = torch.linalg.solve(M, torch.stack(cols, dim=-1))
            got = []
            for i in range(len(rhs)):
                a, b, c, d = (x[..., 4 * i + q] for q in range(4))
                lo, up = torch.complex(a, b), torch.complex(c, d)
                got.append(torch.cat([lo[:, :h], up[:, 1:].flip(1)], dim=1))
            out.append(got)
        if rhs is None:
            return torch.cat(out)
        return [torch.cat([o[i] for o in out]) * self.keep for i in range(len(rhs))]

    def influence(self):
        """Homogeneous w solutions for unit wall values of lap w, on the |my| lines, spread to all."""
        th = self.solve(self.beta, None, self.dirichlet)                 # (mx, h + 1, nz, 2)
        h = self.ny // 2
        th = torch.cat([th[:, :h], th[:, 1:h + 1].flip(1)], dim=1)
        z = torch.zeros_like(th[..., 0])
        pairs = [torch.complex(th[..., i], z) for i in range(2)]
        return [p.real for p in self.solve(0.0, pairs, self.dirichlet)]

    def step(self, s, hist):
        om, w, ph = s
        h = self.terms(om, w, ph)
        H = h if hist is None else tuple(1.5 * a - 0.5 * b for a, b in zip(h, hist))
        lap = lambda a: self.dz(self.dz(a)) - self.k2 * a
        th = lap(w)
        r_om = -(lap(om) + self.beta * om) - 2 * self.re * H[0]
        r_th = -(lap(th) + self.beta * th) - 2 * self.re * H[1]
        r_ps = (self.pe / self.ch ** 2) * (ph / self.dt + H[2])
        om2, tp = self.solve(self.beta, [r_om, r_th], self.dirichlet)
        wp = self.solve(0.0, [tp], self.dirichlet)[0]
        if not hasattr(self, "wh"):
            self.wh = self.influence()
        a, b = self.wh
        top, bot = self.neumann[0], self.neumann[1]
        d = lambda v: (v @ top.to(v.dtype), v @ bot.to(v.dtype))
        (at, ab), (bt, bb), (pt, pb) = d(a), d(b), d(wp)
        det = at * bb - bt * ab
        det = torch.where(det == 0, torch.ones_like(det), det)
        ca, cb = -(pt * bb - pb * bt) / det, -(pb * at - pt * ab) / det
        w2 = (wp + ca[..., None] * a + cb[..., None] * b) * (1 - self.mean) * self.keep
        ps = self.solve(self.lam, [r_ps], self.neumann)[0]
        ph2 = self.solve(self.lam, [ps], self.neumann)[0]
        return (om2, w2, ph2), h

    def objective(self, s):
        """1/2 int |u|^2 + int |grad phi|^2, exact for the interpolants."""
        u, v = self.velocity(s[0], s[1])
        n = np.arange(self.nz)
        q = lambda k: np.where(k % 2 == 0, 2.0 / (1.0 - 1.0 * k * k + (k % 2)), 0.0)
        gram = torch.tensor(0.5 * (q(n[:, None] + n) + q(abs(n[:, None] - n))), dtype=torch.float64,
                            device=DEV)
        weight = torch.full_like(self.kx, 2.0)
        weight[0] = 1.0
        energy = lambda a: (weight * (a.real * (a.real @ gram) + a.imag * (a.imag @ gram))).sum()
        ph = s[2]
        grad = energy(1j * self.kx * ph) + energy(1j * self.ky * ph) + energy(self.dz(ph))
        return LX * LY * (0.5 * (energy(u) + energy(v) + energy(s[1])) + grad)


def _advance(c, f, steps):
    s, hist = c.set_fields(*f), None
    for _ in range(steps):
        s, hist = c.step(s, hist)
    return s


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        out = []
        for m, f in zip(members(case), _member_fields(case, seed)):
            c = _Channel(m["nx"], m["ny"], m["nz"], **_physics(case))
            out += list(_advance(c, f, case["steps"]))
        return out
    if kind in ("step", "run", "gradient") and case["nx"] * case["ny"] * case["nz"] > 6e6:
        return None              # dense solves of a large channel take minutes
    phys = _physics(case) if "dt" in case else dict(re_tau=1.0, we=1.0, ch=1.0, pe=1.0, dt=1.0)
    c = _Channel(case["nx"], case["ny"], case["nz"], **phys)
    if kind == "noalloc":
        return _unfiltered(c, _field(case, seed))
    if kind == "lines":
        x = _lines(case, seed)
        return [c.along_z(c.F, x), x]
    if kind == "transform":
        f = _field(case, seed)
        a = _unfiltered(c, f)
        return [a, c.backward(a)]
    f = _fields(case, seed)
    if kind == "step":
        return list(_advance(c, f, case["steps"]))
    if kind == "run":
        return c.get_fields(_advance(c, f, case["steps"]))
    if kind == "monitor":
        return [None] + c.get_fields(c.set_fields(*f))
    leaves = [t.requires_grad_() for t in f]
    with torch.enable_grad():
        J = c.objective(_advance(c, leaves, case["steps"]))
        J.backward()
    return [J.detach()] + [t.grad for t in leaves]


def _unfiltered(c, f):
    """The analysis transform: as the step's, on the unpadded grid (Nyquist modes dropped)."""
    return c.forward(f)
