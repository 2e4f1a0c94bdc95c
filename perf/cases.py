"""Performance cases: the work that programs built on this package have it do.

Each case builds a solver through the package's public classes, puts a seeded
flow into it, and then advances it (or inverts, differentiates, finds the
eigenvalues of) the problem and reads the whole result.  Time-stepping cases
advance a fixed number of steps per pass from the state the previous pass
left, as a simulation does between two analysis outputs, and copy every field
of the state to the caller's device buffers.

Results of the FP64 form are returned as FP64.  The mixed form transforms and
multiplies in FP32, so its results are returned in FP32.

``exact`` computes the same discretization (Chebyshev tau in the T-to-U form,
3/2-dealiased products, IMEX Runge-Kutta or SBDF) with dense matrices in
64 bits, in torch alone.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1905_10388_gb300 import _lib as L
from paper_1905_10388_gb300.adjoint import RBAdjoint
from paper_1905_10388_gb300.solver import (CFL, Context, FisherKPPSolver, QGInversion, RB3DSolver, RBOnsetEVP,
                                           RBSolver, step_batched)

VARS2 = ("b", "p", "u", "w", "bz", "uz", "wz")
VARS3 = ("b", "p", "u", "v", "w", "bz", "uz", "vz", "wz")
STRAT = "1.688,0.750,0.063"             # Chebyshev coefficients of about 1 + z + z^2/2 on [0, 1]


# --- the cases -----------------------------------------------------------------

def listed():
    return [
        # the small 2D run of the parity tests: latency and launches count
        _rb2d("rb2d_64x32_rk222_fp64", 64, 32, 1e6, "RK222", "fp64", 1e-3, 16),
        # the headline 2D run, in both precisions
        _rb2d("rb2d_512x256_sbdf2_fp64", 512, 256, 1e8, "SBDF2", "fp64", 1e-4, 16),
        _rb2d("rb2d_512x256_sbdf2_mixed", 512, 256, 1e8, "SBDF2", "mixed", 1e-4, 16),
        # a 3D production run (the largest case) and a small 3D one in FP64
        _rb3d("rb3d_128x128x64_rk222_mixed", 128, 128, 64, 1e7, "RK222", "mixed", 5e-4, 4),
        _rb3d("rb3d_32x64x32_rk222_fp64", 32, 64, 32, 1e6, "RK222", "fp64", 1e-3, 4),
        # a parameter sweep: 16 uneven 2D problems stepped together
        dict(name="sweep16_rk222_mixed", kind="batch", count=16, spread=7, scheme="RK222", prec="mixed", steps=4),
        # reaction-diffusion in a wide channel: two variables, a thousand long pencils
        dict(name="fisher_2048x1024_rk222_mixed", kind="fisher", nx=2048, nz=1024, scheme="RK222", prec="mixed",
             dt=1e-3, steps=4, num=3, den=2),
        # the printed example's size, FP64
        dict(name="fisher_128x64_rk222_fp64", kind="fisher", nx=128, nz=64, scheme="RK222", prec="fp64", dt=0.01,
             steps=16, num=3, den=2),
        # optimisation of an initial condition: loss and gradient through 20 steps
        dict(name="adjoint_256x128_rk222_mixed", kind="adjoint", nx=256, nz=128, ra=1e6, scheme="RK222",
             prec="mixed", dt=1e-3, steps=20, checkpoint=10),
        # a run under step-size control: the flow's speed on the grid before every
        # step, a new factorization when the step changes
        dict(name="cfl_256x128_rk222_mixed", kind="cfl", nx=256, nz=128, ra=1e7, scheme="RK222", prec="mixed",
             dt=5e-4, steps=8),
        # stability of the conductive state: growth rate in every pencil
        dict(name="onset_256x64_evp", kind="evp", nx=256, nz=64, ra=1708.0, iters=40),
        # potential-vorticity inversion on host data, as inside an outer host program
        dict(name="qg_512x256_inversion", kind="qg", nx=512, nz=256, strat=STRAT),
    ]


def _rb2d(name, nx, nz, ra, scheme, prec, dt, steps, num=3, den=2):
    c = dict(kind="rb2d", nx=nx, nz=nz, ra=ra, scheme=scheme, prec=prec, dt=dt, steps=steps, num=num, den=den)
    return dict(c, name=name) if name else c


def _rb3d(name, nx, ny, nz, ra, scheme, prec, dt, steps):
    c = dict(kind="rb3d", nx=nx, ny=ny, nz=nz, ra=ra, scheme=scheme, prec=prec, dt=dt, steps=steps)
    return dict(c, name=name) if name else c


def draw(rng):
    def pow2(lo, hi):
        return 2 ** rng.randint(lo, hi)

    kind = rng.choice(["rb2d", "rb2d", "rb2d", "rb2d", "rb3d", "rb3d", "batch", "fisher", "fisher", "adjoint",
                       "cfl", "evp", "qg"])
    prec = rng.choice(["fp64", "mixed"])
    ra = round(10.0 ** rng.uniform(5.0, 8.0), 1)
    if kind == "rb2d":
        scheme = rng.choice(["RK222", "RK222", "SBDF2", "SBDF2", "RK443", "SBDF3", "SBDF1"])
        steps = rng.randint(2, 16)
        if rng.random() < 0.3:           # three times a power of two, on grids 4/3 or 2 times as fine
            num, den = rng.choice([(4, 3), (2, 1)])
            nx, nz = 3 * pow2(4, 7), 3 * pow2(3, 6)
        else:
            num, den = 3, 2
            nx, nz = pow2(5, 9 if prec == "fp64" else 10), pow2(4, 8)
        return _rb2d(None, nx, nz, ra, scheme, prec, round(1e-3 * 32.0 / nz, 9), steps, num, den)
    if kind == "rb3d":
        return _rb3d(None, pow2(4, 7), pow2(4, 6), pow2(4, 6), ra, rng.choice(["RK222", "SBDF2"]), prec,
                     round(5e-4 * rng.uniform(0.5, 1.0), 9), rng.randint(2, 4))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 24), spread=rng.randint(1, 999),
                    scheme=rng.choice(["RK222", "SBDF2"]), prec=prec, steps=rng.randint(2, 6))
    if kind == "fisher":
        return dict(kind="fisher", nx=pow2(5, 11), nz=pow2(4, 10), scheme=rng.choice(["RK222", "SBDF2", "RK443"]),
                    prec=prec, dt=round(10.0 ** rng.uniform(-3.0, -2.0), 6), steps=rng.randint(2, 8), num=3, den=2)
    if kind == "adjoint":
        return dict(kind="adjoint", nx=pow2(5, 8), nz=pow2(4, 7), ra=round(10.0 ** rng.uniform(5.0, 6.0), 1),
                    scheme=rng.choice(["RK222", "RK111"]), prec=prec, dt=1e-3, steps=rng.randint(4, 20),
                    checkpoint=rng.randint(3, 10))
    if kind == "cfl":
        return dict(kind="cfl", nx=pow2(5, 9), nz=pow2(4, 7), ra=ra, scheme=rng.choice(["RK222", "RK443"]),
                    prec=prec, dt=round(10.0 ** rng.uniform(-4.0, -3.3), 7), steps=rng.randint(2, 8))
    if kind == "evp":
        return dict(kind="evp", nx=pow2(5, 9), nz=pow2(4, 7), ra=round(rng.uniform(1500.0, 4000.0), 1),
                    iters=rng.randint(20, 60))
    return dict(kind="qg", nx=pow2(5, 10), nz=pow2(4, 9),
                strat="%.3f,%.3f,%.3f" % (rng.uniform(1.2, 2.0), rng.uniform(0.1, 0.5), rng.uniform(0.02, 0.2)))


# --- seeded inputs ---------------------------------------------------------------

def _smooth(rng, nz, *nh):
    """A smooth random field vanishing at both walls, O(0.1): a few sine modes in
    z whose horizontal structure is noise with a decaying spectrum."""
    z = (1.0 - np.cos(np.pi * (np.arange(nz) + 0.5) / nz)) / 2.0
    modes = min(8, nz // 2)
    f = 0.0
    for m in range(1, modes + 1):
        g = np.fft.rfftn(rng.standard_normal(nh))
        ks = np.meshgrid(*([np.abs(np.fft.fftfreq(n, 1.0 / n)) for n in nh[:-1]] + [np.arange(nh[-1] // 2 + 1)]),
                         indexing="ij")
        g = g / (1.0 + sum(k * k for k in ks))
        g = np.fft.irfftn(g, nh)
        g = g / max(np.abs(g).max(), 1e-30)
        f = f + np.sin(m * np.pi * z).reshape((nz,) + (1,) * len(nh)) * g / (m * m)
    return 0.1 * f


def _flow(seed, nz, *nh):
    """Grid values of the initial state: the buoyancy's noise and the velocities."""
    rng = np.random.default_rng(seed)
    names = ("u", "w") if len(nh) == 1 else ("u", "v", "w")
    return rng.standard_normal((nz,) + nh), {v: _smooth(rng, nz, *nh) for v in names}


def _sweep(case):
    """Sizes, Rayleigh numbers and steps of a sweep's problems."""
    rng = np.random.default_rng(case["spread"])
    n = case["count"]
    nx, nz = rng.choice([64, 128, 256, 512], size=n), rng.choice([32, 64, 128, 256], size=n)
    ra = 10.0 ** rng.uniform(5.0, 8.0, size=n)
    return [_rb2d(None, int(nx[i]), int(nz[i]), float(ra[i]), case["scheme"], case["prec"],
                  1e-3 * 32.0 / float(nz[i]), case["steps"]) for i in range(n)]


# --- what a program has in hand ---------------------------------------------------

def _rb_solver(ctx, c, seed):
    d = (c.get("num", 3), c.get("den", 2))
    nh = (c["nx"],) if c["kind"] != "rb3d" else (c["ny"], c["nx"])
    if c["kind"] == "rb3d":
        s = RB3DSolver(ctx, c["nx"], c["ny"], c["nz"], c["ra"], scheme=c["scheme"], precision=c["prec"])
    else:
        s = RBSolver(ctx, c["nx"], c["nz"], c["ra"], scheme=c["scheme"], precision=c["prec"], dealias=d)
    s.factor(c["dt"])
    noise, vel = _flow(seed, c["nz"], *nh)
    s.set_initial_state(noise, amplitude=1e-2)
    for v, g in vel.items():
        s.set_field(v, g, layout="g")
        s.dz(v, v + "z")
    return s


def _buffers(s):
    return torch.empty((s.S, s.P, s.Nz), dtype=torch.complex128, device="cuda")


def _read(s, out):
    """Every field's coefficients into the caller's device buffer."""
    h = s.ctx.handle
    for i, v in enumerate(s.state_order):
        L.check(h, L.lib().sp_get_field(h, s.pid, s.var[v], ctypes.c_void_p(out[i].data_ptr()), 1, b"c"))
    r = out if s.precision == "fp64" else out.to(torch.complex64)
    return {v: r[i] for i, v in enumerate(s.state_order)}


def prepare(case, seed):
    kind = case["kind"]
    ctx = Context(0)
    st = {"case": case, "ctx": ctx}
    if kind in ("rb2d", "rb3d", "cfl"):
        st["s"] = s = _rb_solver(ctx, case, seed)
        st["out"] = _buffers(s)
        if kind == "cfl":
            st["cfl"] = CFL(s, (("u", "x"), ("w", "z")), initial_dt=case["dt"], **_cfl_rule(case))
    elif kind == "batch":
        st["s"] = [_rb_solver(ctx, c, seed + 1000 * i) for i, c in enumerate(_sweep(case))]
        st["out"] = [_buffers(s) for s in st["s"]]
    elif kind == "fisher":
        s = FisherKPPSolver(ctx, case["nx"], case["nz"], scheme=case["scheme"], precision=case["prec"],
                            dealias=(case["num"], case["den"]))
        s.factor(case["dt"])
        s.set_initial_state(_fisher_u(case, seed))
        st["s"], st["out"] = s, _buffers(s)
    elif kind == "adjoint":
        noise, target, q = _adjoint_inputs(case, seed)
        s = RBSolver(ctx, case["nx"], case["nz"], case["ra"], scheme=case["scheme"], precision=case["prec"])
        s.factor(case["dt"])
        st["s"], st["q"] = s, q
        st["adj"] = RBAdjoint(s, noise, target, amplitude=1e-2, checkpoint=case["checkpoint"])
    elif kind == "evp":
        st["s"] = s = RBOnsetEVP(ctx, case["nx"], case["nz"], case["ra"])
        rng = np.random.default_rng(seed)
        st["x0"] = 1.0 + 0.1 * rng.standard_normal((s.P, s.assembly["n"])) + 0j
    elif kind == "qg":
        st["s"] = QGInversion(ctx, case["nx"], case["nz"], _profile(case))
        st["q"] = _qg_q(case, seed)
    return st


def run(state):
    kind = state["case"]["kind"]
    if kind in ("rb2d", "rb3d", "fisher"):
        s = state["s"]
        s.step(state["case"]["steps"], graph=True)
        return _read(s, state["out"])
    if kind == "cfl":
        state["cfl"].step(state["case"]["steps"])
        return _read(state["s"], state["out"])
    if kind == "batch":
        step_batched(state["s"], state["case"]["steps"])
        return [_stack(_read(s, o)) for s, o in zip(state["s"], state["out"])]
    if kind == "adjoint":
        loss, grad = state["adj"].loss_and_grad(state["q"], state["case"]["steps"])
        if state["case"]["prec"] == "mixed":
            grad = grad.to(torch.float32)
            loss = np.float32(loss)
        return {"loss": loss, "grad": grad}
    if kind == "evp":
        return {"growth": state["s"].growth_rates(0.0, state["case"]["iters"], state["x0"])}
    psi, psiz = state["s"].invert(state["q"])
    return {"psi": psi, "psiz": psiz}


def _stack(fields):
    return torch.stack([fields[v] for v in VARS2])


def _cfl_rule(case):
    return dict(safety=0.4, min_dt=1e-6, max_dt=4e-3, min_change=0.5, max_change=1.5, threshold=0.1)


def _fisher_u(case, seed):
    return np.random.default_rng(seed).random((case["nz"], case["nx"]))


def _adjoint_inputs(case, seed):
    rng = np.random.default_rng(seed)
    nz, nx = case["nz"], case["nx"]
    z = _nodes(nz)[:, None]
    noise = rng.standard_normal((nz, nx))
    target = 1.0 - z + 0.05 * _smooth(rng, nz, nx)
    return noise, target, 0.5 * _smooth(rng, nz, nx)


def _profile(case):
    return [float(t) for t in case["strat"].split(",")]


def _qg_q(case, seed):
    rng = np.random.default_rng(seed)
    p, nz = case["nx"] // 2, case["nz"]
    decay = 1.0 / ((1.0 + np.arange(p))[:, None] * (1.0 + np.arange(nz))[None, :])
    q = (rng.standard_normal((p, nz)) + 1j * rng.standard_normal((p, nz))) * decay
    q[0] = q[0].real
    return q


# --- what a pass cannot do without -------------------------------------------------

_STAGES = {"RK111": 1, "RK222": 2, "RK443": 4}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [work(c) for c in _sweep(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    nx, nz, ny = case["nx"], case["nz"], case.get("ny", 1)
    pencils = ny * nx // 2
    if kind == "evp":
        s, solves, fields, eqs = 7, case["iters"], 0, 0
    elif kind == "qg":
        s, solves, fields, eqs = 2, 1, 0, 0
    elif kind == "fisher":
        s, solves, fields, eqs = 2, case["steps"] * _STAGES.get(case["scheme"], 1), 1, 1
    else:
        s, fields, eqs = (7, 8, 3) if ny == 1 else (9, 15, 4)
        solves = case["steps"] * _STAGES.get(case["scheme"], 1)
        if kind == "adjoint":            # forward, replay, and the transposed solves and products
            solves *= 3
    n = s * nz
    state = pencils * n * 16
    # every solve reads the pencils' factors (about ten nonzeros a row), the state and the
    # right-hand side, and writes the state; each step's products read the state once more
    nbytes = solves * (pencils * n * 10 * 8 + 3 * state)
    flops = solves * pencils * n * 2 * 2 * 10
    g = 1.5
    pts = g * nz * (g * nx) * (g * ny if ny > 1 else 1)
    flops += solves * (fields + eqs) * 2.5 * pts * math.log2(max(2.0, pts)) if fields else 0
    return {"bytes": float(nbytes), "flops": float(flops)}


# --- 64-bit reference ---------------------------------------------------------------

def _nodes(n):
    return (1.0 - np.cos(np.pi * (np.arange(n) + 0.5) / n)) / 2.0


def _tableau(scheme):
    """Implicit and explicit weights of the ARS schemes, stage i from stages j."""
    if scheme == "RK111":
        return [[0, 0], [0, 1]], [[0, 0], [1, 0]]
    if scheme == "RK222":
        g = 1.0 - 1.0 / math.sqrt(2.0)
        d = 1.0 - 1.0 / (2.0 * g)
        return [[0, 0, 0], [0, g, 0], [0, 1 - g, g]], [[0, 0, 0], [g, 0, 0], [d, 1 - d, 0]]
    h = [[0] * 5, [0, 1 / 2, 0, 0, 0], [0, 1 / 6, 1 / 2, 0, 0], [0, -1 / 2, 1 / 2, 1 / 2, 0],
         [0, 3 / 2, -3 / 2, 1 / 2, 1 / 2]]
    a = [[0] * 5, [1 / 2, 0, 0, 0, 0], [11 / 18, 1 / 18, 0, 0, 0], [5 / 6, -5 / 6, 1 / 2, 0, 0],
         [1 / 4, 7 / 4, 3 / 4, -7 / 4, 0]]
    return h, a


_SBDF = {1: ([1, -1], [1]), 2: ([3 / 2, -2, 1 / 2], [2, -1]), 3: ([11 / 6, -3, 3 / 2, -1 / 3], [3, -3, 1])}


class _Reference:
    """M dX/dt + L X = F(X) pencil by pencil with dense matrices; unknowns
    [variable][mode], u and v carried as i times a real-coefficient variable so
    that every pencil matrix is real."""

    def __init__(self, names, nx, nz, scale, lx, ny=None, ly=None):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.names, self.S, self.N = names, len(names), nz
        self.nx, self.ny, self.K = nx, ny, nx // 2
        self.scale = scale
        f8 = dict(dtype=torch.float64, device=self.dev)
        kx = 2 * np.pi * np.arange(self.K) / lx
        if ny:
            iy = np.arange(ny)
            ky = 2 * np.pi * np.where(iy < ny // 2, iy, iy - ny) / ly
            kx, ky = np.tile(kx, ny), np.repeat(ky, self.K)
        else:
            ky = np.zeros_like(kx)
        self.kx, self.ky = torch.tensor(kx, **f8), torch.tensor(ky, **f8)
        self.P = len(kx)
        n = torch.arange(nz, **f8)
        self.U = torch.diag(torch.where(n == 0, 1.0, 0.5)) - torch.diag(torch.full((nz - 2,), 0.5, **f8), 2)
        self.D = torch.diag(2.0 * n[1:], 1)                      # T to U: dz T_n = 2 n U_{n-1} on [0, 1]
        self.I = torch.eye(nz, **f8)
        self.left = torch.where(torch.arange(nz, device=self.dev) % 2 == 0, 1.0, -1.0).to(torch.float64)
        self.right = torch.ones(nz, **f8)
        self.rows = []                                           # (M blocks, L blocks, right-hand side)
        self.zero = (self.kx == 0) & (self.ky == 0)

    def equation(self, name, M, Lh, differential, phase=0):
        self.rows.append(("eq", name, M, Lh, differential, phase))

    def boundary(self, alternatives):
        """alternatives: (variable, side, value, pencil mask)"""
        self.rows.append(("bc", alternatives))

    def assemble(self):
        f8 = dict(dtype=torch.float64, device=self.dev)
        N, n = self.N, self.S * self.N
        self.M, self.L = torch.zeros((self.P, n, n), **f8), torch.zeros((self.P, n, n), **f8)
        self.g = torch.zeros((self.P, n), **f8)
        self.place = {}
        r = 0
        col = {v: i * N for i, v in enumerate(self.names)}
        for row in self.rows:
            if row[0] == "eq":
                _, name, M, Lh, diff, phase = row
                m = N - 1 if diff else N
                for target, terms in ((self.M, M), (self.L, Lh)):
                    for v, op, c in terms:
                        B = self.D if op == "dz" else op if isinstance(op, torch.Tensor) else (
                            self.U if diff else self.I)
                        c = c if isinstance(c, torch.Tensor) else torch.full((self.P,), float(c), **f8)
                        target[:, r:r + m, col[v]:col[v] + N] += c[:, None, None] * B[:m]
                self.place[name] = (r, m, diff, phase)
                r += m
            else:
                for v, side, value, mask in row[1]:
                    e = self.left if side == "left" else self.right
                    self.L[:, r, col[v]:col[v] + N] += mask.to(torch.float64)[:, None] * e
                    self.g[:, r] += mask.to(torch.float64) * value
                r += 1
        assert r == n
        self.lu = {}

    def solve(self, alpha, beta, rhs):
        """rhs, result: complex [P, n]"""
        key = (alpha, beta)
        if key not in self.lu:
            if len(self.lu) >= 4:
                self.lu.pop(next(iter(self.lu)))
            self.lu[key] = torch.linalg.lu_factor(alpha * self.M + beta * self.L)
        b = torch.view_as_real(rhs)
        return torch.view_as_complex(torch.linalg.lu_solve(*self.lu[key], b).contiguous())

    # -- transforms: coefficients [P, N] <-> grid [z][y][x] ------------------------------
    def cheb(self, ng):
        i = torch.arange(ng, dtype=torch.float64, device=self.dev)
        n = torch.arange(self.N, dtype=torch.float64, device=self.dev)
        return torch.cos(n[None, :] * (math.pi * (ng - 0.5 - i) / ng)[:, None])     # T_n(x_i), ascending x

    def sizes(self, scale):
        g = lambda n: n * scale[0] // scale[1]  # noqa: E731
        return g(self.N), g(self.ny) if self.ny else None, g(self.nx)

    def to_grid(self, c, scale):
        ngz, ngy, ngx = self.sizes(scale)
        f = torch.einsum("zn,pn->zp", self.cheb(ngz).to(torch.complex128), c)
        if self.ny:
            f = f.reshape(ngz, self.ny, self.K)
            h = self.ny // 2
            z = torch.zeros((ngz, ngy, self.K), dtype=f.dtype, device=self.dev)
            z[:, :h] = f[:, :h]
            z[:, ngy - h + 1:] = f[:, h + 1:]
            f = torch.fft.ifft(z, dim=1) * ngy
        return torch.fft.irfft(f, ngx, dim=-1) * ngx

    def to_coef(self, g):
        ngz, ngx = g.shape[0], g.shape[-1]
        f = (torch.fft.rfft(g, dim=-1) / ngx)[..., :self.K]
        if self.ny:
            ngy = g.shape[1]
            f = torch.fft.fft(f, dim=1) / ngy
            h = self.ny // 2
            z = torch.zeros((ngz, self.ny, self.K), dtype=f.dtype, device=self.dev)
            z[:, :h] = f[:, :h]
            z[:, h + 1:] = f[:, ngy - h + 1:]
            f = z.reshape(ngz, self.P)
        w = torch.full((self.N,), 2.0 / ngz, dtype=torch.float64, device=self.dev)
        w[0] = 1.0 / ngz
        c = torch.einsum("zn,zp->pn", (self.cheb(ngz) * w).to(torch.complex128), f)
        if not self.ny:
            c = torch.cat([c[:1].real.to(c.dtype), c[1:]])
        return c

    def dz(self, c):
        out = [torch.zeros_like(c[:, 0]) for _ in range(self.N + 2)]
        for m in range(self.N - 2, -1, -1):
            out[m] = out[m + 2] + 2.0 * (m + 1) * c[:, m + 1]
        d = torch.stack(out[:self.N], 1) * 2.0
        return torch.cat([d[:, :1] * 0.5, d[:, 1:]], 1)

    # -- stepping --------------------------------------------------------------------------
    def pack(self, X):
        ph = {"u": -1j, "uz": -1j, "v": -1j, "vz": -1j} if self.S > 2 else {}
        return torch.cat([X[v] * ph.get(v, 1.0) for v in self.names], 1)

    def unpack(self, x):
        ph = {"u": 1j, "uz": 1j, "v": 1j, "vz": 1j} if self.S > 2 else {}
        return {v: x[:, i * self.N:(i + 1) * self.N] * ph.get(v, 1.0) for i, v in enumerate(self.names)}

    def place_rhs(self, F):
        """Left-preconditioned right-hand side of {equation: T coefficients} and boundary values."""
        out = self.g.to(torch.complex128)
        parts, at = [], 0
        for name, c in sorted(F.items(), key=lambda t: self.place[t[0]][0]):
            r, m, diff, phase = self.place[name]
            f = c * (-1j) ** phase
            f = torch.einsum("mn,pn->pm", self.U.to(torch.complex128), f)[:, :m] if diff else f
            parts += [out[:, at:r], out[:, r:r + m] + f]
            at = r + m
        return torch.cat(parts + [out[:, at:]], 1)

    def rhs(self, x):
        X = self.unpack(x)
        grids = {}

        def grid(v, axis=None):
            if (v, axis) not in grids:
                c = X[v] if axis is None else X[v] * (1j * (self.kx if axis == "x" else self.ky))[:, None]
                grids[v, axis] = self.to_grid(c, self.scale)
            return grids[v, axis]

        if self.S == 2:
            return self.place_rhs({"u": self.to_coef(-grid("u") * grid("u"))})
        F = {}
        for e in ("b", "u", "v", "w") if self.ny else ("b", "u", "w"):
            f = grid("u") * grid(e, "x") + grid("w") * grid(e + "z")
            if self.ny:
                f = f + grid("v") * grid(e, "y")
            F[e] = self.to_coef(-f)
        return self.place_rhs(F)

    def mul(self, A, x):
        return torch.view_as_complex(torch.bmm(A, torch.view_as_real(x).contiguous()).contiguous())

    def rk_step(self, x, dt, scheme):
        H, A = _tableau(scheme)
        mx, Fs, Ls = self.mul(self.M, x), [self.rhs(x)], [None]
        for i in range(1, len(H)):
            b = mx + dt * sum(A[i][j] * Fs[j] for j in range(i) if A[i][j])
            b = b - dt * sum(H[i][j] * Ls[j] for j in range(1, i) if H[i][j]) if i > 1 else b
            x = self.solve(1.0, dt * H[i][i], b)
            if i + 1 < len(H):
                Fs.append(self.rhs(x))
                Ls.append(self.mul(self.L, x))
        return x

    def run(self, x, dt, scheme, steps):
        if scheme.startswith("RK"):
            for _ in range(steps):
                x = self.rk_step(x, dt, scheme)
            return x
        order = int(scheme[-1])
        Ms, Fs = [], []
        for it in range(steps):
            o = min(order, it + 1)
            a, c = _SBDF[o]
            Ms, Fs = [self.mul(self.M, x)] + Ms[:order - 1], [self.rhs(x)] + Fs[:order - 1]
            b = sum(-a[j + 1] * Ms[j] + dt * c[j] * Fs[j] for j in range(o))
            x = self.solve(a[0], dt, b)
        return x


def _rb_reference(c):
    ny = c.get("ny")
    R = _Reference(VARS3 if ny else VARS2, c["nx"], c["nz"], (c.get("num", 3), c.get("den", 2)), 4.0, ny,
                   4.0 if ny else None)
    kappa = nu = c["ra"] ** -0.5
    k2 = R.kx ** 2 + R.ky ** 2
    vel = ("u", "v", "w") if ny else ("u", "w")
    for v in ("b",) + vel:
        R.equation(v + "z_def", [], [(v, "dz", 1.0), (v + "z", "I", -1.0)], True)
    R.equation("b", [("b", "I", 1.0)], [("b", "I", kappa * k2), ("bz", "dz", -kappa)], True)
    for v, k in (("u", R.kx), ("v", R.ky)):
        if v in vel:
            R.equation(v, [(v, "I", 1.0)], [(v, "I", nu * k2), (v + "z", "dz", -nu), ("p", "I", k)], True, 1)
    R.equation("w", [("w", "I", 1.0)], [("w", "I", nu * k2), ("wz", "dz", -nu), ("p", "dz", 1.0), ("b", "I", -1.0)],
               True)
    div = [("u", "I", -R.kx), ("wz", "I", 1.0)] + ([("v", "I", -R.ky)] if ny else [])
    R.equation("div", [], div, False)
    every = torch.ones_like(R.zero)
    R.boundary([("b", "left", 1.0, R.zero), ("b", "left", 0.0, ~R.zero)])
    R.boundary([("b", "right", 0.0, every)])
    for v in vel[:-1]:
        R.boundary([(v, "left", 0.0, every)])
        R.boundary([(v, "right", 0.0, every)])
    R.boundary([("w", "left", 0.0, every)])
    R.boundary([("w", "right", 0.0, ~R.zero), ("p", "right", 0.0, R.zero)])
    R.assemble()
    return R


def _rb_start(R, c, seed):
    nh = (c["ny"], c["nx"]) if R.ny else (c["nx"],)
    noise, vel = _flow(seed, c["nz"], *nh)
    z = _nodes(c["nz"]).reshape((-1,) + (1,) * len(nh))
    grids = dict(vel, b=1.0 - z + 1e-2 * noise * z * (1.0 - z))
    X = {v: torch.zeros((R.P, R.N), dtype=torch.complex128, device=R.dev) for v in R.names}
    for v, g in grids.items():
        X[v] = R.to_coef(torch.tensor(g, device=R.dev))
        X[v + "z"] = R.dz(X[v])
    return R.pack(X)


def _dense_cost(c):
    """Bytes and seconds, roughly, of the dense reference."""
    ny = c.get("ny") or 1
    p, s = ny * c["nx"] // 2, 7 if ny == 1 else 9
    if c["kind"] in ("fisher", "qg"):
        s = 2
    n = s * c["nz"]
    factors = {"SBDF2": 2, "SBDF3": 3}.get(c.get("scheme"), 1)
    if c["kind"] == "cfl":
        factors = c["steps"]
    solves = c.get("steps", 1) * _STAGES.get(c.get("scheme"), 1)
    # memory-bound products and solves on the dense matrices, LU at about half the FP64 rate
    return p * n * n * 8.0, p * (n ** 3 * 0.67 / 4e11 * factors + 4 * n * n * 8 * solves / 2e12) + 3e-4 * p * factors


def exact(case, seed):
    kind = case["kind"]
    if kind == "evp":
        return None                      # the iterate after a given number of sweeps, not a closed value
    if kind == "batch":
        cs = _sweep(case)
        if sum(_dense_cost(c)[1] for c in cs) > 12 or max(_dense_cost(c)[0] for c in cs) > 2.5e10:
            return None
        out = []
        for i, c in enumerate(cs):
            R = _rb_reference(c)
            X = R.unpack(R.run(_rb_start(R, c, seed + 1000 * i), c["dt"], c["scheme"], c["steps"]))
            out.append(_stack(X))
        return out
    nbytes, seconds = _dense_cost(case)
    if nbytes > 2.5e10 or seconds > 12:
        return None
    if kind in ("rb2d", "rb3d"):
        R = _rb_reference(case)
        return R.unpack(R.run(_rb_start(R, case, seed), case["dt"], case["scheme"], case["steps"]))
    if kind == "cfl":
        R = _rb_reference(case)
        x, dt = _rb_start(R, case, seed), case["dt"]
        for _ in range(case["steps"]):
            dt = _cfl_dt(R, x, dt, _cfl_rule(case))
            x = R.rk_step(x, dt, case["scheme"])
        return R.unpack(x)
    if kind == "fisher":
        R = _Reference(("u", "uz"), case["nx"], case["nz"], (case["num"], case["den"]), 2 * np.pi)
        R.equation("uz_def", [], [("u", "dz", 1.0), ("uz", "I", -1.0)], True)
        R.equation("u", [("u", "I", 1.0)], [("u", "I", 0.1 * R.kx ** 2 - 1.0), ("uz", "dz", -0.1)], True)
        every = torch.ones_like(R.zero)
        R.boundary([("uz", "left", 0.0, every)])
        R.boundary([("uz", "right", 0.0, every)])
        R.assemble()
        u = R.to_coef(torch.tensor(_fisher_u(case, seed), device=R.dev))
        return R.unpack(R.run(R.pack({"u": u, "uz": R.dz(u)}), case["dt"], case["scheme"], case["steps"]))
    if kind == "qg":
        R = _Reference(("psi", "psiz"), case["nx"], case["nz"], (3, 2), 2 * np.pi)
        N = R.N
        S = torch.zeros((N, N), dtype=torch.float64, device=R.dev)
        for m, s in enumerate(_profile(case)):
            for j in range(N):
                for i in (j + m, abs(j - m)):
                    if i < N:
                        S[i, j] += 0.5 * s
        R.equation("psiz_def", [], [("psi", "dz", 1.0), ("psiz", "I", -1.0)], True)
        R.equation("pv", [], [("psi", "I", -R.kx ** 2), ("psiz", R.D @ S, 1.0)], True)
        every = torch.ones_like(R.zero)
        R.boundary([("psiz", "left", 0.0, every)])
        R.boundary([("psiz", "right", 0.0, ~R.zero), ("psi", "right", 0.0, R.zero)])
        R.assemble()
        q = torch.tensor(_qg_q(case, seed), device=R.dev)
        return R.unpack(R.solve(0.0, 1.0, R.place_rhs({"pv": q})))
    return _adjoint_reference(case, seed)


def _cfl_dt(R, x, dt, rule):
    X = R.unpack(x)
    ngz, _, ngx = R.sizes(R.scale)
    dz = torch.tensor(np.gradient(_nodes(ngz)), device=R.dev)[:, None]
    f = R.to_grid(X["u"], R.scale).abs() / (4.0 / ngx) + R.to_grid(X["w"], R.scale).abs() / dz
    new = rule["safety"] / float(f.max())
    new = min(max(new, rule["min_dt"]), rule["max_dt"])
    new = min(max(new, rule["min_change"] * dt), rule["max_change"] * dt)
    return dt if abs(new - dt) < rule["threshold"] * dt else new


def _adjoint_reference(case, seed):
    """Loss and gradient by differentiating the dense reference."""
    noise, target, q = _adjoint_inputs(case, seed)
    R = _rb_reference(dict(case, num=3, den=2))
    z = torch.tensor(_nodes(case["nz"])[:, None], device=R.dev)
    qt = torch.tensor(q, device=R.dev, requires_grad=True)
    b = R.to_coef(1.0 - z + (1e-2 * torch.tensor(noise, device=R.dev) + qt) * z * (1.0 - z))
    X = {v: torch.zeros((R.P, R.N), dtype=torch.complex128, device=R.dev) for v in R.names}
    X.update(b=b, bz=R.dz(b))
    x = R.run(R.pack(X), case["dt"], case["scheme"], case["steps"])
    r = R.to_grid(R.unpack(x)["b"], (1, 1)) - torch.tensor(target, device=R.dev)
    loss = 0.5 * (r * r).sum()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": qt.grad}
