"""Whole-row-order solves of one or two pencils per CTA and the register
factorization (Sec. "Matrix solvers").

* The pair kernel runs every FMA in the window kernel's order: a batch's
  states equal the problems stepped alone bit for bit, and a lone problem's
  those of the lane substitution on whole pencils; pencil counts on both sides
  of the change from one to two pencils per CTA, and both band widths.
* Bands of 8 to 15 and of more than 15 multipliers (eigenvalue and transposed
  factors) are reached only through their own solvers: a long channel's first
  pencils against the same pencils of a short one, and the adjoint step against
  its form in row blocks.
* Factors of matrices as short as the 32-column window and longer, narrow and
  wide bands, against the oracle after two steps.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import seeded_inputs as si
from oracle import fisher as ofk
from oracle import rb as orb
from oracle import timesteppers as ots
from paper_1905_10388_gb300 import _lib
from paper_1905_10388_gb300.adjoint import RBAdjoint
from paper_1905_10388_gb300.solver import Context, FisherKPPSolver, RB3DSolver, RBOnsetEVP, RBSolver, step_batched
from gpu_util import check_fields, oracle_floor, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.close()


# total pencils 332 (one per CTA) and 704 (two)
@pytest.mark.parametrize("shapes", [((512, 16), (128, 32), (24, 12)), ((512, 16), (512, 32), (384, 12))])
@pytest.mark.parametrize("scheme", ["SBDF2", "RK222"])
def test_batch_equals_problems_alone_bit_for_bit(ctx, shapes, scheme):
    def make():
        out = []
        for i, (nx, nz) in enumerate(shapes):
            s = RBSolver(ctx, nx, nz, 1e5, scheme=scheme, dealias=(4, 3) if nx % 3 == 0 else (3, 2))
            s.set_solve_kernel("window")
            s.factor(1e-3)
            s.set_initial_state(si.rb_noise(40 + i, nz, nx) * 10.0)
            out.append(s)
        return out
    alone, batch = make(), make()
    for s in alone:
        s.step(4)
    step_batched(batch, 4)
    ctx.sync_status()
    for a, b in zip(alone, batch):
        assert np.isfinite(a.get_state()).all()
        assert np.array_equal(a.get_state(), b.get_state())


@pytest.mark.parametrize("shape", [(768, 12), (1536, 12), (32, 32, 16), (24, 96, 12)])
def test_lone_problem_equals_lane_substitution_bit_for_bit(ctx, shape):
    out = []
    for kind in ("window", "lanes"):
        if len(shape) == 3:
            nx, ny, nz = shape
            s = RB3DSolver(ctx, nx, ny, nz, 1e5, scheme="SBDF2", dealias=(4, 3) if nx % 3 == 0 else (3, 2))
            xi = si.rb_noise3(3, nz, ny, nx)
        else:
            nx, nz = shape
            s = RBSolver(ctx, nx, nz, 1e5, scheme="SBDF2", precision="mixed", dealias=(4, 3))
            xi = si.rb_noise(3, nz, nx)
        s.set_solve_kernel(kind)
        s.factor(1e-3)
        s.set_initial_state(xi * 10.0)
        s.step(3)
        s.sync()
        out.append(s.get_state())
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


def test_eigenvalues_of_a_long_channel(ctx):
    """The first of 512 pencils (kl = 8) are those of a channel with 8; their eigenvalues agree to the accuracy the power
    iteration reaches, 1e-9."""
    nz, k = 16, 8
    mus = []
    for nx in (2 * k, 1024):
        s = RBOnsetEVP(ctx, nx, nz, 2000.0)
        mus.append(np.asarray(s.growth_rates(0.0, 60, np.ones((s.P, s.assembly["n"]), complex)))[:k])
    assert np.allclose(mus[0][1:], mus[1][1:], rtol=1e-9, atol=0)


def test_adjoint_of_a_long_channel(ctx):
    """sp_step_adjoint with the transposed factor's wide band and 384 pencils:
    whole-row order (window) against row blocks (auto).  The solves agree to
    FP64 rounding, the FP32 transforms' rounding then differs: 1e-5, the bound
    of the mixed form elsewhere."""
    nx, nz, dt = 768, 96, 1e-3
    rng = np.random.default_rng(21)
    lam, out = None, []
    for kind in ("window", "auto"):
        s = RBSolver(ctx, nx, nz, 1e5, scheme="RK222", precision="mixed", dealias=(4, 3))
        s.set_solve_kernel(kind)
        s.factor(dt)
        assert (s.spike_blocks() > 1) == (kind == "auto")
        RBAdjoint(s, si.rb_noise(1, nz, nx), np.zeros((nz, nx)))
        s.set_initial_state(si.rb_noise(3, nz, nx) * 50.0)
        X0 = s.get_state()
        if lam is None:
            lam = rng.standard_normal(X0.shape) + 1j * rng.standard_normal(X0.shape)
        slot = [s.var[v] for v in orb.RB_VARIABLES]
        Xs, Ls = np.zeros_like(X0), np.zeros_like(X0)
        Xs[slot], Ls[slot] = X0, lam
        Xd, Ld = (torch.as_tensor(a, device="cuda").contiguous() for a in (Xs, Ls))
        h = ctx.handle
        _lib.check(h, _lib.lib().sp_step_adjoint(h, s.pid, dt, Xd.data_ptr(), 1, Ld.data_ptr()))
        ctx.sync_status()
        out.append(Ld.cpu().numpy()[slot])
    for a, b in zip(*out):
        assert rel_err(b, a) < 1e-5


@pytest.mark.parametrize("nz", [16, 32])
def test_factor_of_small_matrices_rb(ctx, nz):
    """n = 112, 224 with kl = 7.  Bar 1e-11: at these sizes w's error against the
    oracle's other formulation is 1.1e-12 with either factorization."""
    nx, ra, dt = 16, 1e5, 1e-3
    xi = si.rb_noise(7, nz, nx)
    s = RBSolver(ctx, nx, nz, ra, scheme="RK222")
    s.factor(dt)
    s.set_initial_state(xi)
    s.step(2)
    s.sync()

    def stepper(sysr):
        st = ots.RungeKuttaIMEX(sysr)
        st.dt = dt
        return st
    ref, floor = oracle_floor(lambda m, lu: orb.RB2D(nx, nz, ra, cheb_method=m, lu_method=lu),
                              lambda sysr: sysr.initial_state(xi), stepper, 2)
    check_fields(s.get_state(), ref, floor, 1e-11, label=f"factor_{nx}x{nz}_rk222_fp64_2steps")


@pytest.mark.parametrize("nz", [16, 32])
def test_factor_of_small_matrices_fisher(ctx, nz):
    """n = 32, 64 with kl = 2."""
    nx, dt = 16, 1e-3
    u0 = si.fisher_noise(5, nz, nx)
    s = FisherKPPSolver(ctx, nx, nz, scheme="RK222")
    s.factor(dt)
    s.set_initial_state(u0)
    s.step(2)
    s.sync()
    sysr = ofk.FisherKPP(nx, nz, s.D, s.R, s.Lx)
    X = sysr.initial_state(u0)
    st = ots.RungeKuttaIMEX(sysr, ots.RK222)
    for _ in range(2):
        X = st.step(X, dt)
    got = s.get_state()
    for i, v in enumerate(ofk.FISHER_VARIABLES):
        assert rel_err(got[i], X[i]) < 1e-12, v
