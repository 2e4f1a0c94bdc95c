"""Solves that follow one another need not be steps of one run: their results
depend on their own inputs alone, bit for bit, whatever was solved before (the
partitioned back substitution starts from the previous solve's inflows only
within a run; rounding errors scale with what it starts from).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1905_10388_gb300 import _lib
from paper_1905_10388_gb300.solver import Context, QGInversion, RBSolver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.close()


# one CTA per pencil (256 and 512 rows) and row blocks of the lane form (512 rows)
@pytest.mark.parametrize("nx,nz", [(64, 128), (512, 256), (2048, 256)])
def test_inversion_does_not_depend_on_the_one_before(ctx, nx, nz):
    rng = np.random.default_rng(5)

    def pv():
        q = rng.standard_normal((nx // 2, nz)) + 1j * rng.standard_normal((nx // 2, nz))
        q[0] = q[0].real
        return q
    q1, q2 = pv(), pv()
    first, later = (QGInversion(ctx, nx, nz, [1.688, 0.75, 0.063]) for _ in range(2))
    want = first.invert(q2)
    later.invert(q1 * 1e12)
    assert later.spike_blocks() > 1
    assert np.array_equal(later.invert(q2), want)


@pytest.mark.parametrize("nx,nz,scheme", [(64, 32, "RK222"), (64, 64, "RK111"), (256, 128, "RK222")])
def test_adjoint_step_does_not_depend_on_the_one_before(ctx, nx, nz, scheme):
    h, dt = ctx.handle, 1e-3
    rng = np.random.default_rng(6)

    def solver():
        s = RBSolver(ctx, nx, nz, 1e6, scheme=scheme)
        s.factor(dt)
        _lib.check(h, _lib.lib().sp_adjoint_init(h, s.pid))
        return s

    def adjoint(s, X, lam):
        X, lam = (torch.as_tensor(a, device="cuda") for a in (X, lam))
        _lib.check(h, _lib.lib().sp_step_adjoint(h, s.pid, dt, X.data_ptr(), 1, lam.data_ptr()))
        ctx.sync_status()
        return lam.cpu().numpy()
    first, later = solver(), solver()
    shape = (first.S, first.P, nz)
    (x1, l1), (x2, l2) = [[(rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / (1 + np.arange(nz)) ** 2
                           for _ in range(2)] for _ in range(2)]
    want = adjoint(first, x2, l2)
    adjoint(later, x1 * 1e3, l1 * 1e10)
    assert later.spike_blocks() > 1
    assert np.isfinite(want).all()
    assert np.array_equal(adjoint(later, x2, l2), want)
