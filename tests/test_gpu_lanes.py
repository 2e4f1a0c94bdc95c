"""The lane substitution on listed factor entries (Sec. "Matrix solvers").

* Whole pencils: every FMA in the window kernel's order, so SBDF2 states agree
  bit for bit; pencil counts that leave the last group of 16 short, row counts
  that are no multiple of the 4-row chunks' 32-row padding, wide and narrow
  bands.
* Row blocks (its form for hundreds to thousands of pencils): the inflows are
  summed in another order, so states agree with the window kernel to rounding;
  for the band shapes of the reaction-diffusion problem at two row counts.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import seeded_inputs as si
from paper_1905_10388_gb300.solver import Context, FisherKPPSolver, RB3DSolver, RBSolver
from gpu_util import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("shape", [(16, 16), (24, 12), (48, 96), (96, 24), (32, 6, 8), (8, 20, 24)])
def test_whole_pencils_equal_window_bit_for_bit(ctx, shape):
    out = []
    for kind in ("window", "lanes"):
        if len(shape) == 3:
            nx, ny, nz = shape
            d = (4, 3) if nz % 3 == 0 else (3, 2)
            nx, ny = (nx, 16) if d == (3, 2) else (24, 12)
            s = RB3DSolver(ctx, nx, ny, nz, 1e5, scheme="SBDF2", dealias=d)
            xi = si.rb_noise3(3, nz, ny, nx)
        else:
            nx, nz = shape
            d = (4, 3) if nx % 3 == 0 else (3, 2)
            s = RBSolver(ctx, nx, nz, 1e5, scheme="SBDF2", dealias=d)
            xi = si.rb_noise(3, nz, nx)
        s.set_solve_kernel(kind)
        s.factor(1e-3)
        s.set_initial_state(xi * 10.0)
        s.step(3)
        s.sync()
        out.append(s.get_state())
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("nz,prec", [(256, "fp64"), (384, "fp64"), (512, "mixed")])
def test_row_blocks_equal_window_to_rounding(ctx, nz, prec):
    d = (4, 3) if nz % 3 == 0 else (3, 2)
    nx = 1536 if nz % 3 == 0 else 2048
    u = si.fisher_noise(5, nz, nx)
    out = []
    for kind in ("window", "auto"):
        s = FisherKPPSolver(ctx, nx, nz, scheme="SBDF2", precision=prec, dealias=d)
        s.set_solve_kernel(kind)
        s.factor(1e-3)
        assert (s.spike_blocks() > 1) == (kind == "auto")
        s.set_initial_state(u)
        s.step(4)
        s.sync()
        out.append(s.get_state())
    for a, b in zip(*out):
        assert rel_err(b, a) < (1e-12 if prec == "fp64" else 1e-9)
