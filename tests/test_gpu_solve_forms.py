"""Which kernels serve a problem's pencil solves (sp_get_solve_kernels), on both
sides of every size at which the choice changes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1905_10388_gb300.solver import Context, FisherKPPSolver, QGInversion, RB3DSolver, RBSolver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.close()


def _upload(s):
    s.set_field(s.state_order[0], np.zeros((s.P, s.Nz), complex))
    return s.solve_kernels()


@pytest.mark.parametrize("kind,kernels", [("window", ["k_pencil_solve"]), ("spike", ["k_pencil_split"]),
                                          ("lanes", ["k_pencil_stage<1>", "k_lane_fwd<0>", "k_lane_bwd<0>",
                                                     "k_pencil_stage<2>"])])
def test_kernels_asked_for_by_name(ctx, kind, kernels):
    s = RBSolver(ctx, 64, 64, 1e6)
    s.set_solve_kernel(kind)
    assert _upload(s) == kernels
