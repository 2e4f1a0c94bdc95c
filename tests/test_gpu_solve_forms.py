"""Which kernels serve a problem's pencil solves (sp_get_solve_kernels), on both
sides of every size at which the choice changes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1905_10388_gb300.solver import Context, FisherKPPSolver, QGInversion, RB3DSolver, RBSolver
from gpu_util import rel_err

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


# 2048 pencils: 512 rows in row blocks, 128 rows whole (the same bits as the
# window order, for a band that cannot be asked for by name)
@pytest.mark.parametrize("nz,blocks", [(256, True), (64, False)])
def test_row_blocks_come_before_whole_pencils(ctx, nz, blocks):
    out = []
    for kind in ("window", "auto"):
        s = FisherKPPSolver(ctx, 4096, nz, scheme="SBDF2", precision="mixed", dealias=(1, 1))
        s.set_solve_kernel(kind)
        s.factor(1e-3)
        if kind == "auto":
            assert ("k_lane_fwd<1>" in s.solve_kernels()) == blocks
            assert ("k_lane_fwd<0>" in s.solve_kernels()) != blocks
        s.set_initial_state(np.random.default_rng(1).random((nz, 4096)))
        s.step(3)
        s.sync()
        out.append(s.get_state())
    assert np.isfinite(out[0]).all()
    if blocks:
        for a, b in zip(*out):
            assert rel_err(b, a) < 1e-9
    else:
        assert np.array_equal(*out)


@pytest.mark.parametrize("nx,nz,kernel", [(768, 64, "k_pencil_solve_narrow"), (1024, 64, "k_pencil_solve_narrow"),
                                          (1536, 12, "k_pencil_pair")])
def test_whole_row_kernel_by_pencils(ctx, nx, nz, kernel):
    d = (3, 2) if nx == 1024 else (4, 3) if nz % 3 == 0 else (2, 1)
    assert _upload(RBSolver(ctx, nx, nz, 1e6, precision="mixed", dealias=d)) == [kernel]
