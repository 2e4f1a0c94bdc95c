"""Which kernels serve a problem's pencil solves (sp_get_solve_kernels), on both
sides of every size at which the choice changes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1905_10388_gb300.solver import Context, FisherKPPSolver, QGInversion, RBOnsetEVP, RBSolver, step_batched
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
                                          ("lanes", ["k_pencil_stage_wide<1>", "k_lane_fwd<0>", "k_lane_bwd<0>",
                                                     "k_pencil_stage_wide<2>"])])
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


PASSES = ["k_spike_fwd<1>", "k_spike_fwd_rec", "k_spike_fwd<2>", "k_spike_bwd<1>", "k_spike_bwd_rec", "k_spike_bwd<2>"]


# one CTA per pencil where all are on the GPU at once and most of it is taken, or
# the chains are short; else passes in launches of their own
@pytest.mark.parametrize("nx,nz,d,passes", [
    (64, 256, (3, 2), False), (64, 384, (2, 1), True), (64, 1024, (3, 2), True), (256, 512, (3, 2), False),
    (256, 1024, (3, 2), True), (384, 96, (4, 3), False), (384, 192, (4, 3), True), (512, 256, (3, 2), False),
    (512, 512, (3, 2), True), (768, 96, (4, 3), True), (1024, 256, (3, 2), True)])
def test_partitioned_form_by_size(ctx, nx, nz, d, passes):
    k = _upload(RBSolver(ctx, nx, nz, 1e6, precision="mixed", dealias=d))
    assert k[1:-1] == PASSES if passes else k == ["k_pencil_split"]


# (nx, nz, dealias, precision, blocks asked for): few long pencils, more than one
# wave of CTAs, N_z = 1024 at two pencil counts, and block counts that one CTA's
# shared memory does not hold
@pytest.mark.parametrize("nx,nz,d,prec,blocks", [
    (64, 384, (2, 1), "fp64", 0), (768, 48, (4, 3), "mixed", 11), (768, 96, (4, 3), "mixed", 0), (1024, 128, (3, 2), "mixed", 0),
    (32, 1024, (3, 2), "fp64", 0), (32, 1024, (3, 2), "fp64", 112), (256, 1024, (3, 2), "mixed", 0)])
def test_passes_equal_window_to_rounding(ctx, nx, nz, d, prec, blocks):
    xi = np.random.default_rng(4).standard_normal((nz, nx))
    out = []
    for kind in ("window", "spike" if blocks else "auto"):
        s = RBSolver(ctx, nx, nz, 1e6, scheme="SBDF2", precision=prec, dealias=d)
        s.set_solve_kernel(kind)
        if blocks and kind != "window":
            s.set_spike_blocks(blocks)
        s.factor(1e-4)
        if kind != "window":
            assert s.solve_kernels()[1:-1] == PASSES
            assert s.spike_blocks() == blocks if blocks else s.spike_blocks() > 1
        s.set_initial_state(xi, amplitude=1e-2)
        s.step(4, graph=True)
        s.sync()
        out.append(s.get_state())
    assert np.isfinite(out[0]).all()
    for a, b in zip(*out):                         # the bars of the partitioned substitution elsewhere
        assert rel_err(b, a) < (1e-11 if prec == "fp64" else 1e-5)


def test_batch_of_long_problems_equals_them_alone_to_rounding(ctx):
    """Two problems that run in passes alone, in one CTA per pencil together."""
    def make():
        out = []
        for i, (nx, nz, d) in enumerate(((64, 384, (2, 1)), (32, 512, (3, 2)))):
            s = RBSolver(ctx, nx, nz, 1e6, scheme="SBDF2", dealias=d)
            s.factor(1e-4)
            assert s.solve_kernels()[1:-1] == PASSES
            s.set_initial_state(np.random.default_rng(i).standard_normal((nz, nx)), amplitude=1e-2)
            out.append(s)
        return out
    alone, batch = make(), make()
    for s in alone:
        s.step(4)
    step_batched(batch, 4)
    ctx.sync_status()
    for a, b in zip(alone, batch):
        X, Y = a.get_state(), b.get_state()
        assert np.isfinite(X).all()
        for x, y in zip(X, Y):
            assert rel_err(y, x) < 1e-11


# kl = 8: 32-lane windows both ways
@pytest.mark.parametrize("nx,nz,kernel", [(256, 32, "k_pencil_solve"), (256, 64, "k_pencil_split"),
                                          (512, 64, "k_pencil_solve"), (512, 128, "k_pencil_split"),
                                          (1024, 128, "k_pencil_solve_narrow")])
def test_wide_lower_band_by_rows(ctx, nx, nz, kernel):
    assert _upload(RBOnsetEVP(ctx, nx, nz, 2000.0)) == [kernel]


# whole-row batches: the window kernel (332 pencils), pencils alone in the pair
# kernel (640 of 1792 rows), two to a CTA (1280 of 224 rows)
@pytest.mark.parametrize("shapes", [[(512, 16), (128, 32), (24, 12)], [(256, 256)] * 5, [(64, 32)] * 40])
def test_whole_row_batches_equal_window_bit_for_bit(ctx, shapes):
    def make():
        out = []
        for i, (nx, nz) in enumerate(shapes):
            s = RBSolver(ctx, nx, nz, 1e6, scheme="SBDF2", precision="mixed", dealias=(4, 3) if nx % 3 == 0 else (3, 2))
            s.set_solve_kernel("window")
            s.factor(1e-4)
            s.set_initial_state(np.random.default_rng(i).standard_normal((nz, nx)), amplitude=1e-2)
            out.append(s)
        return out
    alone, batch = make(), make()
    for s in alone:
        s.step(3)
    step_batched(batch, 3)
    ctx.sync_status()
    for a, b in zip(alone, batch):
        assert np.isfinite(a.get_state()).all()
        assert np.array_equal(a.get_state(), b.get_state())


@pytest.mark.parametrize("nx,nz,kernel", [(32, 16, "k_pencil_solve"), (512, 16, "k_pencil_solve"), (48, 24, "k_pencil_split"),
                                          (512, 32, "k_pencil_split")])
def test_short_pencils_keep_the_window_kernel(ctx, nx, nz, kernel):
    assert _upload(RBSolver(ctx, nx, nz, 1e6, dealias=(4, 3) if nx % 3 == 0 else (3, 2))) == [kernel]


@pytest.mark.parametrize("nx,nz,kernel", [(96, 48, "k_pencil_solve"), (128, 64, "k_pencil_split"), (256, 64, "k_pencil_split"),
                                          (512, 64, "k_pencil_solve"), (512, 128, "k_pencil_split")])
def test_short_pencils_of_a_narrow_band(ctx, nx, nz, kernel):
    assert _upload(FisherKPPSolver(ctx, nx, nz, dealias=(4, 3) if nx % 3 == 0 else (3, 2))) == [kernel]


def test_batch_of_unlike_kernels_equals_problems_alone_bit_for_bit(ctx):
    """Partitioned (64 x 32) and whole-row solves (32 x 16), transforms on
    compile-time lengths and, on 12 points in z, on run-time ones."""
    def make():
        out = [RBSolver(ctx, nx, nz, 1e5, scheme="RK222", precision="mixed") for nx, nz in ((64, 32), (32, 16))]
        out.append(FisherKPPSolver(ctx, 64, 8, scheme="RK222", precision="mixed"))
        for i, s in enumerate(out):
            s.factor(1e-4)
            rng = np.random.default_rng(i)
            if i < 2:
                s.set_initial_state(rng.standard_normal((s.Nz, s.Nx)), amplitude=1e-2)
            else:
                s.set_initial_state(rng.random((s.Nz, s.Nx)))
        return out
    alone, batch = make(), make()
    assert [s.solve_kernels() for s in batch] == [["k_pencil_split"], ["k_pencil_solve"], ["k_pencil_solve"]]
    for s in alone:
        s.step(5)
    step_batched(batch, 5)
    ctx.sync_status()
    for a, b in zip(alone, batch):
        assert np.isfinite(a.get_state()).all()
        assert np.array_equal(a.get_state(), b.get_state())


# the lane form's row blocks with bands wider than the reaction-diffusion one:
# kl + ku = 29 (recurrence of four warps per chain), several block counts
@pytest.mark.parametrize("nx,nz,d,blocks", [(1536, 96, (4, 3), 0), (1536, 96, (4, 3), 3), (1536, 96, (4, 3), 7),
                                            (2048, 128, (1, 1), 0)])
def test_lane_row_blocks_of_a_wide_band_equal_window_to_rounding(ctx, nx, nz, d, blocks):
    xi = np.random.default_rng(4).standard_normal((nz, nx))
    out = []
    for kind in ("window", "auto"):
        s = RBSolver(ctx, nx, nz, 1e6, scheme="SBDF2", precision="mixed", dealias=d)
        s.set_solve_kernel(kind)
        if blocks and kind == "auto":
            s.set_spike_blocks(blocks)
        s.factor(1e-4)
        if kind == "auto":
            assert {"k_lane_fwd<1>", "k_spike_bwd_rec"} <= set(s.solve_kernels())
            assert s.spike_blocks() == blocks if blocks else s.spike_blocks() > 1
        s.set_initial_state(xi, amplitude=1e-2)
        s.step(4)
        s.sync()
        out.append(s.get_state())
    assert np.isfinite(out[0]).all()
    for a, b in zip(*out):
        assert rel_err(b, a) < 1e-5


# kl + ku = 9 (recurrence in 16 lanes per chain), FP64: the partitioned bar
@pytest.mark.parametrize("nx,nz,blocks", [(2048, 256, 0), (2048, 512, 4)])
def test_lane_row_blocks_of_an_inversion_equal_window_to_rounding(ctx, nx, nz, blocks):
    rng = np.random.default_rng(8)
    q = (rng.standard_normal((nx // 2, nz)) + 1j * rng.standard_normal((nx // 2, nz))) / (1 + np.arange(nz))
    q[0] = q[0].real
    out = []
    for kind in ("window", "auto"):
        s = QGInversion(ctx, nx, nz, [1.688, 0.75, 0.063])
        s.set_solve_kernel(kind)
        if blocks and kind == "auto":
            s.set_spike_blocks(blocks)
        out.append(s.invert(q))
        if kind == "auto":
            assert {"k_lane_fwd<1>", "k_spike_bwd_rec_narrow"} <= set(s.solve_kernels())
    for a, b in zip(*out):
        assert rel_err(b, a) < 1e-11


@pytest.mark.parametrize("scheme,prec", [("RK222", "fp64"), ("SBDF2", "mixed")])
def test_batch_beyond_304_pencils_equals_problems_alone_to_rounding(ctx, scheme, prec):
    """On the automatic kernels: whole-row order together (320 pencils), one CTA
    per pencil alone."""
    def make():
        out = []
        for i, (nx, nz) in enumerate(((512, 32), (64, 64), (64, 32))):
            s = RBSolver(ctx, nx, nz, 1e6, scheme=scheme, precision=prec)
            s.factor(1e-4)
            assert s.solve_kernels() == ["k_pencil_split"]
            s.set_initial_state(np.random.default_rng(i).standard_normal((nz, nx)), amplitude=1e-2)
            out.append(s)
        return out
    alone, batch = make(), make()
    for s in alone:
        s.step(5)
    step_batched(batch, 5)
    ctx.sync_status()
    for a, b in zip(alone, batch):
        X, Y = a.get_state(), b.get_state()
        assert np.isfinite(X).all()
        for x, y in zip(X, Y):                     # the bars of partitioned against whole-row solves
            assert rel_err(y, x) < (1e-11 if prec == "fp64" else 1e-5)
