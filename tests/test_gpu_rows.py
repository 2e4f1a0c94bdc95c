"""The right-hand side's transforms and products (Sec. "Arithmetic operators",
"Scaled transforms & dealiasing") against a dense evaluation in numpy: FFT
lengths of every plan shape (two and three passes, with and without the factor
three), padded and unpadded spectra, odd numbers of fields and products, column
tiles cut short, in two and three dimensions.

The dense evaluation sums the same products in FP64.  FP64 results agree to
rounding, amplified at most by the transforms' lengths (1e-12 relative).  The
mixed form's bound comes from the dense evaluation itself.  Two real fields
share a complex x transform, and an FFT leaves errors of a few units in the last
place of its sequence's root mean square at every point, so a field's error is
relative to its pair's magnitude (a velocity paired with an x derivative of a
white spectrum up to k_x ~ 800 is hundreds of times the smaller one).  Every
grid field gets such errors (8 FP32 units of the pair's root mean square,
random), and the mixed result may be off by four times what they do to the
right-hand side.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1905_10388_gb300 import rb as rbmod
from paper_1905_10388_gb300.solver import Context, FisherKPPSolver, RB3DSolver, RBSolver
from gpu_util import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.close()


def _cheb(ng, nc):
    i = np.arange(ng)
    return np.cos(np.arange(nc)[None, :] * (np.pi * (ng - 0.5 - i) / ng)[:, None])


def _state(s, seed):
    rng = np.random.default_rng(seed)
    K = s.Nx // 2
    decay = 1.0 / (1.0 + np.arange(s.Nz))
    X = (rng.standard_normal((s.S, s.Ny, K, s.Nz)) + 1j * rng.standard_normal((s.S, s.Ny, K, s.Nz))) * decay
    if s.ndim == 2:
        X[:, 0, 0] = X[:, 0, 0].real
    else:
        iy = np.arange(s.Ny)
        X[:, :, 0] = 0.5 * (X[:, :, 0] + np.conj(X[:, (-iy) % s.Ny, 0]))
        X[:, s.Ny // 2] = 0.0
    return X.reshape(s.S, s.P, s.Nz)


def _dense_rhs(s, X, terms, scale, ulps=0.0):
    noise = np.random.default_rng(1)
    g = lambda n: n * scale[0] // scale[1]
    ngz, ngx, K = g(s.Nz), g(s.Nx), s.Nx // 2
    T = _cheb(ngz, s.Nz)
    kx = 2 * np.pi * np.arange(K) / s.Lx
    h = s.Ny // 2
    if s.ndim == 3:
        ngy = g(s.Ny)
        iy = np.arange(s.Ny)
        ky = 2 * np.pi * np.where(iy < h, iy, iy - s.Ny) / s.Ly

    def grid(op, var):
        c = X[s.state_order.index(var)].reshape(s.Ny, K, s.Nz)
        if op == "DX":
            c = c * (1j * kx)[None, :, None]
        if op == "DY":
            c = c * (1j * ky)[:, None, None]
        f = np.einsum("zn,ykn->zyk", T, c)
        if s.ndim == 3:
            p = np.zeros((ngz, ngy, K), complex)
            p[:, :h] = f[:, :h]
            p[:, ngy - h + 1:] = f[:, h + 1:]
            f = np.fft.ifft(p, axis=1) * ngy
        f[..., 0].imag = f[..., 0].imag if s.ndim == 3 else 0.0
        return np.fft.irfft(f, ngx, axis=-1) * ngx

    fields = []                                    # in the order of their first use, two to a sequence
    for _, _, oa, va, ob, vb in terms:
        for f in ((oa, va), (ob, vb)):
            if f not in fields:
                fields.append(f)
    G = {f: grid(*f) for f in fields}
    for q in range(0, len(fields), 2):
        pair = fields[q:q + 2]
        rms = np.sqrt(sum(np.mean(G[f] ** 2) for f in pair))
        for f in pair:
            G[f] = G[f] + ulps * 2.0 ** -24 * rms * noise.standard_normal(G[f].shape)
    out = {}
    for eq, coef, oa, va, ob, vb in terms:
        out[eq] = out.get(eq, 0.0) + coef * G[oa, va] * G[ob, vb]
    for eq, f in out.items():
        c = (np.fft.rfft(f, axis=-1) / ngx)[..., :K]
        if s.ndim == 3:
            c = np.fft.fft(c, axis=1) / ngy
            q = np.zeros((ngz, s.Ny, K), complex)
            q[:, :h] = c[:, :h]
            q[:, h + 1:] = c[:, ngy - h + 1:]
            c = q
        w = np.full(s.Nz, 2.0 / ngz)
        w[0] = 1.0 / ngz
        out[eq] = np.einsum("zn,zyk->ykn", T * w, c).reshape(s.P, s.Nz)
    return out


def _check(s, terms, scale, prec):
    X = _state(s, s.Nx + s.Nz)
    s.factor(1e-3)
    s.set_state(X)
    got, ref = s.eval_rhs(), _dense_rhs(s, X, terms, scale)
    off = _dense_rhs(s, X, terms, scale, ulps=8.0) if prec == "mixed" else None
    for e in ref:
        assert rel_err(got[e], ref[e]) < (1e-12 if prec == "fp64" else 4.0 * rel_err(off[e], ref[e])), e


@pytest.mark.parametrize("nx,nz,scale,prec", [
    (12, 24, (4, 3), "fp64"), (16, 16, (3, 2), "fp64"), (24, 48, (4, 3), "mixed"), (32, 64, (3, 2), "fp64"),
    (48, 12, (4, 3), "fp64"), (96, 96, (2, 1), "mixed"), (96, 192, (4, 3), "fp64"), (128, 32, (3, 2), "mixed"),
    (192, 64, (2, 1), "fp64"), (256, 128, (3, 2), "mixed"), (512, 512, (3, 2), "mixed"),
    (384, 24, (4, 3), "fp64"), (1024, 16, (3, 2), "mixed"), (1024, 16, (2, 1), "mixed")])
def test_rhs_2d(ctx, nx, nz, scale, prec):
    s = RBSolver(ctx, nx, nz, 1e5, precision=prec, dealias=scale)
    _check(s, rbmod.BILINEAR_TERMS, scale, prec)


@pytest.mark.parametrize("nx,nz,prec", [(2048, 16, "mixed"), (2048, 1024, "mixed"), (1024, 64, "fp64"), (64, 16, "fp64")])
def test_rhs_one_field(ctx, nx, nz, prec):
    from paper_1905_10388_gb300 import fisher
    s = FisherKPPSolver(ctx, nx, nz, precision=prec)
    _check(s, fisher.bilinear_terms(1.0), (3, 2), prec)


@pytest.mark.parametrize("nx,ny,nz,scale,prec", [
    (16, 16, 16, (3, 2), "fp64"), (32, 16, 32, (3, 2), "mixed"), (24, 12, 24, (4, 3), "fp64"),
    (12, 48, 12, (4, 3), "mixed"), (64, 128, 16, (3, 2), "mixed")])
def test_rhs_3d(ctx, nx, ny, nz, scale, prec):
    s = RB3DSolver(ctx, nx, ny, nz, 1e5, precision=prec, dealias=scale)
    _check(s, rbmod.BILINEAR_TERMS_3D, scale, prec)


@pytest.mark.parametrize("shape", [(64, 32), (256, 64), (64, 32, 32)])
def test_products_near_the_top_of_single_precision(ctx, shape):
    """Products of 4e35 and sums of them over one axis fit FP32 (3.4e38); no
    transform may carry the sum over two.  Single modes: errors of a few FP32
    units, 3e-7 measured, bar 1e-6."""
    out = []
    for prec in ("fp64", "mixed"):
        if len(shape) == 3:
            s = RB3DSolver(ctx, *shape, 1e5, precision=prec)
            nh = (shape[1], shape[0])
        else:
            s = RBSolver(ctx, *shape, 1e5, precision=prec)
            nh = (shape[0],)
        z = np.pi * rbmod.chebyshev_nodes(s.Nz).reshape((-1,) + (1,) * len(nh))
        x = 2 * np.pi * np.arange(nh[-1]) / nh[-1]
        for i, v in enumerate(("b", "u", "w")):
            s.set_field(v, 3e17 * np.sin((i + 1) * z) * np.cos((i + 1) * x + i) * np.ones((s.Nz,) + nh), layout="g")
        out.append(s.eval_rhs())
    size = max(np.linalg.norm(f) for f in out[0].values())     # (3D: v's products are zero but for rounding)
    for e in out[0]:
        assert np.isfinite(out[1][e]).all(), e
        assert np.linalg.norm(out[1][e] - out[0][e]) < 1e-6 * size, e
