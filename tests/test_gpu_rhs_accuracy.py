"""Rounding error of the right-hand side's transforms (Sec. "Scaled transforms &
dealiasing") against an evaluation in extended precision, for FFT lengths of
two and three passes with and without the factor three.

A butterfly that multiplies an element by a twiddle at every level rounds it
more often than one that multiplies each input once.  The plain
Stockham kernels (transforms.cu) have a mean error (geometric, over the sizes
here) of 1.328e-15 in FP64 and 4.311e-7 in the mixed form; the right-hand side
may be 4 % above that.  Level-by-level twiddles are 14 % and 5 % above it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
fft = pytest.importorskip("scipy.fft")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1905_10388_gb300 import fisher as fkmod
from paper_1905_10388_gb300 import rb as rbmod
from paper_1905_10388_gb300.solver import Context, FisherKPPSolver, RBSolver

pytestmark = pytest.mark.gpu

SIZES = [("rb", 64, 32, (3, 2)), ("rb", 128, 64, (3, 2)), ("rb", 96, 48, (4, 3)), ("rb", 32, 256, (3, 2)),
         ("fk", 128, 64, (3, 2)), ("fk", 512, 64, (3, 2)), ("rb", 512, 16, (3, 2))]


def _exact(s, X, terms, scale):
    """{equation: (real, imaginary part)} of the dealiased products, longdouble."""
    ld = np.longdouble
    pi = ld("3.14159265358979323846264338327950288")
    g = lambda n: n * scale[0] // scale[1]
    gx, gz, K = g(s.Nx), g(s.Nz), s.Nx // 2
    n = np.arange(s.Nz)
    T = np.cos(np.outer(pi * (np.arange(gz) + ld(0.5)) / gz, n.astype(ld))) * np.where(n % 2, -1, 1)
    kx = (2 * np.pi * np.arange(K) / s.Lx).astype(ld)

    def grid(op, var):
        c = X[s.var[var]].astype(np.clongdouble)
        if op == "DX":
            c = c * (1j * kx)[:, None]
        f = np.zeros((gx // 2 + 1, gz), np.clongdouble)
        f[:K] = c.real @ T.T + 1j * (c.imag @ T.T)
        return fft.irfft(f, gx, axis=0) * gx

    prod = {}
    for eq, coef, oa, va, ob, vb in terms:
        prod[eq] = prod.get(eq, 0) + ld(coef) * grid(oa, va) * grid(ob, vb)
    w = np.where(n == 0, ld(1), ld(2)) / gz
    out = {}
    for eq, f in prod.items():
        c = fft.rfft(f, axis=0)[:K] / gx
        c[0] = c[0].real
        out[eq] = ((c.real @ T) * w, (c.imag @ T) * w)
    return out


@pytest.mark.parametrize("prec,start", [("fp64", 1.328e-15), ("mixed", 4.311e-7)])
def test_rounding_error_of_the_right_hand_side(prec, start):
    ctx = Context(0)
    logs = []
    for kind, nx, nz, scale in SIZES:
        errs = []
        for seed in range(2):
            rng = np.random.default_rng(seed)
            s = (FisherKPPSolver(ctx, nx, nz, precision=prec, dealias=scale) if kind == "fk"
                 else RBSolver(ctx, nx, nz, 1e6, precision=prec, dealias=scale))
            X = []
            for v in s.problem.variables:
                c = (rng.standard_normal((nx // 2, nz)) + 1j * rng.standard_normal((nx // 2, nz)))
                c = c / ((1 + np.arange(nx // 2))[:, None] * (1 + np.arange(nz)) ** 2)
                c[0] = c[0].real
                s.set_field(v, c)
                X.append(c)
            got = s.eval_rhs()
            ref = _exact(s, X, fkmod.bilinear_terms(1.0) if kind == "fk" else rbmod.BILINEAR_TERMS, scale)
            for e, (re, im) in ref.items():
                d = np.sqrt(np.sum((got[e].real - re) ** 2 + (got[e].imag - im) ** 2))
                errs.append(float(d / np.sqrt(np.sum(re * re + im * im))))
        logs.append(np.log(np.mean(errs)))
    ctx.close()
    assert np.exp(np.mean(logs)) < 1.04 * start
