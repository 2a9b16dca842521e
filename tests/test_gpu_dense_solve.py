"""The dense damped solve of small groups over the exponent range of its
pivots: a normal matrix as large or as small as float64 holds is solved, not
reported as not positive definite."""
from fractions import Fraction

import numpy as np
import pytest

from _helpers import O, device_context
from synthetic.problem import ImageSpec, Problem, SourceSpec

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_01957_gb300 import build
    build()


def _np(t):
    return t.detach().cpu().numpy().astype(np.float64)


def _problem(area, star_at):
    """A flat sky on 16 x 16 pixels of this area (its entry of J^T W J is
    256 area^2) and, at theta[star_at], the flux of a Gaussian (entry of order 0.1)."""
    a = np.sqrt(area)
    rng = np.random.default_rng(3)
    im = ImageSpec(16, 16, a * np.eye(2), np.zeros(2), data=rng.uniform(1.0, 2.0, (16, 16)).astype(np.float32),
                   variance=np.ones((16, 16), dtype=np.float32))
    sky = SourceSpec(O.SKY_FLAT, 0, (0, 16, 0, 16), False, np.full(8, -1, dtype=np.int64), np.zeros(8))
    sources, theta = [sky], []
    if star_at is None:
        sky.pidx[0] = 0
        theta = [0.5 / area]
    else:
        sky.pidx[0] = 1 - star_at
        i = np.full(8, -1, dtype=np.int64)
        i[5] = star_at
        f = np.array([7.7 * a, 8.2 * a, 0.8, 0.3, 2.0 * a, 0.0, 0.0, 0.0])
        sources.append(SourceSpec(O.GAUSSIAN, 0, (0, 16, 0, 16), False, i, f))
        theta = [0.5 / area, 2.0] if star_at else [2.0, 0.5 / area]
    th = np.array(theta)
    return Problem("pivots", [im], sources, th.size, th, th)


def _solve_exactly(M, b):
    """Gaussian elimination in rational numbers."""
    n = len(b)
    A = [[Fraction(float(M[i, j])) for j in range(n)] + [Fraction(float(b[i]))] for i in range(n)]
    for k in range(n):
        for i in range(k + 1, n):
            l = A[i][k] / A[k][k]
            A[i] = [x - l * y for x, y in zip(A[i], A[k])]
    x = [Fraction(0)] * n
    for k in range(n - 1, -1, -1):
        x[k] = (A[k][n] - sum(A[k][j] * x[j] for j in range(k + 1, n))) / A[k][k]
    return np.array([float(v) for v in x])


@pytest.mark.parametrize("entry", [1.0e308, 5.0e307, 4.0e307, 1.0e300, 1.0, 1.0e-300, 3.0e-308, 1.0e-308, 1.0e-310])
@pytest.mark.parametrize("star_at", [None, 0, 1])
def test_pivots_over_the_float64_range(entry, star_at):
    """Pivots past 2^1022 (whose reciprocal is subnormal) and subnormal ones
    (whose reciprocal overflows), alone, first and second of two: the step of the
    device's own damped matrix, exactly solved.  The tolerance: a few roundings of
    the solve, times a condition number (after scaling) of at most 4, and the
    spacing of subnormal entries, 5e-324 / 1e-310."""
    pr = _problem(np.sqrt(entry / 256.0), star_at)
    ctx = device_context(pr, "f64")
    jtwr, csr = ctx.normal_eq(pr.theta_init)
    M, b, lam = ctx.jtwj_dense(csr), _np(jtwr), 1e-3
    assert np.isfinite(M).all() and (np.diag(M) > 0).all()
    assert abs(M.max() / max(entry, M[0, 0]) - 1.0) < 1e-6 or entry < 1.0
    delta, lam_out = ctx.lm_solve(np.array([lam]))
    assert ctx.status() == 0
    assert _np(lam_out)[0] == lam
    # damping: lam max(diag, 1e-12 of the largest)
    D = np.maximum(np.diag(M), 1e-12 * np.diag(M).max())
    want = _solve_exactly(M + lam * np.diag(D), b)
    np.testing.assert_allclose(_np(delta), want, rtol=1e-12)
