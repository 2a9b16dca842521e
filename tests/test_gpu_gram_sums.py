"""The sums of J^T W J over tiles past float32's range."""
import numpy as np
import pytest

from _helpers import O, TOL_GRAD, device_context
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


def _source(type_, image, win, pidx, pfix=()):
    i, f = np.full(8, -1, dtype=np.int64), np.zeros(8)
    i[:len(pidx)] = pidx
    f[:len(pfix)] = pfix
    return SourceSpec(type_, image, win, False, i, f)


@pytest.mark.parametrize("h,w", [(64, 64), (736, 736), (48, 43696)])
def test_entries_past_float32_range(h, w):
    """Weights so large that an entry's sum over tiles lies past float32's 3.4e38
    (a tile's own sum is 2.6e38): the float64 entry is finite.  Pairs of 16, 2116
    and 8193 tiles: summed by a warp, in one run, and in two."""
    var = 1e-36
    rng = np.random.default_rng(5)
    v = (var * rng.uniform(1.0, 1.2, (h, w))).astype(np.float32)
    sd = np.sqrt(var)
    im = ImageSpec(h, w, np.eye(2), np.zeros(2), data=(sd * rng.standard_normal((h, w))).astype(np.float32), variance=v)
    star = [20.3, 21.6, 0.8, 0.3, 2.0]
    pr = Problem("range", [im], [_source(O.SKY_FLAT, 0, (0, w, 0, h), [0]),
                                 _source(O.GAUSSIAN, 0, (4, 37, 5, 38), [-1] * 5 + [1], star)], 2,
                 np.zeros(2), np.array([2.0 * sd, 30.0 * sd]))
    ctx = device_context(pr, "mixed")
    jtwr, csr = ctx.normal_eq(pr.theta_init)
    ref, b = O.normal_equations(pr, pr.theta_init)
    got = ctx.jtwj_dense(csr)
    assert ref[0, 0] > 3.5e38
    # products of columns rounded three times, sums of 64 in float32
    assert np.abs(got / ref - 1.0).max() <= 80 * 2.0 ** -24, (got, ref)
    np.testing.assert_allclose(_np(jtwr), b, rtol=TOL_GRAD)
    delta, _ = ctx.lm_solve(np.array([1e-3]))
    want = np.linalg.solve(got + 1e-3 * np.diag(np.diag(got)), _np(jtwr))
    np.testing.assert_allclose(_np(delta), want, rtol=1e-10)
    assert ctx.status() == 0
