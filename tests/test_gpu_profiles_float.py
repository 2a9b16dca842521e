"""The float32 form of the profiles where its hardware exponentials and
logarithms, and the range of its coefficients, show: steep and flat profiles out
to large radii, and radii far below a pixel."""
import math

import numpy as np
import pytest

from _helpers import O, TOL_GRAD, assert_grad_close, device_context, grad_scale, with_data
from synthetic.problem import ImageSpec, Problem, SourceSpec

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

X0, Y0, Q, PA = 20.3, 18.7, 0.7, 0.5


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_01957_gb300 import build
    build()


def _np(t):
    return t.detach().cpu().numpy().astype(np.float64)


def _problem(type_, slots, h=41, w=301, free=None, sky=None, quad_order=1):
    n = len(slots)
    free = range(n) if free is None else free
    i, f = np.full(8, -1, dtype=np.int64), np.zeros(8)
    f[:n] = slots
    theta = []
    for k in free:
        i[k] = len(theta)
        theta.append(slots[k])
    sources = [SourceSpec(type_, 0, (0, w, 0, h), False, i, f)]
    if sky is not None:
        j = np.full(8, -1, dtype=np.int64)
        j[0] = len(theta)
        theta.append(sky)
        sources.append(SourceSpec(O.SKY_FLAT, 0, (0, w, 0, h), False, j, np.zeros(8)))
    rng = np.random.default_rng(11)
    th = np.array(theta)
    return Problem("profile", [ImageSpec(h, w, np.eye(2), np.zeros(2))], sources, th.size, th, th,
                   quad_order=quad_order, noise=[rng.standard_normal((h, w))], var_floor=[1.0])


SERSICS = [(0.05, 30.0), (0.36, 5.0), (0.36, 60.0), (1.0, 0.5), (4.0, 5.0), (8.0, 0.5), (8.0, 60.0)]
MOFFATS = [(1.05, 0.5), (1.05, 30.0), (3.0, 5.0), (50.0, 0.5), (50.0, 30.0)]


def _value_bound(type_, n, R):
    """Relative error of a pixel's float32 value (one node, the pixel's centre):
    the coordinates' roundings, lg2.approx (2^-22 absolute for arguments in (0.5, 2),
    relative elsewhere), ex2.approx (2^-22 relative), carried through the exponents
    -- 1/(2n) and b t for a Sersic, n for a Moffat."""
    h, w = 41, 301
    eps, hw = 2.0 ** -24, 2.0 ** -22
    i, j = np.mgrid[0:h, 0:w]
    du, dv = np.abs(j + 0.5 - X0), np.abs(i + 0.5 - Y0)
    c, s = abs(math.cos(PA)) / R, abs(math.sin(PA)) / R
    u, e_u = 0.0, 0.0
    X = (math.cos(PA) * (j + 0.5 - X0) + math.sin(PA) * (i + 0.5 - Y0)) / R
    Y = (-math.sin(PA) * (j + 0.5 - X0) + math.cos(PA) * (i + 0.5 - Y0)) / (Q * R)
    for v, ex in ((X, 4 * eps * (c * du + s * dv) + 2 * eps * (c + s)),
                  (Y, (4 * eps * (s * du + c * dv) + 2 * eps * (c + s)) / Q)):
        u = u + v * v
        e_u = e_u + 2 * np.abs(v) * ex + ex * ex
    if type_ == O.SERSIC:
        u = u + 1e-8 / R ** 2
    else:
        u = u + 1.0
    e_u = e_u + 3 * eps * u
    L = np.log2(u)
    e_L = hw * np.maximum(1.0, np.abs(L)) + e_u / (u * math.log(2.0))
    if type_ == O.MOFFAT:
        return math.log(2.0) * (n * e_L + 2 * eps * n * np.abs(L)) + hw + 6 * eps
    b = O.sersic_b(n)
    t = u ** (0.5 / n)
    e_t = math.log(2.0) * (0.5 / n * e_L + 2 * eps * 0.5 / n * np.abs(L)) + hw
    return b * t * e_t + 3 * eps * b * (1.0 + t) + hw + 6 * eps


@pytest.mark.parametrize("type_,n,R", [(O.SERSIC, *p) for p in SERSICS] + [(O.MOFFAT, *p) for p in MOFFATS])
def test_profile_values_within_the_float32_bound(type_, n, R):
    slots = [X0, Y0, Q, PA, n, R, 100.0]
    pr = with_data(_problem(type_, slots))
    got = _np(device_context(pr, "mixed").render(pr.theta_init)[0])
    ref = O.model_images(pr, pr.theta_init)[0]
    bound = _value_bound(type_, n, R) * ref + 1e-36 * max(ref.max(), 1.0)   # (results below 2^-126 are flushed)
    worst = (np.abs(got - ref) / bound).max()
    assert worst <= 1.0, worst


@pytest.mark.parametrize("type_,n,R", [(O.SERSIC, *p) for p in SERSICS[1:]] + [(O.MOFFAT, *p) for p in MOFFATS])
def test_profile_gradients_at_steep_and_flat_profiles(type_, n, R):
    """The gradient over all slots, within the tolerance of the other float32 comparisons."""
    pr = with_data(_problem(type_, [X0, Y0, Q, PA, n, R, 100.0], quad_order=3))
    ctx = device_context(pr, "mixed")
    theta = pr.theta_init * (1.0 + 0.01 * np.array([1, -1, 1, -1, 1, -1, 1]))
    if type_ == O.SERSIC:
        theta[4] = max(theta[4], 0.36)
    _, g = ctx.eval(theta)
    assert_grad_close(_np(g), O.gradient(pr, theta), grad_scale(pr, theta), TOL_GRAD)
    assert ctx.status() == 0


TINY = [(O.GAUSSIAN, R, None) for R in (1e-6, 1e-12, 1e-14, 1e-16, 1e-18)] + \
       [(O.MOFFAT, R, None) for R in (1e-6, 1e-12, 1e-14, 1e-16)] + [(O.MOFFAT, 1e-18, (0, 1, 2, 3, 5, 6))]


@pytest.mark.parametrize("type_,R,free", TINY)
def test_gradient_of_a_source_far_smaller_than_a_pixel(type_, R, free):
    """A star whose radius has run off to nothing between the quadrature nodes:
    its derivatives vanish (the coefficients in front of them, F / R^3, pass
    float32's range), and they stay numbers."""
    slots = [X0, Y0, Q, PA, R, 100.0] if type_ == O.GAUSSIAN else [X0, Y0, Q, PA, 2.5, R, 100.0]
    pr = _problem(type_, slots, h=40, w=44, free=free, sky=1.0, quad_order=3)
    rng = np.random.default_rng(2)
    im = pr.images[0]
    im.data = (1.0 + rng.standard_normal((40, 44))).astype(np.float32)
    im.variance = np.ones((40, 44), dtype=np.float32)
    ctx = device_context(pr, "mixed")
    c, g = ctx.eval(pr.theta_init)
    jtwr, csr = ctx.normal_eq(pr.theta_init)
    g, M = _np(g), ctx.jtwj_dense(csr)
    with np.errstate(all="ignore"):
        want = O.gradient(pr, pr.theta_init)
    assert np.isfinite(g).all() and np.isfinite(_np(jtwr)).all() and np.isfinite(M).all(), (g, M)
    assert abs(g[-1] - want[-1]) <= TOL_GRAD * grad_scale_of_sky(pr)
    np.testing.assert_allclose(g[:-1], 0.0, atol=1e-6)
    assert np.isfinite(_np(c)).all()


def grad_scale_of_sky(pr):
    return 2.0 * np.abs(pr.images[0].data - 1.0).sum()


@pytest.mark.parametrize("R", [1e-3, 1e-5, 1e-8, 1e-12])
def test_gradient_of_the_wings_of_a_tiny_moffat(R):
    """(1 + u)^-1.2 falls off slowly: its wings carry light and derivatives for any radius."""
    pr = with_data(_problem(O.MOFFAT, [X0, Y0, Q, PA, 1.2, R, 100.0 * R ** -0.4], h=40, w=44, sky=1.0, quad_order=3))
    ctx = device_context(pr, "mixed")
    theta = pr.theta_init * (1.0 + 0.01 * np.array([1, -1, 1, -1, 1, -1, 1, 1]))
    _, g = ctx.eval(theta)
    assert_grad_close(_np(g), O.gradient(pr, theta), grad_scale(pr, theta), TOL_GRAD)
    assert ctx.status() == 0


@pytest.mark.parametrize("type_", [O.GAUSSIAN, O.MOFFAT])
def test_a_position_that_is_no_number_stays_one(type_):
    """A fixed centre that is NaN reaches every entry of a free radius and flux, and the status word."""
    from paper_2308_01957_gb300 import _lib
    slots = [math.nan, Y0, Q, PA, 2.0, 100.0] if type_ == O.GAUSSIAN else [math.nan, Y0, Q, PA, 2.5, 2.0, 100.0]
    pr = _problem(type_, slots, h=24, w=24, free=(len(slots) - 2, len(slots) - 1), sky=1.0)
    pr.images[0].data = np.ones((24, 24), dtype=np.float32)
    pr.images[0].variance = np.ones((24, 24), dtype=np.float32)
    ctx = device_context(pr, "mixed")
    _, csr = ctx.normal_eq(pr.theta_init)
    M = ctx.jtwj_dense(csr)
    assert np.isnan(M[:2, :2]).all() and np.isfinite(M[2, 2]), M
    assert ctx.status() == _lib.AP_ERR_NONFINITE
