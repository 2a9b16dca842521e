"""The sums of J^T W J over tiles: past float32's range, and at the sizes where
their form changes (pairs of up to 2048 values, runs of up to 8192 values, tiles of
up to 22 sources)."""
import numpy as np
import pytest

from _helpers import O, TOL_GRAD, configs, device_context, with_data
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


def _check_jtwj(pr, tol=TOL_GRAD, **options):
    from paper_2308_01957_gb300 import api
    ctx = api.Context("mixed", pr.quad_order, device=0, **options)
    ctx.set_problem(api.to_device_images(pr.images), pr.sources, pr.n_params)
    ref, _ = O.normal_equations(pr, pr.theta_init)
    _, csr = ctx.normal_eq(pr.theta_init)
    JtWJ = ctx.jtwj_dense(csr)
    d = np.sqrt(np.maximum(np.diag(ref), 1e-300))
    assert (np.abs(JtWJ - ref) / np.outer(d, d)).max() <= tol
    assert ctx.status() == 0
    return csr


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


@pytest.mark.parametrize("n_tiles", [227, 228, 910, 911, 1821])
@pytest.mark.parametrize("shared", [False, True])
def test_pair_sums_at_run_boundaries(n_tiles, shared):
    """A strip of n 16 x 16 tiles under a plane sky (9 values per tile: 2043 and
    2052 values on both sides of a warp's 2048; 910 tiles fill a run of 8192
    values, 911 start a second, 1821 a third) and a star; shared: two such strips
    with the same parameters, whose pairs add to the same entries."""
    h, w = 16, 16 * n_tiles
    rng = np.random.default_rng(n_tiles)
    images, sources = [], []
    for k in range(2 if shared else 1):
        images.append(ImageSpec(h, w, np.eye(2), np.array([-0.5 * w, -8.0]),
                                data=rng.standard_normal((h, w)).astype(np.float32),
                                variance=rng.uniform(0.5, 1.5, (h, w)).astype(np.float32)))
        sources.append(_source(O.SKY_PLANE, k, (0, w, 0, h), [0, 1, 2]))
        sources.append(_source(O.GAUSSIAN, k, (3, 40, 0, h), [3, 4, -1, -1, -1, 5], [0.0, 0.0, 0.7, 0.4, 2.5, 0.0]))
    theta = np.array([1.0, 1e-3, -2e-3, -0.5 * w + 20.4, 0.7, 50.0])
    _check_jtwj(Problem("strip", images, sources, 6, theta, theta))


@pytest.mark.parametrize("nm", [20, 21])
def test_tiles_at_the_staged_pair_limit(nm):
    """A tile of 22 sources (253 pairs, offsets kept in shared memory) and one of 23 (276, read in place)."""
    pr = with_data(configs.crowded_field(f"pairs_{nm}", configs.SEED_BASE + 97, 16, 16, 1, nm, configs.psf_moffat(5, 2.5)))
    assert len(pr.sources) == nm + 2
    _check_jtwj(pr)


def test_gram_tc_min_changes_nothing():
    """The option is still accepted (a negative one refused): the same entries bit by bit."""
    from paper_2308_01957_gb300 import api
    from paper_2308_01957_gb300._lib import ApError
    pr = with_data(configs.crowded_field("graded_tiles", configs.SEED_BASE + 72, 96, 160, 12, 20,
                                         configs.psf_moffat(5, 2.5)))
    vals = [_check_jtwj(pr, jcol="direct", conv_variant=1, gram_tc_min=m)[2] for m in (0, 1, 257)]
    assert torch.equal(vals[0], vals[1]) and torch.equal(vals[0], vals[2])
    with pytest.raises(ApError):
        api.Context("mixed", pr.quad_order, device=0, gram_tc_min=-1)
