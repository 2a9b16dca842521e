"""Which state a Levenberg-Marquardt call starts from when evaluations were
captured in CUDA graphs since the last one: always the model at its own theta."""
import numpy as np
import pytest

from _helpers import device_context, problem
from _helpers import configs

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


CALLS = {
    "eval": lambda ctx, th: ctx.eval(th),
    "render": lambda ctx, th: ctx.render(th),
    "normal_eq": lambda ctx, th: ctx.normal_eq(th),
    "eval_shifted": lambda ctx, th: ctx.eval_shifted(th),
}


@pytest.mark.parametrize("precision", ["mixed", "f64"])
@pytest.mark.parametrize("call", list(CALLS))
@pytest.mark.parametrize("replayed", [False, True])
@pytest.mark.parametrize("then", ["iterate", "continue"])
def test_evaluation_captured_after_a_fit(then, replayed, call, precision):
    """LM iterations, then an evaluation captured in a graph (and replayed or
    not), then (iterate) a fit from another theta, or (continue) a direct
    evaluation elsewhere and the first fit continued: the same accepts, chi^2 and
    theta as without the captured call."""
    pr = problem("mixed", seed=configs.SEED_BASE + 21, H=45, W=70, K=7)
    ctx = device_context(pr, precision)
    lam = np.full(pr.n_groups, 1e-3)
    other = 0.5 * (pr.theta_init + pr.theta_true)
    if then == "iterate":
        th_ref, _, c_ref, log_ref = ctx.lm_iterate(other, lam, 2, log=True)
    else:
        th_ref, _, c_ref, log_ref = ctx.lm_iterate(pr.theta_init, lam, 4, log=True)
        log_ref = log_ref[2:]
    theta = torch.as_tensor(pr.theta_true, dtype=torch.float64, device="cuda")
    CALLS[call](ctx, theta)
    ctx.lm_iterate(pr.theta_init, lam, 2)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        CALLS[call](ctx, theta)
    if replayed:
        graph.replay()
    if then == "iterate":
        th, _, c, log = ctx.lm_iterate(other, lam, 2, log=True)
    else:
        ctx.eval(other)
        th, _, c, log = ctx.lm_continue(2, log=True)
    np.testing.assert_array_equal(log[:, :, 3], log_ref[:, :, 3])
    np.testing.assert_allclose(log[:, :, :2], log_ref[:, :, :2], rtol=1e-12)
    np.testing.assert_allclose(_np(c), _np(c_ref), rtol=1e-12)
    np.testing.assert_allclose(_np(th), _np(th_ref), rtol=1e-10, atol=1e-12)
    assert ctx.status() == 0
