"""The one-block AIC solve against numpy at its sizes: the smallest, the edges of its 32-row steps, its largest and
the first order beyond it; the refinement's stopping rules and the ways out of it."""
import numpy as np
import pytest

from tests._util import to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_11430_gb300 import api as a
    from paper_2511_11430_gb300 import build

    build.build()
    return a


def _system(n, dominant=True, seed=0):
    rng = np.random.default_rng(seed)
    A = rng.normal(size=(n, n))
    if dominant:
        off = np.abs(A).sum(1) - np.abs(np.diag(A))
        A[np.diag_indices(n)] = np.where(rng.random(n) < 0.5, -1, 1) * (1.3 * off + 0.1)
    return A.astype(np.float32), rng.normal(size=n)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 160, 191, 192, 193, 223, 224, 225])
@pytest.mark.parametrize("dominant", [True, False])
def test_solution_and_backward_error(api, n, dominant):
    A, b = _system(n, dominant, seed=n)
    x, it, be = api.aic_solve(to_dev(A), to_dev(b), tol=1e-12, max_iter=30)
    assert be <= 1e-12 and it <= (3 if dominant else 30)
    ref = np.linalg.solve(A.astype(np.float64), b)
    x = x.cpu().numpy()
    # backward error 1e-12 times the condition number, in the 2-norm
    cond = np.linalg.cond(A.astype(np.float64))
    assert np.linalg.norm(x - ref) <= max(1e-11, 1e-11 * n * cond) * np.linalg.norm(ref)


def test_not_converged_returns_the_best_iterate(api):
    A, b = _system(100, seed=3)
    x, it, be = api.aic_solve(to_dev(A), to_dev(b), tol=0.0, max_iter=3, raise_on_fail=False)
    assert it == 3 and be < 1e-14
    with pytest.raises(Exception):
        api.aic_solve(to_dev(A), to_dev(b), tol=0.0, max_iter=3)
    x0, it0, be0 = api.aic_solve(to_dev(A), to_dev(b), tol=0.0, max_iter=0, raise_on_fail=False)
    assert it0 == 0 and 1e-12 < be0 < 1e-5


def test_non_finite_input_is_reported(api):
    A, b = _system(50, seed=4)
    b[7] = np.nan
    _, _, be = api.aic_solve(to_dev(A), to_dev(b), raise_on_fail=False)
    assert not np.isfinite(be)
    A[3, 4] = np.inf
    with pytest.raises(Exception):
        api.aic_solve(to_dev(A), to_dev(np.ones(50)))
