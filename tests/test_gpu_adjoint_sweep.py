"""The adjoint that runs as a particle sweep with the evaluation points as sources (csrc/vpm_adjoint.cu), where
that sweep's conveniences for particles among themselves must not reach it."""
import numpy as np
import pytest

import oracle
from paper_2511_11430_gb300 import synth
from tests._util import rel_l2, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL_ADJOINT = 1e-5  # as in the other adjoint tests


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_11430_gb300 import api as a
    from paper_2511_11430_gb300 import build

    build.build()
    return a


def _check(dx, dG, w, pts, g, extra=()):
    idx = np.unique(np.concatenate([[0, w.n - 1], synth.sample_targets(6, w.n, 300), extra])).astype(np.int64)
    rx, rG = oracle.p2p_adjoint(w.pos[idx], w.strength[idx], pts, w.sigma, g.T)
    rows = lambda t: t[:, idx].double().cpu().numpy().T
    assert rel_l2(rows(dG), rG) <= TOL_ADJOINT
    assert rel_l2(rows(dx), rx) <= TOL_ADJOINT


@pytest.mark.parametrize("scale", [1e3, 1.0, 1e-3, 1e-6, 1e-9, 1e-12])
def test_loss_gradient_of_any_scale(api, scale):
    """|g| against |Gamma| ~ 1e-3: the two are unrelated quantities, and dL/dx is linear in both.  The points lie
    in the wake, half of them within a core of a particle."""
    w = synth.multirotor(seed=9, n=115_300)
    rng = np.random.default_rng(4)
    pts = w.pos[rng.integers(0, w.n, size=1000)].copy()
    pts[:, :3] += (rng.normal(size=(1000, 3)) * 0.5 * w.sigma).astype(np.float32)
    near = np.argmin(((w.pos[:, None, :3] - pts[None, :8, :3]) ** 2).sum(2), axis=0)
    g = np.ascontiguousarray(rng.normal(size=(3, 1000)) * scale, dtype=np.float32)
    dx, dG = api.induce_backward(to_dev(w.pos), to_dev(w.strength), to_dev(pts), w.sigma, to_dev(g))
    assert api.device_error() == 0
    _check(dx, dG, w, pts, g, near)


@pytest.mark.parametrize("n", [16_383, 16_384, 20_011])
@pytest.mark.parametrize("alias", [True, False])
def test_particles_as_their_own_points(api, n, alias):
    """The points are the particles, in the same tensor or in a copy: in the first case the sweep puts sources
    and targets in curve order, and the strengths that enter are still the particles', not the loss gradient."""
    from paper_2511_11430_gb300 import autograd

    w = synth.multirotor(seed=9, n=n)
    P, S = to_dev(w.pos).requires_grad_(True), to_dev(w.strength).requires_grad_(True)
    g = np.ascontiguousarray(np.random.default_rng(5).normal(size=(3, n)), dtype=np.float32)
    u = autograd.induce(P, S, P.detach() if alias else P.detach().clone(), w.sigma)
    dP, dS = torch.autograd.grad(u, (P, S), to_dev(g))
    assert api.device_error() == 0
    _check(dP[:, :3].t(), dS[:, :3].t(), w, w.pos, g)
