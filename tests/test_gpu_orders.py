"""Particles in no order, and strays, at sizes that take the tensor-core sweep's lists: the answers are those of the
generators' order, against the FP64 oracle at the tolerances of the sums."""
import numpy as np
import pytest

import oracle
from paper_2511_11430_gb300 import synth
from tests._util import TOL_COMP, TOL_PLAIN, rel_l2, to_dev

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


def _wake(n, stray, name="hover"):
    """A wake in no order; `stray`: three particles that many metres off."""
    w = getattr(synth, name)(seed=7, n=n)
    p = np.random.default_rng(3).permutation(n)
    w.pos, w.strength = np.ascontiguousarray(w.pos[p]), np.ascontiguousarray(w.strength[p])
    if stray:
        w.pos[[5, n // 2, n - 1], :3] += np.float32(stray) * np.float32([[1, 0.3, -0.5], [-0.2, 1, 0], [0, -1, 0.7]])
    return w


@pytest.mark.parametrize("stray", [0.0, 1000.0])
@pytest.mark.parametrize("n,compensated", [(16_384, True), (17_003, True), (17_003, False), (60_001, True)])
def test_velocity_and_gradient(api, n, compensated, stray):
    w = _wake(n, stray)
    P, S = to_dev(w.pos), to_dev(w.strength)
    idx = np.unique(np.concatenate([[5, n // 2, n - 1], synth.sample_targets(5, n, 96)]))
    ru, rJ = oracle.p2p(w.pos, w.strength, w.pos[idx], w.sigma)
    tol = TOL_COMP if compensated else TOL_PLAIN
    rows = lambda t: t[:, idx].double().cpu().numpy().T
    for tgt in (P, P.clone()):  # the particles themselves, and points of their own
        u, g = api.induce(P, S, tgt, w.sigma, compensated=compensated)
        uv = api.induce(P, S, tgt, w.sigma, compensated=compensated, grad=False)
        assert rel_l2(rows(u), ru) <= tol and rel_l2(rows(uv), ru) <= tol
        assert rel_l2(rows(g).reshape(-1, 3, 3), rJ) <= tol
    assert api.device_error() == 0


@pytest.mark.parametrize("stray", [0.0, 1000.0])
def test_right_hand_side(api, stray):
    n = 20_011
    w = _wake(n, stray)
    prm = api.Params(sigma=w.sigma, nu=w.nu, c_v=0.0, seg_core=w.seg_core, u_inf=w.u_inf)
    dx, dG, _ = api.rhs(to_dev(w.pos), to_dev(w.strength), to_dev(w.seg_a), to_dev(w.seg_b), prm)
    idx = synth.sample_targets(5, n, 200)
    u, J = oracle.p2p(w.pos, w.strength, w.pos[idx], w.sigma)
    us, Js = oracle.segments(w.seg_a, w.seg_b, w.pos[idx], w.seg_core, 2)
    ref = oracle.stretch(J + Js, w.strength[idx], False) + oracle.pse_at(w.pos, w.strength, np.zeros(n), w.sigma, w.nu, idx)
    assert rel_l2(dx[:, idx].double().cpu().numpy().T, u + us + np.asarray(w.u_inf)) <= TOL_COMP
    assert rel_l2(dG[:, idx].double().cpu().numpy().T, ref) <= TOL_COMP
    assert api.device_error() == 0


def test_adjoint(api):
    n, k = 120_011, 1280
    w = _wake(n, 0.0)
    rng = np.random.default_rng(4)
    pts = np.zeros((k, 4), dtype=np.float32)
    pts[:, :3] = rng.uniform([-1, -1, -1.2], [1, 1, 0.4], size=(k, 3))
    g = np.ascontiguousarray(rng.normal(size=(3, k)), dtype=np.float32)
    dx, dG = api.induce_backward(to_dev(w.pos), to_dev(w.strength), to_dev(pts), w.sigma, to_dev(g))
    idx = synth.sample_targets(6, n, 2000)
    rx, rG = oracle.p2p_adjoint(w.pos[idx], w.strength[idx], pts, w.sigma, g.T)
    assert rel_l2(dx[:, idx].double().cpu().numpy().T, rx) <= 1e-5
    assert rel_l2(dG[:, idx].double().cpu().numpy().T, rG) <= 1e-5
    assert api.device_error() == 0


def _rhs_tree(api, w):
    P, S, a, b = (to_dev(x) for x in (w.pos, w.strength, w.seg_a, w.seg_b))
    prm = api.Params(sigma=w.sigma, nu=w.nu, c_v=w.c_v, seg_core=w.seg_core, u_inf=w.u_inf)
    ws = api.Workspace("cuda")
    run = lambda: api.rhs_tree(P, S, a, b, prm, theta=0.5, order=4, ws=ws)
    out = run()
    t = []
    for _ in range(3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record()
        run()
        e1.record()
        torch.cuda.synchronize()
        t.append(e0.elapsed_time(e1))
    return out, min(t)


def test_tree_exchange_with_strays(api):
    """The treecode's exchange takes the particles in curve order.  Three of them a thousand metres off must not
    leave the rest in a few of the curve's cells: in no order every tile reaches every particle, and the call took
    seven times as long.  (The tree itself differs with the strays, so the times are only of one size.)"""
    n = 600_000
    (_, dG, _), t0 = _rhs_tree(api, _wake(n, 0.0, "multirotor"))
    w = _wake(n, 1000.0, "multirotor")
    (_, dGs, nut), t1 = _rhs_tree(api, w)
    assert t1 < 4.0 * t0, (t0, t1)
    # the exchange itself, at sampled particles: what nu adds to dGamma/dt
    P, S, a, b = (to_dev(x) for x in (w.pos, w.strength, w.seg_a, w.seg_b))
    prm = lambda nu: api.Params(sigma=w.sigma, nu=nu, c_v=0.0, seg_core=w.seg_core, u_inf=w.u_inf)
    big = 1.0  # so that the exchange outweighs the stretching, whose difference cancels but for rounding
    d = api.rhs_tree(P, S, a, b, prm(big))[1] - api.rhs_tree(P, S, a, b, prm(0.0))[1]
    idx = synth.sample_targets(5, n, 200)
    ref = oracle.pse_at(w.pos, w.strength, np.zeros(n), w.sigma, big, idx)
    assert rel_l2(d[:, idx].double().cpu().numpy().T, ref) <= 1e-5
    assert api.device_error() == 0


@pytest.mark.parametrize("n", [65, 128, 129, 4_096, 4_097, 65_537])
def test_tree_exchange_at_the_edges_of_tiles_and_groups(api, n):
    """Tiles of 128 particles, groups of 32 tiles; a cloud about a core size apart, so that every size has pairs
    within the exchange's 7 core sizes."""
    sigma = n ** (-1.0 / 3.0)
    pos, G = synth.random_cloud(3, n, box=1.0, sigma=sigma)
    P, S = to_dev(pos), to_dev(G)
    none = torch.empty((0, 4), dtype=torch.float32, device="cuda")
    prm = lambda nu: api.Params(sigma=sigma, nu=nu, c_v=0.0)
    d = api.rhs_tree(P, S, none, none, prm(1.0))[1] - api.rhs_tree(P, S, none, none, prm(0.0))[1]
    idx = np.unique(np.concatenate([[0, n - 1], synth.sample_targets(5, n, min(n, 200))]))
    ref = oracle.pse_at(pos, G, np.zeros(n), sigma, 1.0, idx)
    assert rel_l2(d[:, idx].double().cpu().numpy().T, ref) <= 1e-5
    assert api.device_error() == 0
