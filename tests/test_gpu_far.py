"""The tensor-core far sweep (csrc/vpm_far.cuh) against the FP64 oracle where it can go wrong: at the sizes
where it starts, ragged tiles and groups, few targets, sources at the edge of the acceptance test, scales,
and non-finite sources.  Tolerances are those of the pair sums."""
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


def _f32(a):
    return np.ascontiguousarray(a, dtype=np.float32)


def _pad(x):
    return _f32(np.concatenate([x, np.zeros((len(x), 1))], 1))


def _check(api, pos, G, tgt, sigma, compensated=True, k=96):
    P, S, T = to_dev(pos), to_dev(G), to_dev(tgt)
    u, g = api.induce(P, S, T, sigma, compensated=compensated)
    uv = api.induce(P, S, T, sigma, compensated=compensated, grad=False)
    torch.cuda.synchronize()
    assert api.device_error() == 0
    idx = np.unique(np.concatenate([[0, len(tgt) - 1], synth.sample_targets(5, len(tgt), k)]))
    ru, rJ = oracle.p2p(pos, G, tgt[idx], sigma)
    tol = TOL_COMP if compensated else TOL_PLAIN
    rows = lambda t: t[:, idx].double().cpu().numpy().T
    assert rel_l2(rows(u), ru) <= tol
    assert rel_l2(rows(g).reshape(-1, 3, 3), rJ) <= tol
    assert rel_l2(rows(uv), ru) <= tol


@pytest.mark.parametrize("n", [16383, 16384, 17000, 20011, 30721])
@pytest.mark.parametrize("compensated", [True, False])
def test_wake_sizes(api, n, compensated):
    w = synth.multirotor(seed=3, n=n)
    _check(api, w.pos, w.strength, w.pos, w.sigma, compensated)


@pytest.mark.parametrize("n_src,n_tgt", [(280_000, 1), (262_145, 257), (140_001, 1280), (129, 1_100_000), (1, 2_100_000)])
def test_unequal_counts(api, n_src, n_tgt):
    w = synth.hover(seed=4, n=max(n_src, 4))
    rng = np.random.default_rng(2)
    tgt = _pad(rng.uniform([-1, -1, -1.2], [1, 1, 0.4], size=(n_tgt, 3)))
    _check(api, w.pos[:n_src], w.strength[:n_src], tgt, w.sigma)


@pytest.mark.parametrize("dist", [1.95, 2.02, 2.3, 6.0, 400.0])
@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e3])
def test_compact_clouds_at_the_acceptance_edge(api, dist, scale):
    """Every tile spans the whole cloud; the targets lie just inside or outside the acceptance distance (twice
    the radius), so no averaging over far tiles hides the error of a pair."""
    rng = np.random.default_rng(7)
    n, m = 1024, 270_336
    x = rng.normal(size=(n, 3))
    x = x / np.linalg.norm(x, axis=1, keepdims=True) * rng.uniform(0, 1, size=(n, 1)) ** (1 / 3)
    e = rng.normal(size=(m, 3))
    # targets in a small cap, so that the groups' boxes are small too
    y = np.array([dist, 0, 0]) + 0.01 * e / np.linalg.norm(e, axis=1, keepdims=True)
    G = rng.normal(size=(n, 3)) + np.array([0.0, 0.0, 2.0])
    _check(api, _pad(scale * x), _pad(1e-3 * scale * G), _pad(scale * y), 0.02 * scale)


@pytest.mark.parametrize("kind", ["point", "zero", "one_strong", "offset"])
def test_degenerate_tiles(api, kind):
    w = synth.hover(seed=5, n=60_000)
    pos, G = w.pos.copy(), w.strength.copy()
    if kind == "point":  # a whole tile (and more) at one point: radius zero
        pos[1000:1400, :3] = pos[1000, :3]
    elif kind == "zero":
        G[5000:9000] = 0.0
    elif kind == "one_strong":
        G[::97] *= 1e4
    else:
        pos[:, :3] += np.float32([40.0, -25.0, 10.0])
    _check(api, pos, G, pos, w.sigma)


def test_non_finite_source_stays_non_finite(api):
    """A source with a non-finite strength reaches every target, as in the pair sweep."""
    w = synth.hover(seed=6, n=60_000)
    G = w.strength.copy()
    G[12345, 1] = np.inf
    u, g = api.induce(to_dev(w.pos), to_dev(G), to_dev(w.pos), w.sigma)
    far = np.linalg.norm(w.pos[:, :3] - w.pos[12345, :3], axis=1) > 0.2
    assert not torch.isfinite(u[:, torch.from_numpy(far).cuda()].sum(0)).any()


def test_stretching_of_far_units(api):
    """The transposed and the classic stretching at sampled particles, whose far part is formed from the far sums."""
    w = synth.multirotor(seed=8, n=40_000)
    idx = synth.sample_targets(3, w.n, 64)
    u, J = oracle.p2p(w.pos, w.strength, w.pos[idx], w.sigma)
    us, Js = oracle.segments(w.seg_a, w.seg_b, w.pos[idx], w.seg_core, 2)
    for classic in (False, True):
        prm = api.Params(sigma=w.sigma, nu=0.0, c_v=0.0, seg_core=w.seg_core, classic=classic)
        dx, dG, _ = api.rhs(to_dev(w.pos), to_dev(w.strength), to_dev(w.seg_a), to_dev(w.seg_b), prm)
        ref = oracle.stretch(J + Js, w.strength[idx], classic)
        assert rel_l2(dx[:, idx].double().cpu().numpy().T, u + us) <= TOL_COMP
        assert rel_l2(dG[:, idx].double().cpu().numpy().T, ref) <= TOL_COMP


@pytest.mark.parametrize("n,k", [(115_300, 1000), (30_721, 4000), (930_000, 1), (460_801, 129)])
@pytest.mark.parametrize("compensated", [True, False])
def test_adjoint_by_the_sweep(api, n, k, compensated):
    """The adjoint of a problem large enough for the tensor cores: the particle sweep with the points as sources."""
    w = synth.multirotor(seed=9, n=n)
    rng = np.random.default_rng(4)
    pts = _pad(rng.uniform([-2, -1, -0.6], [2, 1, 0.3], size=(k, 3)))
    pts[0, :3] = w.pos[n // 2, :3]  # a point on a particle: nothing from that pair
    g = _f32(rng.normal(size=(3, k)))
    dx, dG = api.induce_backward(to_dev(w.pos), to_dev(w.strength), to_dev(pts), w.sigma, to_dev(g),
                                 compensated=compensated)
    torch.cuda.synchronize()
    assert api.device_error() == 0
    idx = np.unique(np.concatenate([[0, n // 2, n - 1], synth.sample_targets(6, n, 3000)]))
    rx, rG = oracle.p2p_adjoint(w.pos[idx], w.strength[idx], pts, w.sigma, g.T)
    tol = 1e-5 if compensated else 1e-3
    assert rel_l2(dx[:, idx].double().cpu().numpy().T, rx) <= tol
    assert rel_l2(dG[:, idx].double().cpu().numpy().T, rG) <= tol
