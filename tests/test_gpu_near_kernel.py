"""The near pairs' blob kernel (near_kh2 of csrc/vpm_kernel.cuh) pair by pair, from a thousandth of a core to beyond
the 7 core sizes where the point-vortex form takes over."""
import numpy as np
import pytest

import oracle
from tests._util import to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -24
# K and h: within 3e-7 near (the fit and its evaluation); 3 and 5 times rsqrt.approx's 2^-22.9 beyond.  r^2: two
# roundings, with dlnK/dlnr^2 <= 3/2 and dlnh/dlnr^2 <= 5/2.  Then the cross product, the products and the sum.
TOL_U = max(3e-7, 3 * 2.0 ** -22.9) + 3 * EPS + 4 * EPS
TOL_J = 2 * (max(3e-7, 5 * 2.0 ** -22.9) + 5 * EPS + 6 * EPS)  # two terms of like size


@pytest.mark.parametrize("sigma", [0.0125, 1.0, 30.0])
@pytest.mark.parametrize("compensated", [True, False])
def test_single_pairs(sigma, compensated):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_11430_gb300 import api, build

    build.build()
    rng = np.random.default_rng(1)
    rho = np.concatenate([np.geomspace(1e-3, 12.0, 6000), np.linspace(6.9, 7.1, 500), [7.0]])
    e = rng.normal(size=(len(rho), 3))
    tgt = np.zeros((len(rho), 4), dtype=np.float32)
    tgt[:, :3] = sigma * rho[:, None] * e / np.linalg.norm(e, axis=1, keepdims=True)
    pos = np.zeros((1, 4), dtype=np.float32)
    G = np.array([[0.3, -0.7, 0.5, 0.0]], dtype=np.float32)
    u, g = api.induce(to_dev(pos), to_dev(G), to_dev(tgt), sigma, compensated=compensated)
    uv = api.induce(to_dev(pos), to_dev(G), to_dev(tgt), sigma, compensated=compensated, grad=False)
    ru, rJ = oracle.p2p(pos, G, tgt, sigma)
    # per pair, against the size that the pair can have: |K| |Gamma| |r|, and |J| of the pair
    K = np.linalg.norm(ru, axis=1) / np.linalg.norm(np.cross(G[0, :3].astype(float), tgt[:, :3].astype(float)), axis=1)
    size = K * np.linalg.norm(G[0, :3]) * np.linalg.norm(tgt[:, :3].astype(float), axis=1)
    for v in (u, uv):
        assert (np.linalg.norm(v.double().cpu().numpy().T - ru, axis=1) / size).max() <= TOL_U
    dJ = np.abs(g.double().cpu().numpy().T.reshape(-1, 3, 3) - rJ).max((1, 2))
    assert (dJ / (2 * K * np.linalg.norm(G[0, :3]))).max() <= TOL_J
    assert api.device_error() == 0


@pytest.mark.parametrize("n", [300, 17_003])
@pytest.mark.parametrize("sigma", [1e-6, 1e-9, 1e-15, 1e-25])
def test_point_vortices(sigma, n):
    """Cores so small that sigma^-5, sigma^-3 or sigma^2 leave FP32: point vortices, none of which acts on itself
    or on one in the same place."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_11430_gb300 import api, build, synth
    from tests._util import TOL_COMP, rel_l2

    build.build()
    w = synth.hover(seed=2, n=n)
    pos = w.pos.copy()
    pos[10:20, :3] = pos[10, :3]
    idx = np.unique(np.concatenate([np.arange(8, 22), synth.sample_targets(5, n, 96)]))
    P, S = to_dev(pos), to_dev(w.strength)
    u, g = api.induce(P, S, P, sigma)
    uv = api.induce(P, S, P, sigma, grad=False)
    ru, rJ = oracle.p2p(pos, w.strength, pos[idx], sigma)
    rows = lambda t: t[:, idx].double().cpu().numpy().T
    assert rel_l2(rows(u), ru) <= TOL_COMP and rel_l2(rows(uv), ru) <= TOL_COMP
    assert rel_l2(rows(g).reshape(-1, 3, 3), rJ) <= TOL_COMP
    assert api.device_error() == 0
