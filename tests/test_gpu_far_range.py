"""The tensor-core far sweep over the whole range of FP32 values that the pair sweep takes, against the FP64 oracle
at the tolerances of the pair sums."""
import numpy as np
import pytest

import oracle
from paper_2511_11430_gb300 import synth
from tests._util import TOL_COMP, rel_l2, to_dev

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


def _check(api, pos, G, tgt, sigma, idx):
    P, S, T = to_dev(pos), to_dev(G), to_dev(tgt)
    u, g = api.induce(P, S, T, sigma)
    uv = api.induce(P, S, T, sigma, grad=False)
    assert api.device_error() == 0
    ru, rJ = oracle.p2p(pos, G, tgt[idx], sigma)
    rows = lambda t: t[:, idx].double().cpu().numpy().T
    assert rel_l2(rows(u), ru) <= TOL_COMP
    assert rel_l2(rows(uv), ru) <= TOL_COMP
    assert rel_l2(rows(g).reshape(-1, 3, 3), rJ) <= TOL_COMP


@pytest.mark.parametrize("size", [1e30, 1e-28, 1e-30, 1e-31, 1e-34])
def test_strengths_of_any_size(api, size):
    """Strengths of about `size`: the features' FP16 pairs are scaled by the tile's largest."""
    w = synth.hover(seed=5, n=60_000)
    G = np.float32(w.strength * (size / 1e-3))
    _check(api, w.pos, G, w.pos, w.sigma, synth.sample_targets(5, w.n, 96))


@pytest.mark.parametrize("d", [1e18, 3e19, 1e30, 1e37])
@pytest.mark.parametrize("which", ["sources", "targets", "both"])
def test_distances_whose_squares_overflow(api, d, which):
    """200 particles so far off that r^2 is not finite in FP32 (from 1.8e19): they contribute nothing to the
    others and the others nothing to them."""
    w = synth.hover(seed=5, n=60_000)
    off = w.pos.copy()
    off[:200, 0] += np.float32(d)
    src, tgt = (w.pos if which == "targets" else off), (w.pos if which == "sources" else off)
    idx = np.concatenate([np.arange(0, 200, 20), 200 + synth.sample_targets(5, w.n - 200, 96)])
    _check(api, src, w.strength, tgt, w.sigma, idx)
