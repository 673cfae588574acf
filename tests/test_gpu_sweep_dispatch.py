"""The pair sweep where its plan changes form: teams of four warps or whole blocks, for particle and for segment
tiles, both kinds of tile in one launch or two, and ragged counts about the teams' 256 targets and 64 sources,
against the FP64 oracle at the tolerances of the pair sums."""
import ctypes

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


def _targets(n, seed=3):
    rng = np.random.default_rng(seed)
    x = rng.uniform([-1, -1, -1.2], [1, 1, 0.4], size=(n, 3))
    return np.ascontiguousarray(np.concatenate([x, np.zeros((n, 1))], 1), dtype=np.float32)


def _idx(n):
    return np.unique(np.concatenate([[0, n - 1], synth.sample_targets(5, n, 64)])) if n > 64 else np.arange(n)


def _close(u, g, ru, rJ, idx, tol):
    rows = lambda t: t[:, idx].double().cpu().numpy().T
    assert rel_l2(rows(u), ru) <= tol
    assert rel_l2(rows(g).reshape(-1, 3, 3), rJ) <= tol


@pytest.mark.parametrize("n_src,n_tgt", [(1, 1), (63, 255), (64, 256), (65, 257), (129, 1023), (2000, 1025), (15000, 300)])
@pytest.mark.parametrize("compensated", [True, False])
def test_team_edges(api, n_src, n_tgt, compensated):
    w = synth.hover(seed=2, n=max(n_src, 4))
    pos, G, tgt = w.pos[:n_src], w.strength[:n_src], _targets(n_tgt)
    idx = _idx(n_tgt)
    u, g = api.induce(to_dev(pos), to_dev(G), to_dev(tgt), w.sigma, compensated=compensated)
    _close(u, g, *oracle.p2p(pos, G, tgt[idx], w.sigma), idx, TOL_COMP if compensated else TOL_PLAIN)
    assert api.device_error() == 0


@pytest.mark.parametrize("n_src", [127 * 128, 128 * 128])
def test_teams_or_blocks_without_a_workspace(api, n_src):
    """16,256 and 16,384 units of 1,024 targets by 128 sources: the first with teams, the second with whole
    blocks (on this route never on the tensor cores)."""
    from paper_2511_11430_gb300 import _lib

    lib = _lib.load()
    w = synth.hover(seed=4, n=n_src)
    n_tgt = 128 * 1024
    tgt = _targets(n_tgt)
    P, S, T = to_dev(w.pos), to_dev(w.strength), to_dev(tgt)
    u = torch.full((3, n_tgt), float("nan"), device="cuda")
    g = torch.full((9, n_tgt), float("nan"), device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    st = lib.vpm_induce_noalloc(p(P), p(S), n_src, p(T), n_tgt, ctypes.c_float(w.sigma), 1, p(u), p(g),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0, lib.vpm_last_error()
    idx = _idx(n_tgt)
    _close(u, g, *oracle.p2p(w.pos, w.strength, tgt[idx], w.sigma), idx, TOL_COMP)
    assert api.device_error() == 0


@pytest.mark.parametrize("m", [1, 65, 127 * 128, 128 * 128])
def test_segments_by_teams_or_blocks(api, m):
    """508 and 512 units of segment tiles on 4,096 targets; closed rings and, for odd counts, single segments."""
    w = synth.hover(seed=5, n=4)
    rep = -(-m // w.m)
    shift = np.repeat(np.float32(0.01) * np.arange(rep, dtype=np.float32), w.m)[:m]
    sa, sb = np.tile(w.seg_a, (rep, 1))[:m].copy(), np.tile(w.seg_b, (rep, 1))[:m].copy()
    sa[:, 2] -= shift
    sb[:, 2] -= shift
    tgt = _targets(4096)
    idx = np.arange(4096)  # all: the far field of a few closed rings cancels, so a sample has no scale of its own
    u, g = api.segments_induce(to_dev(sa), to_dev(sb), to_dev(tgt), w.seg_core, 2, compensated=True)
    _close(u, g, *oracle.segments(sa, sb, tgt[idx], w.seg_core, 2), idx, TOL_COMP)
    assert api.device_error() == 0


@pytest.mark.parametrize("m", [1024, 1028])
def test_one_launch_or_two_for_the_segments(api, m):
    """Eight segment tiles go with the particle tiles, nine have their own launch."""
    w = synth.hover(seed=6, n=3000)
    sa, sb = w.seg_a[:m], w.seg_b[:m]
    prm = api.Params(sigma=w.sigma, nu=0.0, c_v=0.0, seg_core=w.seg_core)
    dx, dG, _ = api.rhs(to_dev(w.pos), to_dev(w.strength), to_dev(sa), to_dev(sb), prm)
    u, J = oracle.p2p(w.pos, w.strength, w.pos, w.sigma)
    us, Js = oracle.segments(sa, sb, w.pos, w.seg_core, 2)
    assert rel_l2(dx.double().cpu().numpy().T, u + us) <= TOL_COMP
    assert rel_l2(dG.double().cpu().numpy().T, oracle.stretch(J + Js, w.strength, False)) <= TOL_COMP
    assert api.device_error() == 0
