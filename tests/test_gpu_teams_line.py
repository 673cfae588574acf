"""Where the pair sweep without a workspace goes from warpgroup teams to whole blocks, against the FP64 oracle."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2511_11430_gb300 import synth
from tests._util import TOL_COMP, TOL_PLAIN, rel_l2, to_dev

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compensated", [True, False])
@pytest.mark.parametrize("n_src,n_tgt", [(31 * 128, 131_072), (32 * 128, 131_072), (32 * 128 + 1, 130_817),
                                         (1024 * 128, 7_169), (1024 * 128, 4_097), (1024 * 128, 7_000)])
def test_line(n_src, n_tgt, compensated):
    """4,096 units of 1,024 targets by 128 sources; eight target tiles (7,169 targets) or fewer."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_11430_gb300 import _lib, api, build

    build.build()
    lib = _lib.load()
    w = synth.hover(seed=4, n=n_src)
    tgt = np.zeros((n_tgt, 4), dtype=np.float32)
    tgt[:, :3] = np.random.default_rng(3).uniform([-1, -1, -1.2], [1, 1, 0.4], size=(n_tgt, 3))
    P, S, T = to_dev(w.pos), to_dev(w.strength), to_dev(tgt)
    u = torch.full((3, n_tgt), float("nan"), device="cuda")
    g = torch.full((9, n_tgt), float("nan"), device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    st = lib.vpm_induce_noalloc(p(P), p(S), n_src, p(T), n_tgt, ctypes.c_float(w.sigma), int(compensated), p(u), p(g),
                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0, lib.vpm_last_error()
    idx = np.unique(np.concatenate([[0, n_tgt - 1], synth.sample_targets(5, n_tgt, 64)]))
    ru, rJ = oracle.p2p(w.pos, w.strength, tgt[idx], w.sigma)
    tol = TOL_COMP if compensated else TOL_PLAIN
    rows = lambda t: t[:, idx].double().cpu().numpy().T
    assert rel_l2(rows(u), ru) <= tol
    assert rel_l2(rows(g).reshape(-1, 3, 3), rJ) <= tol
    assert api.device_error() == 0
