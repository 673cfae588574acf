"""The work a rotor-wake program has this framework do, as cases that can be timed and compared.

A case names one public call (``kind``), the synthetic wake it works on (``wake``: the generators of
``synth``, which stand for the rotors of the paper) and its size:

  rhs        api.rhs            the right-hand side of one time-step stage, particles and blade segments
  induce     api.induce         velocity and gradient of the particles on themselves
  points     api.induce         their velocity at the blades' control points (Neumann condition)
  adjoint    autograd.induce    that velocity, the downwash loss and its gradients, forward and backward
  segments   api.segments_induce  velocity and gradient of the blades' segments on the particles
  aic        api.aic_build, api.aic_solve   the blade circulations of one time step
  tree       api.tree_induce    the treecode's velocity and gradient
  rhs_tree   api.rhs_tree       the right-hand side by the treecode

``exact`` restates each direct sum in plain FP64 torch (the treecode against the direct sum it
approximates).
"""
import math

import numpy as np
import torch

from paper_2511_11430_gb300 import api, autograd, synth

WAKES = {"small_hover": synth.small_hover, "hover": synth.hover, "bvi": synth.bvi, "multirotor": synth.multirotor}
THETA, ORDER = 0.5, 4  # the treecode's usual setting
# pairs that exact() takes in a few seconds
EXACT_PAIRS = 2.0e10


def listed():
    return [
        # one stage of a two-bladed test rotor: a development run, and every wake's first steps
        {"name": "rhs_small_2k", "kind": "rhs", "wake": "small_hover", "n": 2000, "compensated": True, "classic": False},
        # a wake some revolutions old; a size that is no multiple of anything
        {"name": "rhs_hover_20k", "kind": "rhs", "wake": "hover", "n": 20011, "compensated": True, "classic": False},
        # the four-bladed hover wake, the ordinary stage of a production run
        {"name": "rhs_hover_100k", "kind": "rhs", "wake": "hover", "n": 100000, "compensated": True, "classic": False},
        # forward flight with blade-vortex interaction, in plain sums and with the classic stretching
        {"name": "rhs_bvi_60k_plain", "kind": "rhs", "wake": "bvi", "n": 59999, "compensated": False, "classic": True},
        # two rotors side by side: the large direct sum
        {"name": "induce_two_rotors_400k", "kind": "induce", "wake": "multirotor", "n": 400000, "compensated": True},
        # the wake's velocity at 1,280 control points, once per time step
        {"name": "points_200k", "kind": "points", "wake": "hover", "n": 200000, "compensated": True},
        # the gradient of a downwash loss with respect to the wake
        {"name": "adjoint_200k", "kind": "adjoint", "wake": "hover", "n": 200000, "compensated": True},
        # the blades' 5,120 segments on the hover wake
        {"name": "segments_100k", "kind": "segments", "wake": "hover", "n": 100000, "compensated": True, "vatistas_n": 2},
        # blade circulations: the small rotor and the four-bladed one
        {"name": "aic_160", "kind": "aic", "blades": 2, "span": 20, "chord": 4},
        {"name": "aic_1280", "kind": "aic", "blades": 4, "span": 40, "chord": 8},
        # a million particles by the treecode, and a stage's right-hand side by it
        {"name": "tree_bvi_1m", "kind": "tree", "wake": "bvi", "n": 1000000},
        {"name": "rhs_tree_hover_300k", "kind": "rhs_tree", "wake": "hover", "n": 300001},
    ]


def draw(rng):
    kind = rng.choice(["rhs", "rhs", "rhs", "induce", "induce", "points", "adjoint", "segments", "aic", "tree", "rhs_tree"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    wake = rng.choice(["small_hover", "hover", "bvi", "multirotor"])
    if kind == "aic":
        return {"kind": kind, "blades": rng.choice([2, 3, 4]), "span": rng.randint(8, 40), "chord": rng.randint(2, 8)}
    lo = 8000 if wake == "bvi" else 1500  # the three filaments of the BVI wake are 6,000 of its particles
    if kind == "rhs":
        return {"kind": kind, "wake": wake, "n": size(lo, 150000), "compensated": rng.random() < 0.75,
                "classic": rng.random() < 0.25}
    if kind in ("induce", "points", "adjoint"):
        return {"kind": kind, "wake": wake, "n": size(lo, 300000), "compensated": rng.random() < 0.75}
    if kind == "segments":
        return {"kind": kind, "wake": wake, "n": size(lo, 200000), "compensated": rng.random() < 0.75,
                "vatistas_n": rng.choice([1, 2, 2])}
    return {"kind": kind, "wake": wake if wake != "small_hover" else "hover",
            "n": size(100000, 1000000 if kind == "tree" else 400000)}


def _wake(case, seed):
    return WAKES[case["wake"]](seed=int(seed), n=int(case["n"]))


def _blades(case, seed):
    """A rotor's lattice at a collective, azimuth and inflow of its own."""
    rng = np.random.default_rng(int(seed))
    lat = synth.blade_lattice(case["blades"], case["span"], case["chord"], pitch_deg=float(rng.uniform(5.0, 11.0)),
                              phase=float(rng.uniform(0.0, 2.0 * np.pi)))
    pad = lambda a: np.concatenate([a, np.zeros(a.shape[:-1] + (1,))], axis=-1).astype(np.float32)
    rings, colloc, normal, vrel = (pad(a) for a in lat[:4])
    w_ind = rng.normal(scale=4.0, size=(3, colloc.shape[0])).astype(np.float32)  # what the wake induces there
    return rings, colloc, normal, vrel, w_ind


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "aic":
        rings, colloc, normal, vrel, w_ind = (_cuda(a) for a in _blades(case, seed))
        return {"kind": kind, "rings": rings, "colloc": colloc, "normal": normal, "v_rel": vrel, "w_ind": w_ind,
                "core": 0.01, "ws": api.Workspace("cuda")}
    w = _wake(case, seed)
    s = {"kind": kind, "pos": _cuda(w.pos), "str": _cuda(w.strength), "sigma": w.sigma, "ws": api.Workspace("cuda"),
         "compensated": case.get("compensated", True)}
    if kind in ("rhs", "rhs_tree"):
        s["seg_a"], s["seg_b"] = _cuda(w.seg_a), _cuda(w.seg_b)
        s["params"] = api.Params(sigma=w.sigma, nu=w.nu, c_v=w.c_v, seg_core=w.seg_core, u_inf=w.u_inf,
                                 compensated=case.get("compensated", True), classic=case.get("classic", False))
    elif kind == "segments":
        s["seg_a"], s["seg_b"], s["core"], s["vn"] = _cuda(w.seg_a), _cuda(w.seg_b), w.seg_core, case["vatistas_n"]
    elif kind in ("points", "adjoint"):
        s["colloc"] = _cuda(w.colloc)
        if kind == "adjoint":
            s["normal"] = _cuda(np.ascontiguousarray(w.normal[:, :3].T))
            s["pos"].requires_grad_(True)
            s["str"].requires_grad_(True)
    return s


def run(s):
    kind = s["kind"]
    if kind == "rhs":
        return api.rhs(s["pos"], s["str"], s["seg_a"], s["seg_b"], s["params"], ws=s["ws"])
    if kind == "induce":
        return api.induce(s["pos"], s["str"], s["pos"], s["sigma"], compensated=s["compensated"], ws=s["ws"])
    if kind == "points":
        return api.induce(s["pos"], s["str"], s["colloc"], s["sigma"], compensated=s["compensated"], grad=False,
                          ws=s["ws"])
    if kind == "adjoint":
        u = autograd.induce(s["pos"], s["str"], s["colloc"], s["sigma"], s["compensated"])
        loss = (u * s["normal"]).sum(0).square().sum()
        return (u.detach(),) + torch.autograd.grad(loss, (s["pos"], s["str"]))
    if kind == "segments":
        return api.segments_induce(s["seg_a"], s["seg_b"], s["pos"], s["core"], s["vn"], compensated=s["compensated"],
                                   ws=s["ws"])
    if kind == "aic":
        A, b = api.aic_build(s["rings"], s["colloc"], s["normal"], s["core"], v_rel=s["v_rel"], w_ind=s["w_ind"])
        x, _, _ = api.aic_solve(A, b, ws=s["ws"])
        return A, b, x
    if kind == "tree":
        return api.tree_induce(s["pos"], s["str"], s["sigma"], theta=THETA, order=ORDER, ws=s["ws"])
    return api.rhs_tree(s["pos"], s["str"], s["seg_a"], s["seg_b"], s["params"], theta=THETA, order=ORDER, ws=s["ws"])


def _rings(case):
    return {"small_hover": 160, "hover": 1280, "bvi": 1280, "multirotor": 1920}[case["wake"]]


def work(case):
    kind = case["kind"]
    if kind == "aic":
        n = case["blades"] * case["span"] * case["chord"]
        return {"bytes": 4.0 * n * n * 2 + 16.0 * n * 8, "flops": 2.0 / 3.0 * n ** 3 + 4 * 60.0 * n * n + 6.0 * n * n}
    n = float(case["n"])
    k = float(_rings(case))
    if kind == "rhs":  # 54 flops a particle pair, 120 a segment pair, FFMA as two
        return {"bytes": 32 * n + 128 * k + 28 * n, "flops": 54 * n * n + 120 * 4 * k * n}
    if kind == "induce":
        return {"bytes": 32 * n + 48 * n, "flops": 54 * n * n}
    if kind == "points":
        return {"bytes": 32 * n + 28 * k, "flops": 26 * n * k}
    if kind == "adjoint":
        return {"bytes": 32 * n + 44 * k + 32 * n, "flops": (26 + 54) * n * k}
    if kind == "segments":
        return {"bytes": 16 * n + 128 * k + 48 * n, "flops": 120 * 4 * k * n}
    # the treecode: 54 flops for each of the particles within 7 core sizes (about five hundred) and as
    # many again for the expansions
    segs = 128 * k if kind == "rhs_tree" else 0.0
    return {"bytes": 32 * n + (28 if kind == "rhs_tree" else 48) * n + segs, "flops": 54 * n * 1000}


# ---- the same results in plain FP64 torch -----------------------------------------------------
FOUR_PI = 4.0 * math.pi


def _pair_kernels(r2, sigma):
    """K and H = K'(r)/r of the Gaussian blob at squared distances r2 (consumed), zero at zero distance."""
    zero = r2 == 0
    r2 = r2.masked_fill(zero, 1.0)
    r = r2.sqrt()
    rho = r / sigma
    e = math.sqrt(2.0 / math.pi) * rho * torch.exp(-0.5 * rho * rho)
    g = torch.special.erf(rho / math.sqrt(2.0)) - e
    # below rho = 0.3 the closed form cancels: the incomplete-gamma series with positive terms
    low = rho < 0.3
    if bool(low.any()):
        x = 0.5 * rho[low] ** 2
        t = torch.zeros_like(x)
        for k in range(12, -1, -1):
            t = t * x + 1.0 / math.gamma(k + 2.5)
        g[low] = x ** 1.5 * torch.exp(-x) * t
    K = g / (FOUR_PI * r2 * r)
    # K'(r)/r = (rho g'(rho) - 3 g)/(4 pi r^5), g'(rho) = sqrt(2/pi) rho^2 exp(-rho^2/2)
    H = (rho * rho * e - 3.0 * g) / (FOUR_PI * r2 * r2 * r)
    if bool(low.any()):
        x = 0.5 * rho[low] ** 2
        t = torch.zeros_like(x)
        for k in range(12, -1, -1):
            t = t * x + 1.5 / math.gamma(k + 3.5)
        H[low] = -(2.0 ** -1.5) * torch.exp(-x) * t / (FOUR_PI * sigma ** 5)
    return K.masked_fill_(zero, 0.0), H.masked_fill_(zero, 0.0)


def _r2(y, x):
    r2 = torch.zeros((y.shape[0], x.shape[0]), dtype=torch.float64, device=y.device)
    for a in range(3):
        r2 += (y[:, a, None] - x[None, :, a]).square()
    return r2


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _skew(s):
    """The matrix [s x] of each row of s."""
    z = torch.zeros_like(s[:, 0])
    return torch.stack([z, -s[:, 2], s[:, 1], s[:, 2], z, -s[:, 0], -s[:, 1], s[:, 0], z], 1).reshape(-1, 3, 3)


def _p2p(x, G, y, sigma, grad=True):
    """u [m, 3] and J [m, 3, 3] at the points y."""
    m = _cross(G, x)
    # with c = G x r = G x y - m: u = S x y - sum K m; J = [S x] + sum H c r^T, r = y - x
    FK = torch.cat([G, m], 1)
    FH = torch.cat([G, m, (G[:, :, None] * x[:, None, :]).reshape(-1, 9), (m[:, :, None] * x[:, None, :]).reshape(-1, 9)], 1)
    us, Js = [], []
    step = max(1, int(1.0e8 // max(1, x.shape[0])))
    for i in range(0, y.shape[0], step):
        yc = y[i:i + step]
        K, H = _pair_kernels(_r2(yc, x), sigma)
        a = K @ FK
        us.append(_cross(a[:, :3], yc) - a[:, 3:])
        if grad:
            b = H @ FH
            c = _cross(b[:, :3], yc) - b[:, 3:6]
            Gx = b[:, 6:15].reshape(-1, 3, 3)  # sum H G_c x_b
            mx = b[:, 15:].reshape(-1, 3, 3)
            cx = torch.stack([_cross(Gx[:, :, k], yc) for k in range(3)], 2) - mx  # sum H c_a x_b
            Js.append(_skew(a[:, :3]) + c[:, :, None] * yc[:, None, :] - cx)
    u = torch.cat(us)
    return (u, torch.cat(Js)) if grad else u


def _segments(a, b, g, y, core, vn):
    us, Js = [], []
    r0 = b - a
    L2 = r0.square().sum(1)
    e = (core * core * L2) ** vn
    step = max(1, int(2.0e7 // max(1, a.shape[0])))
    eye = torch.eye(3, dtype=torch.float64, device=y.device)
    for i in range(0, y.shape[0], step):
        yc = y[i:i + step]
        r1 = yc[:, None, :] - a[None]
        r2 = yc[:, None, :] - b[None]
        n1, n2 = r1.norm(dim=2), r2.norm(dim=2)
        c = _cross(r1, r2)
        c2 = c.square().sum(2)
        d = (r0 * r1).sum(2) / n1 - (r0 * r2).sum(2) / n2
        D = (c2 ** vn + e) ** (1.0 / vn)
        f = g / (FOUR_PI * D)
        us.append((f * d)[:, :, None].mul(c).sum(1))
        # J = f (d [r0 x] + c (grad d - d grad D / D)^T)
        gd = (r0[None] - r1 * ((r0 * r1).sum(2) / n1.square())[:, :, None]) / n1[:, :, None]
        gd = gd - (r0[None] - r2 * ((r0 * r2).sum(2) / n2.square())[:, :, None]) / n2[:, :, None]
        gD = 2.0 * (c2 ** (vn - 1) * (c2 ** vn + e) ** (1.0 / vn - 1.0))[:, :, None] * _cross(c, r0[None].expand_as(c))
        w = gd - (d / D)[:, :, None] * gD
        J = torch.einsum("ts,tsa,tsb->tab", f, c, w)
        J = J + _skew(torch.einsum("ts,sa->ta", f * d, r0))
        Js.append(J)
    return torch.cat(us), torch.cat(Js)


def _exact_rhs(w, classic):
    t = lambda a: torch.from_numpy(a).cuda().double()
    pos, G = t(w.pos), t(w.strength)[:, :3]
    x, vol = pos[:, :3].contiguous(), pos[:, 3]
    u, J = _p2p(x, G, x, w.sigma)
    sa, sb = t(w.seg_a), t(w.seg_b)
    us, Js = _segments(sa[:, :3].contiguous(), sb[:, :3].contiguous(), sa[:, 3], x, w.seg_core, 2)
    u, J = u + us, J + Js
    g = J @ J.transpose(1, 2)
    aa = torch.diagonal(g, dim1=1, dim2=2).sum(1)
    B = (g[:, 0, 0] * g[:, 1, 1] - g[:, 0, 1] ** 2 + g[:, 0, 0] * g[:, 2, 2] - g[:, 0, 2] ** 2
         + g[:, 1, 1] * g[:, 2, 2] - g[:, 1, 2] ** 2)
    nut = torch.where((aa > 0) & (B > 0), w.c_v * w.sigma ** 2 * (B.clamp_min(0) / aa.clamp_min(1e-300)).sqrt(), 0.0)
    s = torch.einsum("nab,nb->na" if classic else "nba,nb->na", J, G)
    # exchange: sum_j nu_ij (v_i G_j - v_j G_i) zeta, nu_ij = nu + (nu_t,i + nu_t,j)/2
    F = torch.cat([G, vol[:, None], nut[:, None] * G, (nut * vol)[:, None]], 1)
    p = torch.empty_like(G)
    s2 = w.sigma ** 2
    zeta0 = (2.0 * math.pi * s2) ** -1.5
    step = max(1, int(1.0e8 // w.n))
    for i in range(0, w.n, step):
        Z = torch.exp(_r2(x[i:i + step], x) * (-0.5 / s2)) * zeta0
        b = Z @ F
        q = slice(i, i + step)
        base = (w.nu + 0.5 * nut[q])[:, None]
        p[q] = vol[q][:, None] * (base * b[:, :3] + 0.5 * b[:, 4:7]) - G[q] * (base * b[:, 3:4] + 0.5 * b[:, 7:8])
    p *= 2.0 / s2
    uinf = torch.tensor(w.u_inf, dtype=torch.float64, device="cuda")
    return (u + uinf).t().contiguous(), (s + p).t().contiguous(), nut


def exact(case, seed):
    kind = case["kind"]
    t = lambda a: torch.from_numpy(a).cuda().double()
    if kind == "aic":
        rings, colloc, normal, vrel, w_ind = (t(a) for a in _blades(case, seed))
        n = colloc.shape[0]
        y, nrm = colloc[:, :3].contiguous(), normal[:, :3]
        A = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        for k in range(4):
            a, b = rings[:, k, :3], rings[:, (k + 1) % 4, :3]
            r0 = b - a
            e = (0.01 ** 2 * r0.square().sum(1)) ** 2
            r1, r2 = y[:, None, :] - a[None], y[:, None, :] - b[None]
            c = _cross(r1, r2)
            d = (r0 * r1).sum(2) / r1.norm(dim=2) - (r0 * r2).sum(2) / r2.norm(dim=2)
            A += d / (FOUR_PI * (c.square().sum(2) ** 2 + e).sqrt()) * torch.einsum("tsa,ta->ts", c, nrm)
        b = -((vrel[:, :3] + w_ind.t()) * nrm).sum(1)
        return A, b, torch.linalg.solve(A, b)
    k = _rings(case)
    n = float(case["n"])
    if (n * k if kind in ("points", "adjoint") else n * n if kind != "segments" else n * 4 * k * 20) > EXACT_PAIRS:
        return None
    w = _wake(case, seed)
    if kind in ("rhs", "rhs_tree"):
        return _exact_rhs(w, case.get("classic", False))
    pos, G = t(w.pos)[:, :3].contiguous(), t(w.strength)[:, :3].contiguous()
    if kind in ("induce", "tree"):
        u, J = _p2p(pos, G, pos, w.sigma)
        return u.t().contiguous(), J.reshape(-1, 9).t().contiguous()
    y = t(w.colloc)[:, :3].contiguous()
    if kind == "points":
        return _p2p(pos, G, y, w.sigma, grad=False).t().contiguous()
    if kind == "segments":
        sa, sb = t(w.seg_a), t(w.seg_b)
        u, J = _segments(sa[:, :3].contiguous(), sb[:, :3].contiguous(), sa[:, 3], pos, w.seg_core, case["vatistas_n"])
        return u.t().contiguous(), J.reshape(-1, 9).t().contiguous()
    # the downwash loss sum_k (u_k . n_k)^2 and its gradients
    u = _p2p(pos, G, y, w.sigma, grad=False)
    nrm = t(w.normal)[:, :3]
    g = 2.0 * (u * nrm).sum(1)[:, None] * nrm
    dx, dG = torch.zeros_like(pos), torch.zeros_like(G)
    step = max(1, int(2.0e7 // y.shape[0]))
    for i in range(0, pos.shape[0], step):
        x, Gc = pos[i:i + step], G[i:i + step]
        r = y[None] - x[:, None]  # [particles, points, 3]
        K, H = _pair_kernels(r.square().sum(2), w.sigma)
        gx = g[None].expand_as(r)
        dG[i:i + step] = (K[:, :, None] * _cross(r, gx)).sum(1)
        c = _cross(Gc[:, None].expand_as(r), gx)
        q = H * (_cross(Gc[:, None].expand_as(r), r) * gx).sum(2)
        dx[i:i + step] = (K[:, :, None] * c - q[:, :, None] * r).sum(1)
    pad = lambda a: torch.cat([a, torch.zeros_like(a[:, :1])], 1)
    return u.t().contiguous(), pad(dx), pad(dG)
