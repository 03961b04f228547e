"""What a user of the framework has it compute: layer potentials by Global QBX on
the geometries of qbx_workloads, direct and FMM-accelerated, in FP64 and mixed
precision, alone and in batches, the scattering solve and the plan set-up.

A mixed-precision evaluation forms its sums in FP32 and promises 1e-6, so a
caller keeps its results as complex64; the mixed cases return them in that type.
"""
import math

import numpy as np
import torch

from paper_1602_05301_gb300 import qbx
from qbx_workloads import concat_geometries, discretise_curve, ellipse, fourier_radial
from qbx_workloads.configs import grid_targets

ARMS, AMPLITUDE = 5, 0.3   # the starfish r(t) = 1 + 0.3 cos(5 t + phase)


def listed():
    return [
        # the smallest call: one circle, single layer, all pairs; nodes on both sides and two
        # rings of targets (the configuration circle-k1)
        dict(name="direct-circle", kind="curve", mode="direct", precision="fp64", layers="S",
             k=1.0, panels=32, q=16, p=8, sides=2, q_src=0, surface="both", grid=31, p_fmm=0,
             amplitude=0.0),
        # all pairs at the size where the FMM starts to pay: combined field on a starfish
        dict(name="direct-starfish", kind="curve", mode="direct", precision="fp64", layers="DS",
             k=10.0, panels=128, q=16, p=12, sides=2, q_src=0, surface="both", grid=64, p_fmm=0,
             amplitude=AMPLITUDE),
        # a field plot around one scatterer, in both precisions (starfish-k10)
        dict(name="starfish-k10-fp64", kind="curve", mode="fmm", precision="fp64", layers="DS",
             k=10.0, panels=512, q=16, p=12, sides=2, q_src=0, surface="none", grid=316,
             p_fmm=20, amplitude=AMPLITUDE),
        dict(name="starfish-k10-mixed", kind="curve", mode="fmm", precision="mixed", layers="DS",
             k=10.0, panels=512, q=16, p=12, sides=2, q_src=0, surface="none", grid=316,
             p_fmm=20, amplitude=AMPLITUDE),
        # the QBX coefficients of every centre, for a caller that evaluates the disks itself
        dict(name="starfish-k10-coefficients", kind="curve", mode="fmm", precision="fp64",
             layers="DS", k=10.0, panels=512, q=16, p=12, sides=2, q_src=0, surface="none",
             grid=100, p_fmm=20, amplitude=AMPLITUDE, alpha=True),
        # a finely resolved scatterer at a high wavenumber (starfish-k50)
        dict(name="starfish-k50-mixed", kind="curve", mode="fmm", precision="mixed", layers="DS",
             k=50.0, panels=8192, q=16, p=16, sides=2, q_src=0, surface="none", grid=316,
             p_fmm=30, amplitude=AMPLITUDE),
        # ragged sizes, a library-made source grid, the mean of both limits at the nodes
        dict(name="ragged-oversampled", kind="curve", mode="fmm", precision="fp64", layers="S",
             k=7.0, panels=137, q=10, p=7, sides=2, q_src=24, surface="mean", grid=75, p_fmm=17,
             amplitude=AMPLITUDE),
        # many scatterers in a wide box: targets everywhere and near the curves (an eighth of
        # ellipses-200 in FP64, and the whole of it in mixed precision, the headline workload)
        dict(name="ellipses-25-fp64", kind="ellipses", precision="fp64", layers="D", k=20.0,
             curves=25, panels=8192, q=16, p=16, p_fmm=30, uniform=112_500, near=12_500),
        dict(name="ellipses-200-mixed", kind="ellipses", precision="mixed", layers="D", k=20.0,
             curves=200, panels=65536, q=16, p=16, p_fmm=30, uniform=900_000, near=100_000),
        # independent curves with their own wavenumbers in one graph, every node an exterior
        # on-surface target: one step of many boundary integral solvers (batch-256)
        dict(name="batch-32-mixed", kind="batch", precision="mixed", curves=32, panels_min=16,
             panels_max=1024, q=16, p=12, p_fmm=20),
        # a sound-soft scattering problem solved by GMRES to the paper's tolerance, the plan
        # made inside the call
        dict(name="scattering-starfish", kind="solve", precision="fp64", k=10.0, panels=96, q=16,
             p=12, q_src=64, p_fmm=30, amplitude=0.2),
        # a new geometry taken into use: centres, tree, lists, association, tables
        dict(name="plan-starfish", kind="plan", k=10.0, panels=512, q=16, p=12, sides=2,
             surface="none", grid=316, p_fmm=20, amplitude=AMPLITUDE),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["direct", "curve", "curve", "curve", "ellipses", "ellipses", "batch",
                       "solve", "plan"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "direct":
        q = rng.choice([8, 10, 12, 16])
        panels = _log_int(rng, 30, 160)
        return dict(kind="curve", mode="direct", precision="fp64",
                    layers=rng.choice(["S", "D", "DS"]), k=round(rng.uniform(1.0, 10.0), 2),
                    panels=panels, q=q, p=rng.randint(3, 16), sides=2,
                    q_src=rng.choice([0, 0, 2 * q]), surface=rng.choice(["both", "mean"]),
                    grid=_log_int(rng, 20, 80), p_fmm=0, amplitude=0.2)
    if kind == "curve":
        alpha = prec == "fp64" and rng.random() < 0.3
        panels = _log_int(rng, 64, 2048 if alpha else 8192)
        k = round(min(rng.uniform(2.0, 50.0), 0.35 * panels), 2)
        return dict(kind="curve", mode="fmm", precision=prec,
                    layers=rng.choice(["S", "D", "DS"]), k=k, panels=panels,
                    q=rng.choice([10, 13, 16]), p=rng.randint(10 if alpha else 5, 16), sides=2,
                    q_src=0, surface=rng.choice(["none", "both", "mean"]) if panels < 1024 else "none",
                    grid=_log_int(rng, 60, 330), p_fmm=rng.randint(18, 30), amplitude=AMPLITUDE,
                    alpha=alpha)
    if kind == "ellipses":
        n = _log_int(rng, 6, 60)
        share = rng.uniform(0.5, 1.5)
        return dict(kind="ellipses", precision=prec, layers=rng.choice(["S", "D", "DS"]),
                    k=round(rng.uniform(5.0, 20.0), 2), curves=n, panels=int(300 * n * share),
                    q=16, p=rng.randint(8, 16), p_fmm=rng.randint(20, 30),
                    uniform=int(4500 * n * rng.uniform(0.4, 1.6)), near=500 * n)
    if kind == "batch":
        return dict(kind="batch", precision=prec, curves=_log_int(rng, 4, 32), panels_min=16,
                    panels_max=_log_int(rng, 64, 1024), q=16, p=rng.choice([8, 12]), p_fmm=20)
    if kind == "solve":
        return dict(kind="solve", precision="fp64", k=round(rng.uniform(3.0, 12.0), 2),
                    panels=_log_int(rng, 48, 96), q=16, p=rng.choice([10, 12]), q_src=64,
                    p_fmm=30, amplitude=0.2)
    return dict(kind="plan", k=round(rng.uniform(2.0, 20.0), 2), panels=_log_int(rng, 64, 1024),
                q=16, p=rng.choice([8, 12, 16]), sides=2, surface=rng.choice(["none", "both"]),
                grid=_log_int(rng, 60, 330), p_fmm=rng.randint(20, 30), amplitude=AMPLITUDE)


# ---------------------------------------------------------------- inputs
def _modes(t, rng, modes=20):
    """Random complex Fourier modes |n| <= modes at the curve parameters t."""
    m = 2 * modes + 1
    c = (rng.standard_normal(m) + 1j * rng.standard_normal(m)) / math.sqrt(2.0)
    z = np.exp(1j * t)
    v = np.full(t.shape, c[-1])
    for a in c[-2::-1]:
        v = v * z + a
    return v * np.conj(z) ** modes


def _starfish(case, rng):
    a = np.zeros(ARMS)
    a[ARMS - 1] = case["amplitude"]
    curve = fourier_radial(a, np.full(ARMS, rng.uniform(0.0, 2.0 * np.pi)))
    return discretise_curve(*curve, case["panels"], case["q"], k=case["k"])


def _with_surface(geom, surface, off):
    """Targets: the nodes (one or both one-sided limits, or their mean), then `off`."""
    n = geom.n
    sides = {"none": [], "exterior": [1], "both": [1, -1], "mean": [0]}[surface]
    xy = np.concatenate([geom.node_xy] * len(sides) + [off])
    node = np.concatenate([np.arange(n)] * len(sides) + [np.full(len(off), -1)]).astype(np.int64)
    side = np.concatenate([np.full(n, s) for s in sides] + [np.zeros(len(off))]).astype(np.int8)
    return np.ascontiguousarray(xy), node, side


def _ellipses(case, rng):
    n, k = case["curves"], case["k"]
    side = 100.0 * math.sqrt(n / 200.0)
    axes, rot = rng.uniform(0.5, 2.0, (n, 2)), rng.uniform(0.0, np.pi, n)
    rad = axes.max(axis=1)
    ctr = np.empty((0, 2))
    for i in range(n):
        while True:
            c = rng.uniform(rad[i], side - rad[i], 2)
            if (np.hypot(*(ctr - c).T) >= rad[:i] + rad[i] + 0.5).all():
                ctr = np.concatenate([ctr, c[None]])
                break
    a, b = axes.T
    h = ((a - b) / (a + b)) ** 2
    per = np.pi * (a + b) * (1 + 3 * h / (10 + np.sqrt(4 - 3 * h)))  # Ramanujan
    npan = np.maximum(64, np.floor(case["panels"] * per / per.sum())).astype(int)
    parts = [discretise_curve(*ellipse(a[i], b[i], rot[i], ctr[i]), int(npan[i]), case["q"], k=k)
             for i in range(n)]
    geom = concat_geometries(parts)
    sigma = np.concatenate([_modes(g.param_t, rng) for g in parts])
    nodes = rng.integers(0, geom.n, case["near"])
    off = rng.uniform(0.0, 0.5, case["near"]) * geom.panel_h[geom.panel_of_node[nodes]]
    off *= np.where(rng.random(case["near"]) < 0.5, 1.0, -1.0)
    tgt = np.concatenate([rng.uniform(0.0, side, (case["uniform"], 2)),
                          geom.node_xy[nodes] + off[:, None] * geom.normal_xy[nodes]])
    return geom, sigma, tgt


def _batch_curve(case, i, rng):
    """Curve i of a batch: its panel count by the case alone (spread over the range), shape
    and wavenumber by rng; 0.5 k per panel resolves the wavelength (Condition 4)."""
    lo, hi = case["panels_min"], case["panels_max"]
    n = lo + (i * 0.618034 % 1.0) * (hi - lo)
    a, phi = rng.uniform(0.0, 0.05, 5), rng.uniform(0.0, 2.0 * np.pi, 5)
    k = rng.uniform(1.0, min(40.0, 0.5 * n))
    geom = discretise_curve(*fourier_radial(a, phi), int(n), case["q"], k=k)
    return geom, _modes(geom.param_t, rng)


def _problems(case, seed):
    """The independent problems of a case: geometry, density, targets, layer factors."""
    rng = np.random.Generator(np.random.PCG64(seed))
    if case["kind"] == "batch":
        out = []
        for i in range(case["curves"]):
            geom, sigma = _batch_curve(case, i, rng)
            xy, node, side = _with_surface(geom, "exterior", np.empty((0, 2)))
            out.append(dict(geom=geom, sigma=sigma, xy=xy, node=node, side=side, sides=1,
                            cS=1j * float(geom.k[0]), cD=1.0, q_src=0))
        return out
    if case["kind"] == "ellipses":
        geom, sigma, tgt = _ellipses(case, rng)
        xy, node, side, sides, q_src = tgt, None, None, 2, 0
    elif case["kind"] == "solve":
        geom, th = _starfish(case, rng), rng.uniform(0.0, 2.0 * np.pi)
        sigma = -np.exp(1j * case["k"] * (geom.node_xy @ np.array([math.cos(th), math.sin(th)])))
        xy, node, side = _with_surface(geom, "exterior", np.empty((0, 2)))
        sides, q_src = 1, case["q_src"]
    else:
        geom = _starfish(case, rng)
        sigma = _modes(geom.param_t, rng)
        grid = grid_targets(case["grid"], -2.0, 2.0) + rng.uniform(-0.03, 0.03, 2)
        xy, node, side = _with_surface(geom, case["surface"], grid)
        sides, q_src = case["sides"], case.get("q_src", 0)
    layers = case.get("layers", "DS")
    return [dict(geom=geom, sigma=sigma, xy=xy, node=node, side=side, sides=sides, q_src=q_src,
                 cS=1j * case["k"] if "S" in layers else None, cD=1.0 if "D" in layers else None)]


def _handle(case, pr):
    return qbx.LayerPotential(pr["geom"].as_dict(), case["p"], sides=pr["sides"], q_src=pr["q_src"])


def _build(lp, case, pr):
    mode = qbx.QBX_DIRECT if case.get("mode") == "direct" else qbx.QBX_FMM
    return lp.build(pr["xy"], pr["node"], pr["side"], mode=mode, p_fmm=case["p_fmm"])


def prepare(case, seed):
    prs = _problems(case, seed)
    prec = qbx.QBX_MIXED if case.get("precision") == "mixed" else qbx.QBX_FP64
    st = dict(case=case, precision=prec)
    if case["kind"] == "plan":   # host arrays, as a geometry program hands them over
        return dict(st, problem=prs[0])
    lps = [_handle(case, pr) for pr in prs]
    if case["kind"] == "solve":  # the call makes its own plan and returns host arrays
        return dict(st, lp=lps[0], rhs=prs[0]["sigma"])
    for lp, pr in zip(lps, prs):
        _build(lp, case, pr)
    cS, cD = [pr["cS"] for pr in prs], [pr["cD"] for pr in prs]
    sigma = torch.from_numpy(np.concatenate([pr["sigma"] for pr in prs])).cuda()
    n_tgt = sum(lp.n_targets for lp in lps)
    st.update(lp=lps[0], cS=cS[0], cD=cD[0], sigma=sigma,
              out=torch.empty(n_tgt, dtype=torch.complex128, device="cuda"), alpha=None)
    if case.get("alpha"):
        st["alpha"] = torch.empty((lps[0].n_centres, 2 * case["p"] + 1), dtype=torch.complex128,
                                  device="cuda")
    if case["kind"] == "batch":
        st.update(batch=qbx.Batch(lps), cS=np.array(cS), cD=np.array(cD, dtype=complex))
    return st


def run(st):
    case, stream = st["case"], torch.cuda.current_stream().cuda_stream
    if case["kind"] == "plan":
        lp = _handle(case, st["problem"])
        assoc = _build(lp, case, st["problem"])
        lp.close()
        return assoc
    if case["kind"] == "solve":
        sigma, _, _ = st["lp"].solve_dirichlet(st["rhs"], p_fmm=case["p_fmm"], tol=1e-5,
                                               precision=st["precision"], stream=stream)
        return sigma
    if case["kind"] == "batch":
        st["batch"].eval(sigma_S=st["sigma"], sigma_D=st["sigma"], cS=st["cS"], cD=st["cD"],
                         out=st["out"], precision=st["precision"], stream=stream)
        got = [st["out"]]
    else:
        kw = {}
        if st["cS"] is not None:
            kw.update(sigma_S=st["sigma"], cS=st["cS"])
        if st["cD"] is not None:
            kw.update(sigma_D=st["sigma"], cD=st["cD"])
        st["lp"].eval(out=st["out"], alpha_out=st["alpha"], precision=st["precision"],
                      stream=stream, **kw)
        got = [st["out"]] + ([st["alpha"]] if st["alpha"] is not None else [])
    if st["precision"] == qbx.QBX_MIXED:
        got = [g.to(torch.complex64) for g in got]
    return got


def _sizes(case):
    """(sources, centres formed, all other targets, targets) of a pass, as expected."""
    if case["kind"] == "batch":
        n = case["curves"] * case["q"] * (case["panels_min"] + case["panels_max"]) // 2
        return n, n, 0, n
    if case["kind"] == "ellipses":
        n, t = case["panels"] * case["q"], case["uniform"] + case["near"]
        return n, case["near"], t - case["near"], t
    n = case["panels"] * case["q"]
    if case["kind"] == "solve":
        return case["panels"] * case["q_src"], n, 0, n
    on = {"none": 0, "both": 2 * n, "mean": 2 * n}[case["surface"]]
    off = case["grid"] ** 2
    nodes = {"none": 0, "both": 2 * n, "mean": n}[case["surface"]]
    src = case["panels"] * (case.get("q_src") or case["q"])
    ctr = 2 * n if case.get("alpha") else max(on, 64)
    return src, ctr, off, nodes + off


def work(case):
    """Bytes: geometry, density and targets in, results out. Flops: the near-field pairs
    (all pairs in direct mode, the 9 neighbouring leaves of 32 sources in FMM mode) at 8
    flops a complex product, and 8 (2 p_fmm + 1)^2 per leaf and translation (27 + 2)."""
    src, ctr, off, tgt = _sizes(case)
    p, layers = case["p"], len(case.get("layers", "DS"))
    P = 2 * p + 1
    data = src * (40 + 16) + tgt * 32 + (ctr * P * 16 if case.get("alpha") else 0)
    if case["kind"] == "plan":
        return dict(bytes=data, flops=60 * (src + ctr + tgt))
    near = src if case.get("mode") == "direct" else min(src, 9 * 32)
    flops = ctr * near * 8 * P * layers + off * near * 40 * layers + 16 * P * ctr
    if case.get("mode") != "direct":
        flops += (src + ctr + off) / 64 * 29 * 8 * (2 * case["p_fmm"] + 1) ** 2
    return dict(bytes=data, flops=flops * (40 if case["kind"] == "solve" else 1))


# ---------------------------------------------------------------- the same in 64 bits
def _lagrange(x, u):
    """Values and derivatives at u of the Lagrange basis of the nodes x."""
    q = len(x)
    L, D = np.ones((len(u), q)), np.zeros((len(u), q))
    for i in range(q):
        for r in range(q):
            if r != i:
                f = (u - x[r]) / (x[i] - x[r])
                D[:, i] = D[:, i] * f + L[:, i] / (x[i] - x[r])
                L[:, i] *= f
    return L, D


def _sources(pr):
    """xy, normal, weight of the source grid and the density-to-source matrix (or None)."""
    g, qs = pr["geom"], pr["q_src"]
    if not qs:
        return g.node_xy, g.normal_xy, g.weight, None
    x, _ = np.polynomial.legendre.leggauss(g.q)
    u, w = np.polynomial.legendre.leggauss(qs)
    L, D = _lagrange(x, u)
    xy = g.node_xy.reshape(-1, g.q, 2)
    s, d = (np.einsum("jr,nrc->njc", B, xy).reshape(-1, 2) for B in (L, D))
    speed = np.hypot(*d.T)
    return s, np.stack([d[:, 1], -d[:, 0]], 1) / speed[:, None], np.tile(w, g.n_panels) * speed, L


# torch.special's Bessel functions are good to about 1e-7 only; these are the CUDA math
# library's, elementwise in 64 bits
_J0, _Y0, _J1, _Y1 = (torch.cuda.jiterator._create_jit_fn(
    "template <typename T> T of_%s(T x) { return ::%s(x); }" % (f, f))
    for f in ("j0", "y0", "j1", "y1"))


def _hankel(x):
    return torch.complex(_J0(x), _Y0(x)), torch.complex(_J1(x), _Y1(x))


def _graf(c, s, k, p):
    """W_l(s - c) = H_l(k r) e^{i l th} for l = 0..p+1 as pairs (W_l, W_-l)."""
    d = s[None] - c[:, None]
    r = torch.hypot(d[..., 0], d[..., 1])
    x, e1 = k * r, torch.complex(d[..., 0], d[..., 1]) / r
    h0, h1 = _hankel(x)
    e = torch.ones_like(e1)
    for l in range(p + 2):
        yield l, h0 * e, h0 * e.conj() * (-1) ** l
        h0, h1, e = h1, h1 * (2 * (l + 1) / x) - h0, e * e1


def _bessel_j(x, p):
    """J_0..J_p of the (small) arguments x by the ascending series."""
    out, lead = [], torch.ones_like(x)
    for l in range(p + 1):
        term, s = lead.clone(), lead.clone()
        for m in range(1, 40):
            term = term * (-(x / 2) ** 2 / (m * (m + l)))
            s = s + term
        out.append(s)
        lead = lead * (x / 2) / (l + 1)
    return out


def _disk_basis(t, c, k, p):
    """J_l(k rho) e^{-i l theta}, l = -p..p, of the targets t about their centres c: [n, 2p+1]."""
    d = t - c
    rho = torch.hypot(d[:, 0], d[:, 1])
    e = torch.where(rho > 0, torch.complex(d[:, 0], d[:, 1]) / rho, 1.0 + 0j)
    J = _bessel_j(k * rho, p)
    return torch.stack([(-1) ** l * J[l] * e ** l for l in range(p, 0, -1)] +
                       [J[l] * e.conj() ** l for l in range(p + 1)], 1)


def _associate(xy, pr, ctr, rad, node_n, eps=0.1):
    best = torch.full((len(xy),), -1, dtype=torch.int64, device=xy.device)
    step = max(1, 20_000_000 // len(ctr))
    order = torch.argsort(ctr[:, 0])
    cx, lim = ctr[order], ((1 + eps) * rad[order]) ** 2
    reach = float((1 + eps) * rad.max())
    by = torch.argsort(xy[:, 0])
    for a in range(0, len(xy), step):
        i = by[a:a + step]
        t = xy[i]
        ends = torch.stack([t[:, 0].min() - reach, t[:, 0].max() + reach])
        lo, hi = torch.searchsorted(cx[:, 0].contiguous(), ends).tolist()
        if hi > lo:
            d2 = ((t[:, None] - cx[None, lo:hi]) ** 2).sum(-1)
            m, j = torch.where(d2 <= lim[None, lo:hi], d2, torch.inf).min(1)
            best[i] = torch.where(m < torch.inf, order[lo:hi][j], -1)
    if pr["node"] is not None:
        node, side = (torch.from_numpy(pr[x]).to(xy.device) for x in ("node", "side"))
        best = torch.where(node >= 0, torch.where(side >= 0, node, node + node_n), best)
    return best


def _setting(pr):
    dev = torch.device("cuda")
    g = pr["geom"]
    up = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)
    s, nrm, w, L = _sources(pr)
    h = g.panel_h[g.panel_of_node][:, None]
    ctr = np.concatenate([g.node_xy + a * 0.5 * h * g.normal_xy for a in (1.0, -1.0)[:pr["sides"]]])
    rad = np.tile(0.5 * h[:, 0], pr["sides"])
    return float(g.k[0]), up(s), up(nrm), up(w), L, up(ctr), up(rad), up(pr["xy"]), g.n


def _potential(case, pr):
    p = case["p"]
    k, s, nrm, w, L, ctr, rad, xy, n = _setting(pr)
    sig = torch.from_numpy(pr["sigma"]).to(s.device)
    if L is not None:
        Lt = torch.from_numpy(L).to(s.device).to(torch.complex128)
        sig = (sig.reshape(-1, Lt.shape[1]) @ Lt.T).reshape(-1)
    zero = torch.zeros_like(sig)
    qs = 0.25j * w * pr["cS"] * sig if pr["cS"] is not None else zero
    ds = 0.25j * w * pr["cD"] * sig if pr["cD"] is not None else zero
    nu = torch.complex(nrm[:, 0], nrm[:, 1])
    rhs = torch.stack([qs, 0.5 * k * ds * nu, 0.5 * k * ds * nu.conj()], 1)
    assoc = _associate(xy, pr, ctr, rad, n)
    mean = torch.zeros_like(assoc, dtype=torch.bool)
    if pr["node"] is not None:
        mean = torch.from_numpy((pr["node"] >= 0) & (pr["side"] == 0)).to(s.device)
    formed = torch.zeros(len(ctr), dtype=torch.bool, device=s.device)
    formed[assoc[assoc >= 0]] = True
    formed[assoc[mean] + n] = True
    formed = torch.ones_like(formed) if case.get("alpha") else formed
    ids = formed.nonzero()[:, 0]
    alpha = torch.zeros((len(ctr), 2 * p + 1), dtype=torch.complex128, device=s.device)
    step = max(1, 12_000_000 // len(s))
    for a in range(0, len(ids), step):
        i = ids[a:a + step]
        M = torch.zeros((len(i), 2 * p + 5, 3), dtype=torch.complex128, device=s.device)
        for l, wp, wn in _graf(ctr[i], s, k, p):
            M[:, p + 2 + l], M[:, p + 2 - l] = wp @ rhs, wn @ rhs
        alpha[i] = M[:, 2:-2, 0] + M[:, 1:-3, 1] - M[:, 3:-1, 2]
    u = torch.empty(len(xy), dtype=torch.complex128, device=s.device)
    on = (assoc >= 0).nonzero()[:, 0]
    if len(on):
        u[on] = (alpha[assoc[on]] * _disk_basis(xy[on], ctr[assoc[on]], k, p)).sum(1)
        m = mean.nonzero()[:, 0]
        if len(m):
            c = assoc[m] + n
            u[m] = 0.5 * (u[m] + (alpha[c] * _disk_basis(xy[m], ctr[c], k, p)).sum(1))
    off = (assoc < 0).nonzero()[:, 0]
    for a in range(0, len(off), step):
        t = xy[off[a:a + step]]
        d = t[:, None] - s[None]
        r = torch.hypot(d[..., 0], d[..., 1])
        v = torch.zeros(len(t), dtype=torch.complex128, device=s.device)
        if pr["cS"] is not None:
            v = v + torch.complex(_J0(k * r), _Y0(k * r)) @ qs
        if pr["cD"] is not None:
            f = k * (d * nrm[None]).sum(-1) / r
            v = v + torch.complex(_J1(k * r) * f, _Y1(k * r) * f) @ ds
        u[off[a:a + step]] = v
    return [u, alpha] if case.get("alpha") else [u]


def exact(case, seed):
    if case["kind"] in ("plan", "solve"):
        # centre indices; an iterate whose distance from the solution is the solver's
        # tolerance, not the arithmetic's
        return None
    prs = _problems(case, seed)
    pairs = sum(len(pr["xy"]) * len(pr["sigma"]) for pr in prs)
    if pairs > 2.2e10:
        return None
    if case["kind"] == "batch":
        if pairs * case["p"] > 6e10:
            return None
        return [torch.cat([_potential(case, pr)[0] for pr in prs])]
    return _potential(case, prs[0])
