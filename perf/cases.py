"""The calls whose speed matters, as a user's program makes them through the public entry points.

A case is one call (or the short sequence that belongs together) on one grid, covariance model and site
set: a draw of an ensemble, the maps made of it, the unconditional fields alone, the solve alone, a new
event's set-up and first ensemble, a step of a covariance fit, a gradient, a batch of events, the closed-form
standard errors.  ``exact`` restates each of them in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2109_11044_gb300 as ce

# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
# nu, range and tau2 are exact in 32 bits, so that a context set up with them is the one that a float32
# parameter tensor names (condsim_loss redoes the set-up where the two differ).
_BASE = dict(sigma=1.0, range=0.125, tau2=0.078125, nu=1.5, layout="cluster70", np=3, prec="f16x3", trend=-1)


def _case(kind, **kw):
    return {"kind": kind, **_BASE, **kw}


def listed():
    return [
        # a small map: 64 x 64 nodes, 200 sites, 10 realizations in the default precision; launches and latency count
        _case("draw", name="draw64", m=64, n=200, R=10, nu=0.5, range=0.1015625, tau2=0.046875, layout="uniform", np=2,
              prec="fp32"),
        # the ShakeMap-sized ensemble: 512 x 512 nodes, 2000 clustered stations, 100 realizations
        _case("draw", name="draw512", m=512, n=2000, R=100, sigma=0.6015625, range=0.1484375, tau2=0.1015625),
        # a large map: 2048 x 2048 nodes, 4000 sites, 8 x 8 neighbourhood
        _case("draw", name="draw2048", m=2048, n=4000, R=32, nu=0.5, range=0.078125, tau2=0.046875,
              layout="uniform+3clusters", np=4),
        # ensemble mean and standard-deviation maps of a ragged grid and site count, in the default precision
        _case("maps", name="maps300", m=300, n=1100, R=50, prec="fp32"),
        # nearest-neighbour Kriging with the circulant correction: 600 sites, about 4500 surrogate nodes
        _case("nn", name="nn512", m=512, n=600, R=50, sigma=0.6015625, range=0.1484375, tau2=0.1015625, layout="uniform",
              k=8, circulant=True),
        # unconditional fields alone, on a grid between the powers of two (embedding 2048)
        _case("fields", name="fields750", m=750, R=64, nu=0.5),
        # the solve alone, on many sites
        _case("solve", name="solve4500", m=256, n=4500, R=100, nu=0.5, range=0.1015625, tau2=0.046875,
              layout="uniform+3clusters"),
        # a new event on a standing grid: site set-up, then the first ensemble
        _case("event", name="event512", m=512, n=2000, R=100, sigma=0.6015625, range=0.1484375, tau2=0.1015625),
        # one step of a covariance fit: set-up at the step's parameters, loss and gradient
        _case("fit", name="fit256", m=256, n=1000, R=16, np=2, prec="fp32"),
        # gradients at fixed parameters: 1024 x 1024 nodes, 3000 sites, centred 200 x 200 window
        _case("grad", name="grad1024", m=1024, n=3000, R=64, np=4, window=200),
        # a queue of uneven events drawn together
        _case("batch", name="batch12", events=12, sizes=2, m=1024, n=3000, R=32, np=4, layout="uniform"),
        # closed-form standard errors at every node, exact and of the draws
        _case("se", name="se256", m=256, n=1000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# a drawn case costs at most this many operations (the largest listed case of its kind has more)
_MOST_FLOPS = {"draw": 1.0e12, "correct": 2.0e11, "maps": 3.0e10, "nn": 1.0e11, "fields": 1.2e11, "solve": 4.0e9,
               "event": 1.0e11, "fit": 2.0e10, "grad": 2.0e11, "batch": 6.0e11, "se": 2.5e11}


def draw(rng):
    """One more case of the listed ones' ranges."""
    while True:
        kind = rng.choice(["draw", "draw", "draw", "correct", "maps", "nn", "fields", "solve", "event", "fit", "grad", "batch",
                           "se"])
        c = _case(kind, layout=rng.choice(["uniform", "cluster70", "uniform+3clusters"]), np=rng.randint(1, 4))
        # a smooth covariance of long range, with little nugget or on a very fine grid, cancels by 10^3 and more in
        # 32 bits: nothing to compare there
        c.update(rng.choice([dict(nu=0.5, range=rng.randint(13, 64) / 256, tau2=rng.randint(3, 24) / 128),
                             dict(nu=1.5, range=rng.randint(13, 38) / 256, tau2=rng.randint(10, 24) / 128)]))
        if kind == "draw":
            c.update(m=_log_int(rng, 61, 2048), n=_log_int(rng, 50, 5000), R=_log_int(rng, 1, 256),
                     prec=rng.choice(["f16x3", "f16x3", "f16x3", "fp32"]),
                     trend=rng.choice([-1, -1, -1, -1, 0, 1]))
            if c["prec"] == "fp32":
                c["m"] = min(c["m"], 700)
            if c["nu"] == 1.5:
                c["m"] = min(c["m"], 1024)
        elif kind == "correct":   # the contraction alone, in every precision form
            c.update(m=_log_int(rng, 61, 700), n=_log_int(rng, 50, 2000), R=_log_int(rng, 1, 200),
                     prec=rng.choice(["fp32", "f16x3", "tf32x3", "bf16x3"]))
        elif kind == "maps":
            c.update(m=_log_int(rng, 61, 500), n=_log_int(rng, 50, 1500), R=_log_int(rng, 2, 150),
                     prec=rng.choice(["fp32", "f16x3"]))
        elif kind == "nn":
            c.update(m=_log_int(rng, 64, 700), n=_log_int(rng, 50, 600), R=_log_int(rng, 1, 100), layout="uniform",
                     k=rng.choice([1, 4, 8]), circulant=rng.random() < 0.6)
        elif kind == "fields":
            c.update(m=_log_int(rng, 61, 2048), R=_log_int(rng, 1, 200))
        elif kind == "solve":
            c.update(m=256, n=_log_int(rng, 50, 4500), R=_log_int(rng, 1, 130), prec=rng.choice(["fp32", "f16x3"]))
        elif kind == "event":
            c.update(m=_log_int(rng, 61, 700), n=_log_int(rng, 50, 2500), R=_log_int(rng, 4, 100))
        elif kind == "fit":
            c.update(m=_log_int(rng, 61, 400), n=_log_int(rng, 50, 1500), R=_log_int(rng, 2, 32), np=rng.randint(1, 3),
                     prec=rng.choice(["fp32", "f16x3"]))
        elif kind == "grad":
            m = _log_int(rng, 128, 1024)
            c.update(m=m, n=_log_int(rng, 100, 3000), R=_log_int(rng, 2, 64), window=max(16, m // 5))
        elif kind == "batch":
            c.update(events=rng.randint(2, 12), sizes=rng.randint(1, 10 ** 6), m=1024, n=2000, R=_log_int(rng, 8, 32), np=4,
                     layout="uniform")
        elif kind == "se":
            c.update(m=_log_int(rng, 61, 256), n=_log_int(rng, 35, 1000))
        if work(c)["flops"] <= _MOST_FLOPS[kind]:
            return c


def _batch_events(case):
    """The events of a batch: grid side, sites and covariance of each, fixed by the case."""
    rng = np.random.default_rng(case["sizes"])
    sides = [s for s in (128, 192, 256, 384, 512, 768, 1024) if s <= case["m"]]
    events = []
    for _ in range(case["events"]):
        nu = float(rng.choice([0.5, 1.5]))
        events.append(dict(case, kind="draw", m=int(rng.choice(sides)), nu=nu,
                           n=int(round(math.exp(rng.uniform(math.log(100), math.log(case["n"]))))),
                           range=float(rng.uniform(0.05, 0.3 if nu == 0.5 else 0.15)), tau2=float(rng.uniform(0.06, 0.2))))
    return events


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _clustered(rng, count, centre, sd):
    out = np.empty((0, 2))
    while out.shape[0] < count:
        pts = centre + sd * rng.standard_normal((2 * (count - out.shape[0]) + 8, 2))
        out = np.concatenate([out, pts[np.all((pts >= 0.0) & (pts <= 1.0), axis=1)]])
    return out[:count]


def _inputs(case, seed):
    """Sites on the unit square (n x 2, FP64), float32 data at them and the simulation's seed."""
    rng = np.random.default_rng([seed, 17])
    n, lay = case["n"], case["layout"]
    if lay == "uniform":
        sites = rng.uniform(size=(n, 2))
    elif lay == "cluster70":
        nc = int(round(0.7 * n))
        sites = np.concatenate([_clustered(rng, nc, rng.uniform(0.2, 0.8, 2), 0.1), rng.uniform(size=(n - nc, 2))])
    else:
        nc = n // 10
        parts = [_clustered(rng, nc, rng.uniform(0.2, 0.8, 2), 0.03) for _ in range(3)]
        sites = np.concatenate([rng.uniform(size=(n - 3 * nc, 2)), *parts])
    sites = sites[rng.permutation(n)]
    # a random-Fourier-feature field of the case's range and smoothness, plus the nugget
    nf = 256
    freq = rng.standard_normal((nf, 2)) / (case["range"] * np.sqrt(rng.chisquare(2 * case["nu"], (nf, 1)) / (2 * case["nu"])))
    z = case["sigma"] * math.sqrt(2.0 / nf) * np.cos(sites @ freq.T + rng.uniform(0, 2 * math.pi, nf)).sum(1)
    z = z + math.sqrt(case["tau2"]) * rng.standard_normal(n)
    if case["trend"] >= 0:
        z = z + 1.5 + 0.7 * sites[:, 0]
    return sites, z.astype(np.float32), int(rng.integers(1, 1 << 40))


def _context(case):
    return ce.Context(case["m"], 0.0, 0.0, 1.0 / (case["m"] - 1), case["sigma"], case["range"], case["nu"], case["tau2"])


def _sited(case, sites):
    ctx = _context(case)
    if case["kind"] == "nn":
        ctx.krige_weights(sites, "nn", k=case["k"], prec=case["prec"])
        ctx.set_nn_correction("circulant" if case["circulant"] else "direct")
    else:
        ctx.krige_weights(sites, "local", np_=case["np"], prec=case["prec"])
        if case["trend"] >= 0:
            ctx.set_trend(case["trend"])
    return ctx


def _fit_theta(case):
    """The parameters of a fit's step, away from those of the context it starts from."""
    return [case["sigma"] * 1.0625, case["range"] * 1.125, case["tau2"] * 0.875]


def _window(case):
    w = case.get("window", case["m"] // 2)
    a = (case["m"] - w) // 2
    return (a, a + w, a, a + w)


def _solve_rhs(case, seed):
    g = torch.Generator().manual_seed(seed + 5)
    return torch.randn((case["R"], case["n"]), generator=g, dtype=torch.float32)


def _weights(case, seed):
    """Weights A^-1 e of random residuals e, R x n float32: of the size and alternation that the solve gives."""
    s = torch.from_numpy(_inputs(case, seed)[0]).to(_dev())
    A = _matern(_dist(s, s), case["sigma"], case["range"], case["nu"])
    A += case["tau2"] * torch.eye(len(s), dtype=_F64, device=A.device)
    E = _solve_rhs(case, seed).to(A.device).to(_F64)
    return torch.cholesky_solve(E.T, torch.linalg.cholesky(A)).T.contiguous().float()


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "fields":
        st["ctx"] = _context(case)
        st["seed"] = int(np.random.default_rng([seed, 3]).integers(1, 1 << 40))
        return st
    if kind == "batch":
        ctxs, zs, seeds, outs = [], [], [], []
        for e, ev in enumerate(_batch_events(case)):
            sites, z, s = _inputs(ev, seed * 100 + e)
            ctxs.append(_sited(ev, sites))
            zs.append(torch.from_numpy(z).cuda())
            seeds.append(s)
            outs.append(torch.empty((ev["R"], ev["m"], ev["m"]), dtype=torch.float32, device="cuda"))
        st["outs"] = outs
        st["batch"] = ce.Batch(ctxs, zs, [case["R"]] * len(ctxs), seeds, [0] * len(ctxs), outs)
        return st
    sites, z, st["seed"] = _inputs(case, seed)
    st["z"] = torch.from_numpy(z).cuda()
    if kind == "event":
        st["sites"] = sites
        st["ctx"] = _context(case)
        return st
    st["ctx"] = _sited(case, sites)
    if kind == "solve":
        st["E"] = _solve_rhs(case, seed).cuda()
    if kind == "correct":
        st["B"] = _weights(case, seed)
    if kind in ("fit", "grad"):
        theta = _fit_theta(case) if kind == "fit" else [case["sigma"], case["range"], case["tau2"]]
        st["theta"] = torch.tensor(theta, dtype=torch.float32, requires_grad=True)
        st["z"].requires_grad_(True)
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(st):
    case, kind = st["case"], st["kind"]
    if kind in ("draw", "nn"):
        return st["ctx"].condsim(st["z"], case["R"], st["seed"])
    if kind == "maps":
        v = st["ctx"].condsim(st["z"], case["R"], st["seed"])
        mean, sd = st["ctx"].ensemble_stats(st["ctx"].moments(v, case["R"]), case["R"])
        return {"v": v, "mean": mean, "sd": sd}
    if kind == "fields":
        return st["ctx"].unconditional(case["R"], st["seed"])
    if kind == "solve":
        return st["ctx"].solve(st["E"])
    if kind == "correct":
        return st["ctx"].correct(st["B"], torch.zeros((case["R"], case["m"], case["m"]), device="cuda"))
    if kind == "event":
        st["ctx"].krige_weights(st["sites"], "local", np_=case["np"], prec=case["prec"])
        return st["ctx"].condsim(st["z"], case["R"], st["seed"])
    if kind in ("fit", "grad"):
        loss = ce.condsim_loss(st["ctx"], st["theta"], st["z"], case["R"], st["seed"], _window(case))
        dtheta, dz = torch.autograd.grad(loss, [st["theta"], st["z"]])
        return {"dtheta": dtheta, "dz": dz}
    if kind == "batch":
        st["batch"].launch()
        return list(st["outs"])
    if kind == "se":
        exact, approx = st["ctx"].se_map()
        return {"exact": exact, "approx": approx}
    raise ValueError(kind)


def work(case):
    """Bytes and operations a pass cannot do without: inputs and the set-up's arrays read once, outputs written
    once; the pruned 2-D transforms, the off-grid gather, the solve, the contraction with a covariance of about
    ten operations an element, n^3 for the FP64 inverse."""
    kind, m = case["kind"], case["m"]
    if kind == "batch":
        parts = [work(e) for e in _batch_events(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    M, n, R = m * m, case.get("n", 0), case.get("R", 0)
    P = 1 << (2 * m - 1).bit_length()
    fft = (R + 1) // 2 * 5.0 * P * math.log2(P) * (P + m)
    b_fft = 4.0 * P * P + 4.0 * R * M
    if kind == "fields":
        return {"bytes": b_fft, "flops": fft}
    rows = min(n * case["k"], M) if kind == "nn" else n
    solve, b_solve = 2.0 * rows * rows * R, 8.0 * rows * rows + 8.0 * R * rows
    if kind == "solve":
        return {"bytes": b_solve, "flops": solve}
    if kind == "se":
        return {"bytes": 8.0 * n * n + 8.0 * M, "flops": 4.0 * M * n * n}
    corr = fft if kind == "nn" and case["circulant"] else M * rows * (2.0 * R + 10.0)
    if kind == "correct":
        return {"bytes": 4.0 * R * M + 4.0 * R * n, "flops": corr}
    flops = fft + 2.0 * R * n * 4 * case["np"] ** 2 + solve + corr
    nbytes = b_fft + b_solve
    if kind == "maps":
        nbytes += 4.0 * R * M + 24.0 * M
        flops += 3.0 * R * M
    if kind in ("event", "fit"):
        flops += 1.0 * n ** 3
        nbytes += 8.0 * n * n
    if kind in ("fit", "grad"):
        w = _window(case)
        nw = (w[1] - w[0]) * (w[3] - w[2])
        flops += 2 * fft + 2 * solve + 4.0 * nw * n * R
        nbytes += 8.0 * R * M + 8.0 * n * n
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------
_F64 = torch.float64


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _matern(d, sigma, theta, nu):
    if nu == 1.5:
        t = math.sqrt(3.0) * d / theta
        return sigma ** 2 * (1.0 + t) * torch.exp(-t)
    return sigma ** 2 * torch.exp(-d / theta)


def _dist(a, b):
    return torch.sqrt((a[:, None, 0] - b[None, :, 0]) ** 2 + (a[:, None, 1] - b[None, :, 1]) ** 2)


def _philox(c0, c1, c2, seed):
    """Philox4x32-10 at counters (c0, c1, c2, 0), int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF
    k0, k1 = seed & mask, (seed >> 32) & mask
    c = [c0, c1 + torch.zeros_like(c0), c2 + torch.zeros_like(c0), torch.zeros_like(c0)]

    def mul(const, x):
        lo = const * (x & 0xFFFF)
        t = const * (x >> 16) + (lo >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _normals(a, b):
    u1, u2 = (a.to(_F64) + 0.5) * 2.0 ** -32, (b.to(_F64) + 0.5) * 2.0 ** -32
    r = torch.sqrt(-2.0 * torch.log(u1))
    return r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)


def _spectrum(case, theta):
    """(P, sqrt(lambda / P^2)) of the embedding, grown while it is indefinite, negative eigenvalues clipped."""
    h, dev = 1.0 / (case["m"] - 1), _dev()
    P = 1
    while P < 2 * case["m"]:
        P *= 2
    for _ in range(4):
        a = torch.arange(P, device=dev, dtype=_F64)
        w = torch.minimum(a, P - a)
        d = h * torch.sqrt(w[:, None] ** 2 + w[None, :] ** 2)
        lam = torch.fft.fft2(_matern(d, theta[0], theta[1], case["nu"])).real
        if float(lam.detach().min()) >= -1e-6 * float(lam.detach().max()):
            break
        P *= 2
    pos = lam > 0
    return P, torch.where(pos, torch.sqrt(torch.where(pos, lam, torch.ones_like(lam))), torch.zeros_like(lam)) / P


def _fields(case, P, s, seed, R):
    dev, m = _dev(), case["m"]
    ctr = torch.arange(P // 2 * P, device=dev, dtype=torch.int64).reshape(P // 2, P)
    y = []
    for p in range((R + 1) // 2):
        x = _philox(ctr, torch.tensor(p, device=dev), torch.tensor(0, device=dev), seed)
        eps = torch.cat([torch.complex(*_normals(x[0], x[1])), torch.complex(*_normals(x[2], x[3]))])
        w = torch.fft.fft2(s * eps)[:m, :m]
        y += [w.real.clone(), w.imag.clone()]
    return torch.stack(y[:R])


def _nugget(n, R, seed):
    dev = _dev()
    i = torch.arange((n + 3) // 4, device=dev, dtype=torch.int64)[None, :].expand(R, -1).contiguous()
    r = torch.arange(R, device=dev, dtype=torch.int64)[:, None]
    x = _philox(i, r, torch.tensor(1, device=dev), seed)
    z = torch.stack([*_normals(x[0], x[1]), *_normals(x[2], x[3])], -1)
    return z.reshape(R, -1)[:, :n]


def _windows(case, sites, theta):
    """Window nodes, weights W_1 and conditional variance of every site."""
    m, npr, h = case["m"], case["np"], 1.0 / (case["m"] - 1)
    g = torch.floor((sites - 0.0) / h).long()
    start = torch.clamp(g - npr + 1, 0, m - 2 * npr)
    o = torch.arange(2 * npr, device=sites.device)
    ii = (start[:, 1, None, None] + o[None, :, None]).expand(-1, -1, 2 * npr).reshape(len(sites), -1)
    jj = (start[:, 0, None, None] + o[None, None, :]).expand(-1, 2 * npr, -1).reshape(len(sites), -1)
    k21 = _matern(torch.sqrt((sites[:, 0, None] - jj * h) ** 2 + (sites[:, 1, None] - ii * h) ** 2), theta[0], theta[1], case["nu"])
    w = torch.stack([o.repeat_interleave(2 * npr), o.repeat(2 * npr)], -1).to(_F64) * h
    W = torch.linalg.solve(_matern(_dist(w, w), theta[0], theta[1], case["nu"]), k21.T).T
    return ii * m + jj, W, theta[0] ** 2 - (W * k21).sum(1)


def _add_correction(case, pts, Bt, y):
    """y (R x M) += (K(grid, pts) Bt)^T, Bt: points x R."""
    m, h = case["m"], 1.0 / (case["m"] - 1)
    step = max(1, (1 << 27) // pts.shape[0])
    for a in range(0, m * m, step):
        g = torch.arange(a, min(m * m, a + step), device=y.device)
        nodes = torch.stack([g % m, g // m], -1).to(_F64) * h
        y[:, a:a + step] += (_matern(_dist(nodes, pts), case["sigma"], case["range"], case["nu"]) @ Bt).T
    return y


def _exact_local(case, seed):
    sites, z, sim = _inputs(case, seed)
    dev, R, m, h = _dev(), case["R"], case["m"], 1.0 / (case["m"] - 1)
    theta = (case["sigma"], case["range"])
    s, zt = torch.from_numpy(sites).to(dev), torch.from_numpy(z).to(dev).to(_F64)
    P, sq = _spectrum(case, theta)
    y = _fields(case, P, sq, sim, R).reshape(R, -1)
    idx, W, gamma = _windows(case, s, theta)
    phi = torch.sqrt(case["tau2"] + torch.clamp(gamma, min=0.0))
    E = torch.empty((R, case["n"]), dtype=_F64, device=dev)
    for r in range(R):
        E[r] = zt - (W * y[r][idx]).sum(1)
    E -= phi * _nugget(case["n"], R, sim)
    A = _matern(_dist(s, s), *theta, case["nu"]) + case["tau2"] * torch.eye(case["n"], dtype=_F64, device=dev)
    L = torch.linalg.cholesky(A)
    B = torch.cholesky_solve(E.T, L)
    if case["trend"] >= 0:
        def basis(u):   # 1, and the centred grid coordinates over m
            one = torch.ones((len(u), 1), dtype=_F64, device=dev)
            return one if case["trend"] == 0 else torch.cat([one, (u / h - 0.5 * (m - 1)) / m], 1)
        X = basis(s)
        F = torch.cholesky_solve(X, L)
        beta = torch.linalg.solve(X.T @ F, F.T @ E.T)
        B = B - F @ beta
        g = torch.arange(m * m, device=dev)
        y += (basis(torch.stack([g % m, g // m], -1).to(_F64) * h) @ beta).T
    return _add_correction(case, s, B, y).reshape(R, m, m)


def _nn_nodes(case, sites):
    m, h, dev = case["m"], 1.0 / (case["m"] - 1), sites.device
    g = torch.floor(sites / h).long()
    o = torch.arange(-2, 4, device=dev)
    ii = (g[:, 1, None, None] + o[None, :, None]).expand(-1, -1, 6).reshape(len(sites), -1)
    jj = (g[:, 0, None, None] + o[None, None, :]).expand(-1, 6, -1).reshape(len(sites), -1)
    d2 = (sites[:, 0, None] - jj * h) ** 2 + (sites[:, 1, None] - ii * h) ** 2
    d2 = torch.where((ii < 0) | (ii >= m) | (jj < 0) | (jj >= m), torch.full_like(d2, math.inf), d2)
    order = torch.sort(d2, dim=1, stable=True).indices[:, :case["k"]]   # candidates ascend in the flat index
    return torch.unique((ii * m + jj).gather(1, order))


def _exact_nn(case, seed):
    sites, z, sim = _inputs(case, seed)
    dev, R, m, h, n = _dev(), case["R"], case["m"], 1.0 / (case["m"] - 1), case["n"]
    theta = (case["sigma"], case["range"])
    s, zt = torch.from_numpy(sites).to(dev), torch.from_numpy(z).to(dev).to(_F64)
    J = _nn_nodes(case, s)
    pts = torch.stack([J % m, J // m], -1).to(_F64) * h
    A = _matern(_dist(s, s), *theta, case["nu"]) + case["tau2"] * torch.eye(n, dtype=_F64, device=dev)
    K = _matern(_dist(pts, s), *theta, case["nu"])
    WN = torch.cholesky_solve(K.T, torch.linalg.cholesky(A)).T
    sig = case["sigma"] ** 2 - (WN * K).sum(1)
    P, sq = _spectrum(case, theta)
    y = _fields(case, P, sq, sim, R).reshape(R, -1)
    phi = torch.sqrt(torch.clamp(sig, min=0.0) + case["tau2"])
    E = (WN @ zt) - (y[:, J] + phi * _nugget(len(J), R, sim))
    AN = _matern(_dist(pts, pts), *theta, case["nu"]) + torch.diag(case["tau2"] + sig)
    B = torch.cholesky_solve(E.T, torch.linalg.cholesky(AN))
    if not case["circulant"]:
        return _add_correction(case, pts, B, y).reshape(R, m, m)
    lam = (sq * P) ** 2
    for r in range(R):
        b = torch.zeros((P, P), dtype=_F64, device=dev)
        b[J // m, J % m] = B[:, r]
        y[r] += torch.fft.ifft2(lam * torch.fft.fft2(b)).real[:m, :m].reshape(-1)
    return y.reshape(R, m, m)


def _exact_grad(case, seed):
    """Gradients of (1/R) sum_r mean_window v_r^2 + log-likelihood by automatic differentiation."""
    sites, z, sim = _inputs(case, seed)
    dev, R, m, h, n = _dev(), case["R"], case["m"], 1.0 / (case["m"] - 1), case["n"]
    th = _fit_theta(case) if case["kind"] == "fit" else [case["sigma"], case["range"], case["tau2"]]
    th = torch.tensor(th, dtype=torch.float32).to(_F64).to(dev).requires_grad_(True)   # the values the call is given
    s, zt = torch.from_numpy(sites).to(dev), torch.from_numpy(z).to(dev).to(_F64).requires_grad_(True)
    P, sq = _spectrum(case, th)
    y = _fields(case, P, sq, sim, R).reshape(R, -1)
    idx, W, gamma = _windows(case, s, th)
    phi = torch.sqrt(th[2] + gamma)
    E = torch.stack([zt - (W * y[r][idx]).sum(1) for r in range(R)]) - phi * _nugget(n, R, sim)
    A = _matern(_dist(s, s), th[0], th[1], case["nu"]) + th[2] * torch.eye(n, dtype=_F64, device=dev)
    L = torch.linalg.cholesky(A)
    B = torch.cholesky_solve(torch.cat([E.T, zt[:, None]], 1), L)
    i0, i1, j0, j1 = _window(case)
    g = torch.arange(m * m, device=dev).reshape(m, m)[i0:i1, j0:j1].reshape(-1)
    K = _matern(_dist(torch.stack([g % m, g // m], -1).to(_F64) * h, s), th[0], th[1], case["nu"])
    v = y[:, g] + (K @ B[:, :R]).T
    ll = -0.5 * (zt @ B[:, R]) - torch.log(torch.diagonal(L)).sum() - 0.5 * n * math.log(2 * math.pi)
    dth, dz = torch.autograd.grad((v ** 2).mean() + ll, [th, zt])
    return {"dtheta": dth, "dz": dz}


def _exact_se(case, seed):
    sites, _, _ = _inputs(case, seed)
    dev, m, h, n = _dev(), case["m"], 1.0 / (case["m"] - 1), case["n"]
    theta = (case["sigma"], case["range"])
    s = torch.from_numpy(sites).to(dev)
    g = torch.arange(m * m, device=dev)
    nodes = torch.stack([g % m, g // m], -1).to(_F64) * h
    K = _matern(_dist(s, nodes), *theta, case["nu"])
    A = _matern(_dist(s, s), *theta, case["nu"]) + case["tau2"] * torch.eye(n, dtype=_F64, device=dev)
    w = torch.cholesky_solve(K, torch.linalg.cholesky(A))
    exact = torch.sqrt(torch.clamp(theta[0] ** 2 - (K * w).sum(0), min=0.0))
    idx, W, gamma = _windows(case, s, theta)
    a = torch.arange(m, device=dev, dtype=_F64) * h
    tab = _matern(torch.sqrt(a[:, None] ** 2 + a[None, :] ** 2), *theta, case["nu"])
    U = torch.zeros((n, m * m), dtype=_F64, device=dev)
    gi, gj = (g // m)[None, :], (g % m)[None, :]
    for k in range(idx.shape[1]):
        p = idx[:, k, None]
        U += W[:, k, None] * tab[(p // m - gi).abs(), (p % m - gj).abs()]
    Q = torch.stack([(U[:, idx[j]] * W[j]).sum(1) for j in range(n)], 1)
    Q += torch.diag(case["tau2"] + torch.clamp(gamma, min=0.0))
    var = theta[0] ** 2 - 2 * (w * U).sum(0) + (w * (Q @ w)).sum(0)
    return {"exact": exact.reshape(m, m), "approx": torch.sqrt(torch.clamp(var, min=0.0)).reshape(m, m)}


def exact(case, seed):
    kind = case["kind"]
    with torch.set_grad_enabled(kind in ("fit", "grad")):
        if kind in ("draw", "event"):
            return _exact_local(case, seed)
        if kind == "maps":
            v = _exact_local(case, seed)
            return {"v": v, "mean": v.mean(0), "sd": v.std(0)}
        if kind == "nn":
            return _exact_nn(case, seed)
        if kind == "fields":
            sim = int(np.random.default_rng([seed, 3]).integers(1, 1 << 40))
            return _fields(case, *_spectrum(case, (case["sigma"], case["range"])), sim, case["R"])
        if kind == "solve":
            sites, _, _ = _inputs(case, seed)
            s = torch.from_numpy(sites).to(_dev())
            A = _matern(_dist(s, s), case["sigma"], case["range"], case["nu"])
            A += case["tau2"] * torch.eye(len(s), dtype=_F64, device=A.device)
            E = _solve_rhs(case, seed).to(A.device).to(_F64)
            return torch.cholesky_solve(E.T, torch.linalg.cholesky(A)).T.contiguous()
        if kind == "correct":
            s = torch.from_numpy(_inputs(case, seed)[0]).to(_dev())
            y = torch.zeros((case["R"], case["m"] ** 2), dtype=_F64, device=s.device)
            B = _weights(case, seed).to(_F64)
            return _add_correction(case, s, B.T, y).reshape(case["R"], case["m"], case["m"])
        if kind in ("fit", "grad"):
            return _exact_grad(case, seed)
        if kind == "batch":
            return [_exact_local(ev, seed * 100 + e) for e, ev in enumerate(_batch_events(case))]
        if kind == "se":
            return _exact_se(case, seed)
    raise ValueError(kind)
