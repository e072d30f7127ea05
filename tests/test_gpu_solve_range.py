"""The FP32-form solve from 1800 rows on, for right-hand sides whose elements span many
binades: one value far above the others (a bad station), a single non-zero, values that
decay across the domain, values near the ends of the FP32 range.

Tolerance, element by element: the products are rounded to FP32 in chains of at most four
(4 x 2^-24 of sum_j |A^-1_ij e_j|), and the FP64 inverse carries about 2^-53 cond(A) of its
largest value: 2^-22 (|A^-1| |e|)_i + 2^-53 cond(A) max |A^-1| max |e|."""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ce():
    from paper_2109_11044_gb300.build import build
    build()
    import paper_2109_11044_gb300 as mod
    mod.load_library()
    return mod


@pytest.mark.parametrize("n,prec", [(1800, "fp32"), (1847, "f16x3")])
def test_wide_right_hand_sides(ce, n, prec):
    wl = workloads.workload("plain64").scaled(n=n)
    sites = workloads.make_sites(wl)
    ctx = ce.Context.from_workload(wl).krige_weights(sites, "local", np_=wl.np_, prec=prec)
    prob = oracle.Problem(wl.m, wl.x0, wl.y0, wl.h, wl.sigma, wl.range, wl.nu, wl.tau2)
    A = prob.cov(sites, sites) + wl.tau2 * np.eye(n)
    lam = np.linalg.eigvalsh(A)
    Ainv = np.linalg.inv(A)
    E = np.random.default_rng(n).standard_normal((131, n)).astype(np.float32)
    wide = [0, 3, 4, 40, 41, 64, 95, 96, 127, 128, 130]
    for r, f in zip(wide[:5], (3e2, 1e4, 1e6, 1e9, 1e20)):
        E[r, 17 * r + 5] = f
    E[41] = 0.0
    E[41, n - 1] = 1.0
    E[64] *= np.exp(-25.0 * sites[:, 0]).astype(np.float32)
    E[95] *= np.float32(1e33)
    E[96] *= np.float32(1e-33)
    E[127, :n // 2] = 0.0
    E[128, -3:] = 1e7
    E[130, :40] *= 1e-6
    B = ctx.solve(torch.from_numpy(E).cuda()).cpu().numpy()
    E64 = E.astype(np.float64)
    want = np.linalg.solve(A, E64.T).T
    tol = 2.0 ** -22 * (np.abs(E64) @ np.abs(Ainv)) + \
        2.0 ** -53 * lam[-1] / lam[0] * np.abs(Ainv).max() * np.abs(E64).max(1, keepdims=True)
    bad = np.abs(B - want) > tol
    assert not bad.any(), [(r, int(bad[r].sum()), float((np.abs(B - want) / tol)[r].max())) for r in np.flatnonzero(bad.any(1))]
    for rows in ([0], [4, 5], wide, list(range(33))):   # no solution depends on the others
        part = ctx.solve(torch.from_numpy(E[rows]).cuda()).cpu().numpy()
        assert np.array_equal(part, B[rows])
