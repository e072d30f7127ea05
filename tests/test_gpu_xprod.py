"""The solve from exact 8-bit digits on the tensor cores (1800 rows and more) at the edges of
its 128-row tiles, 64-column chunks, 256-column accumulation units and blocks of 128
right-hand sides, against an FP64 solve.

Tolerance: output rounding is 2^-25 of a value's own binade (RMS 0.3 x 2^-24 = 1.8e-8 of the
value, at most 6e-8), the digits leave 2^-40 sqrt(n) of the largest products; held to 1e-7
(L2 norm) per right-hand side, the accuracy the header states."""
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


@pytest.mark.parametrize("n", [1800, 1919, 1921, 2048, 2305])
def test_digit_solve_edges(ce, n):
    wl = workloads.workload("plain64").scaled(n=n)
    sites = workloads.make_sites(wl)
    ctx = ce.Context.from_workload(wl).krige_weights(sites, "local", np_=wl.np_, prec="f16x3")
    prob = oracle.Problem(wl.m, wl.x0, wl.y0, wl.h, wl.sigma, wl.range, wl.nu, wl.tau2)
    A = prob.cov(sites, sites) + wl.tau2 * np.eye(n)
    E = np.random.default_rng(n).standard_normal((257, n)).astype(np.float32)
    E[3] *= 1e20
    E[4] *= 1e-20
    E[5] = 0.0
    want = np.linalg.solve(A, E.astype(np.float64).T).T
    full = ctx.solve(torch.from_numpy(E).cuda()).cpu().numpy().astype(np.float64)
    err = np.linalg.norm(full - want, axis=1) / np.maximum(np.linalg.norm(want, axis=1), 1e-300)
    assert err.max() < 1e-7 and not full[5].any()
    for R in (1, 16, 17, 128, 129):   # a right-hand side's solution does not depend on the others
        part = ctx.solve(torch.from_numpy(E[:R]).cuda()).cpu().numpy()
        assert np.array_equal(part, full[:R].astype(np.float32))


def test_digit_solve_keeps_non_finite_rows_apart(ce):
    wl = workloads.workload("plain64").scaled(n=1800)
    sites = workloads.make_sites(wl)
    ctx = ce.Context.from_workload(wl).krige_weights(sites, "local", np_=wl.np_)
    E = torch.randn((3, 1800), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    clean = ctx.solve(E)
    bad = E.clone()
    bad[1, 7] = float("nan")
    got = ctx.solve(bad)
    assert torch.isnan(got[1]).all()
    assert torch.equal(got[0], clean[0]) and torch.equal(got[2], clean[2])
