"""The FP64 block-sweep inverse of the prediction matrix at the edges of its 32-column
pivots, 64-column sweeps and 128-row tiles, against the oracle's Cholesky: the Gaussian
log-likelihood (log-determinant and quadratic form in FP64) and a solve.

Tolerances: the inverse carries a relative error of about n eps cond(A); cond(A) is at
most n (sigma^2 + tau^2) / tau^2, i.e. below 1.5e4 for tau^2 = 0.05 and below 7e6 for
tau^2 = 1e-4 at n = 700, so n eps cond stays below 1.2e-9 and 6e-7.  The solve is held to
the FP32 bar of 1e-5 of its largest value."""
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


@pytest.mark.parametrize("tau2,tol", [(0.05, 1.2e-9), (1e-4, 6e-7)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 257, 700])
def test_inverse_edges(ce, n, tau2, tol):
    wl = workloads.workload("plain64").scaled(n=n, tau2=tau2)
    sites = workloads.make_sites(wl)
    z = workloads.make_data(wl, sites).astype(np.float32)
    ctx = ce.Context.from_workload(wl).krige_weights(sites, "local", np_=wl.np_)
    prob = oracle.Problem(wl.m, wl.x0, wl.y0, wl.h, wl.sigma, wl.range, wl.nu, wl.tau2)
    oracle.setup_local(prob, sites, z, wl.np_)
    ref = oracle.log_likelihood(prob)
    assert abs(ctx.loglik(torch.from_numpy(z).cuda()) - ref) <= tol * abs(ref)
    E = np.random.default_rng(n).standard_normal((3, n)).astype(np.float32)
    B = ctx.solve(torch.from_numpy(E).cuda()).cpu().numpy().astype(np.float64)
    want = oracle.solve_B(prob, E).T
    assert np.abs(B - want).max() <= 1e-5 * np.abs(want).max()


def test_coincident_sites_without_nugget_are_not_spd(ce):
    wl = workloads.workload("plain64").scaled(n=70, tau2=0.0)
    sites = workloads.make_sites(wl)
    sites[69] = sites[3]
    ctx = ce.Context.from_workload(wl)
    with pytest.raises(ce.CEError) as err:
        ctx.krige_weights(sites, "local", np_=wl.np_)
    assert err.value.status == ce.CE_ERR_NOT_SPD
