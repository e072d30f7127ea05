"""The ensemble's register passes (torus sizes 1024, 2048 and 4096: 1, 2 and 4 warps per line)
at ragged and edge field sizes: just past a torus size's smallest, its largest, a field of at
most 1024 nodes a side on a 4096 torus (one output per partial transform) and one node more
(two for the first), odd numbers of realizations and a lone pair, against the oracle's FP64
transform of the same noise.

Tolerance: 24 butterfly stages of FP32 rounding, 0.3 x 2^-24 x sqrt(24) = 9e-8 RMS of the
fields, and normals within 1e-6 of their size: 2e-6 in the L2 norm."""
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


@pytest.mark.parametrize("m,P,nu,range_,R", [
    (257, 1024, 0.5, 0.05, 3), (512, 1024, 0.5, 0.02, 2), (513, 2048, 0.5, 0.05, 5), (1024, 2048, 0.5, 0.01, 1),
    (1024, 4096, 1.5, 0.3, 3), (1025, 4096, 0.5, 0.01, 2), (1541, 4096, 0.5, 0.05, 3), (2048, 4096, 0.5, 0.01, 1)])
def test_register_passes(ce, m, P, nu, range_, R):
    wl = workloads.workload("plain64").scaled(m=m, nu=nu, range=range_)
    ctx = ce.Context.from_workload(wl)
    lam, P_oracle, _ = oracle.ce_eigenvalues(wl.m, wl.h, wl.sigma, wl.range, wl.nu)
    assert ctx.info()["P"] == P == P_oracle
    want = oracle.ce_unconditional(lam, m, 11, 4, R).reshape(R, m, m)
    got = ctx.unconditional(R, seed=11, r_offset=4).cpu().numpy()
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    assert err < 2e-6, err


@pytest.mark.parametrize("m,P", [(300, 1024), (600, 2048), (1030, 4096)])
def test_register_adjoint(ce, m, P):
    """The gradient's adjoint passes at the same torus sizes: the derivative of the loss along
    (sigma, range) against the oracle's central difference at fixed noise, held to its own
    error (step 1e-4) as the small grids' test holds it: 2e-3."""
    wl = workloads.workload("plain64").scaled(m=m, nu=0.5, sigma=0.8, range=0.15, tau2=0.06, n=20, R=3, site_seed=9)
    sites = workloads.make_sites(wl)
    z = workloads.make_data(wl, sites).astype(np.float32)
    win = (m // 8, m // 2, m // 4, m - 7)
    ctx = ce.Context.from_workload(wl).krige_weights(sites, "local", np_=2)
    assert ctx.info()["P"] == P
    _, gt, _, L = ctx.condsim_grad(torch.from_numpy(z).cuda(), 3, 31, win)
    up, dn = (oracle.diff_loss(wl.m, wl.x0, wl.y0, wl.h, wl.sigma * (1 + s), wl.range * (1 - s), wl.nu, wl.tau2, sites,
                               z.astype(np.float64), 2, 31, 0, 3, win) for s in (1e-4, -1e-4))
    want = (up - dn) / 2e-4
    got = gt[0] * wl.sigma - gt[1] * wl.range
    assert abs(L - 0.5 * (up + dn)) < 1e-4 * abs(L)
    assert abs(got - want) < 2e-3 * max(abs(gt[0] * wl.sigma), abs(gt[1] * wl.range)), (got, want)
