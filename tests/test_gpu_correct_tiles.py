"""The FP32 correction at the edges of its tiles: realization tiles of 16, 32, 64 and 128, node
tiles of 32, 64 and 128 (which one a call gets depends on nodes x realizations; the grids' node
counts are ragged in all three), 70 sites (two chunks of 32 and a remainder), isotropic and
anisotropic, against the oracle's FP64 correction.

Tolerance: 70 rounded products of values of order one, summed in chunks of 32 FP32 additions
(RMS 0.3 x 2^-24 sqrt(32) = 1e-7 of the largest partial sum) and one rounding of the result:
1e-6 in the L2 norm.  Every tile makes the same sum, so a realization computed alone has the
same bits."""
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


@pytest.mark.parametrize("m", [77, 143, 203])
@pytest.mark.parametrize("aniso", [None, (0.45, 0.7)])
def test_fp32_correction_tiles(ce, m, aniso):
    wl = workloads.workload("plain64").scaled(m=m, n=70, nu=1.5 if m == 143 else 0.5)
    sites = workloads.make_sites(wl)
    ctx = ce.Context.from_workload(wl)
    if aniso:
        ctx.set_anisotropy(*aniso)
    ctx.krige_weights(sites, "local", np_=wl.np_, prec="fp32")
    prob = oracle.Problem(wl.m, wl.x0, wl.y0, wl.h, wl.sigma, wl.range, wl.nu, wl.tau2, aniso=aniso)
    oracle.setup_local(prob, sites, workloads.make_data(wl, sites), wl.np_)
    B = np.random.default_rng(m).standard_normal((129, 70)).astype(np.float32)
    y = np.random.default_rng(m + 1).standard_normal((129, m, m)).astype(np.float32)
    want = oracle.correction(prob, y.astype(np.float64), B.T.astype(np.float64)).reshape(129, m, m)
    Bd, yd = torch.from_numpy(B).cuda(), torch.from_numpy(y).cuda()
    alone = ctx.correct(Bd[128:], yd[128:].clone()).cpu().numpy()[0]
    for R in (1, 15, 16, 17, 32, 33, 64, 65, 128, 129):
        v = ctx.correct(Bd[129 - R:].contiguous(), yd[129 - R:].clone()).cpu().numpy()
        err = np.linalg.norm(v - want[129 - R:]) / np.linalg.norm(want[129 - R:])
        assert err < 1e-6, (R, err)
        assert np.array_equal(v[-1], alone), R
