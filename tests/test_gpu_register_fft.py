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
