"""A set-up of many sites with little device memory left: it fits wherever the FP64 matrix and
the FP32 pair of its inverse do, with the digits where they fit once the matrix is gone and with
the FP32 products otherwise.  6000 sites: matrix and pair 276 MiB each, digits 345 MiB, 15 MiB of
other arrays; the rest of the device is held by one tensor."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MIB = 1 << 20


@pytest.fixture(scope="module")
def ce():
    from paper_2109_11044_gb300.build import build
    build()
    import paper_2109_11044_gb300 as mod
    mod.load_library()
    return mod


def test_set_up_with_little_memory(ce):
    n = 6000
    wl = workloads.workload("plain64").scaled(n=n)
    sites = workloads.make_sites(wl)
    E = torch.randn((2, n), generator=torch.Generator().manual_seed(3)).cuda()
    ctx = ce.Context.from_workload(wl).krige_weights(sites, "local", np_=2)
    want, held = ctx.solve(E), ctx.info()["device_bytes"]
    ctx.close()
    small = ce.Context.from_workload(wl).krige_weights(sites[:1500], "local", np_=2)
    small.solve(E[:, :1500].contiguous())   # the FP32 products' kernels are loaded
    small.close()
    for left, digits in ((780, True), (595, False)):
        ctx = ce.Context.from_workload(wl)
        torch.cuda.empty_cache()
        filler = torch.empty(torch.cuda.mem_get_info()[0] - left * MIB, dtype=torch.uint8, device="cuda")
        try:
            ctx.krige_weights(sites, "local", np_=2)
            got = ctx.solve(E)
            bytes_now = ctx.info()["device_bytes"]
        finally:
            del filler
            torch.cuda.empty_cache()
        assert (held - bytes_now < 100 * MIB) == digits
        if digits:
            assert torch.equal(got, want)
        else:   # both within 1e-7 of the FP64 solve
            assert np.linalg.norm((got - want).cpu()) <= 2e-7 * np.linalg.norm(want.cpu())
        ctx.close()
