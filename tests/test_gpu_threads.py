"""One context per host thread: set-ups, solves, standard errors and gradients of different
sizes run side by side in one process (a kernel's shared-memory limit belongs to the
process), with the results that they have alone."""
import threading
import time

import numpy as np
import pytest

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


def _side_by_side(jobs, seconds=3.0):
    """Every job (a callable that returns an array) in a thread of its own, over and over."""
    errors, stop = [], time.monotonic() + seconds

    def loop(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                want = None
                while time.monotonic() < stop and not errors:
                    got = job()
                    want = got if want is None else want
                    assert np.array_equal(got, want)
        except BaseException as e:   # noqa: BLE001 (reported by the caller)
            errors.append(repr(e))

    threads = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_setups_of_different_sizes(ce):
    def job(m, n):
        wl = workloads.workload("plain64").scaled(m=m, n=n)
        sites = workloads.make_sites(wl)

        def run():
            ctx = ce.Context.from_workload(wl)
            ctx.krige_weights(sites, "local", np_=2)
            out = np.array([ctx.info()["logdet"]])
            ctx.close()
            return out
        return run

    _side_by_side([job(64, 20), job(700, 2500), job(33, 300)])


def test_solves_of_different_sizes(ce):
    def job(n, R):
        wl = workloads.workload("plain64").scaled(n=n)
        ctx = ce.Context.from_workload(wl).krige_weights(workloads.make_sites(wl), "local", np_=2)
        E = torch.randn((R, n), generator=torch.Generator().manual_seed(n)).cuda()
        torch.cuda.synchronize()
        return lambda: ctx.solve(E).cpu().numpy()

    _side_by_side([job(1800, 1), job(2000, 128), job(1900, 40)])


@pytest.mark.parametrize("prec", ["fp32", "f16x3"])
def test_draws_and_gradients_of_different_sizes(ce, prec):
    def job(n, R, grad):
        wl = workloads.workload("plain64").scaled(n=n)
        sites = workloads.make_sites(wl)
        ctx = ce.Context.from_workload(wl).krige_weights(sites, "local", np_=2, prec=prec)
        z = torch.tensor(workloads.make_data(wl, sites), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        if not grad:
            return lambda: ctx.condsim(z, R, 5).cpu().numpy()
        # the draws of the gradient call: its sums are joined in no fixed order
        return lambda: ctx.condsim_grad(z, R, 5, (8, 40, 8, 40))[0].cpu().numpy()

    _side_by_side([job(150, 3, False), job(150, 128, False), job(90, 2, True), job(90, 128, True)])
