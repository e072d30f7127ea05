"""Statuses that kernels record: a call that synchronises reports them itself, a set-up neither
hides nor leaves one behind.  The expired waits are made by a wait limit of zero rounds
(ce_set_wait_limit), which ends a launch with CE_ERR_TIMEOUT and nothing else."""
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


def _sited(ce, n, prec, m=64):
    wl = workloads.workload("plain64").scaled(m=m, n=n)
    sites = workloads.make_sites(wl)
    z = torch.tensor(workloads.make_data(wl, sites), dtype=torch.float32, device="cuda")
    return ce.Context.from_workload(wl).krige_weights(sites, "local", np_=2, prec=prec), sites, z


def _expires(ce, call):
    with pytest.raises(ce.CEError) as e:
        call()
    assert e.value.status == ce.CE_ERR_TIMEOUT


@pytest.mark.parametrize("n,prec", [(200, "f16x3"), (1800, "fp32")])
def test_synchronous_calls_report_an_expired_wait(ce, n, prec):
    ctx, _, z = _sited(ce, n, prec)
    zh, out = z.cpu().pin_memory(), torch.empty((4, 64, 64), pin_memory=True)
    win = (8, 40, 8, 40)
    grad = ctx.condsim_grad(z, 4, 3, win)
    host = ctx.condsim_host(zh, 4, 3, out_host=out).clone()
    ctx.set_wait_limit(0)
    _expires(ce, lambda: ctx.condsim_grad(z, 4, 3, win))
    _expires(ce, lambda: ctx.condsim_host(zh, 4, 3, out_host=out))
    ctx.sync()   # each was reported once
    ctx.set_wait_limit(1 << 22)
    again = ctx.condsim_grad(z, 4, 3, win)
    assert torch.equal(again[0], grad[0]) and np.allclose(again[1], grad[1], rtol=1e-5) and np.isclose(again[3], grad[3], rtol=1e-6)
    assert torch.equal(ctx.condsim_host(zh, 4, 3, out_host=out), host)
    ctx.sync()


@pytest.mark.parametrize("n", [60, 300])
def test_standard_errors_report_an_expired_wait(ce, n):
    ctx, _, _ = _sited(ce, n, "fp32")
    exact, approx = ctx.se_map()
    ctx.set_wait_limit(0)
    _expires(ce, ctx.se_map)
    ctx.sync()
    ctx.set_wait_limit(1 << 22)
    again = ctx.se_map()
    assert torch.equal(again[0], exact) and torch.equal(again[1], approx)


@pytest.mark.parametrize("R", [1, 16, 130])
def test_expired_wait_in_the_digit_solve(ce, R):
    ctx, _, _ = _sited(ce, 1800, "fp32")
    E = torch.randn((R, 1800), generator=torch.Generator().manual_seed(R)).cuda()
    want = ctx.solve(E)
    ctx.set_wait_limit(0)
    ctx.solve(E)
    _expires(ce, ctx.sync)
    ctx.set_wait_limit(1 << 22)
    assert torch.equal(ctx.solve(E), want)
    ctx.sync()


@pytest.mark.parametrize("n", [60, 200, 700])
def test_expired_wait_in_the_set_up(ce, n):
    ctx, sites, z = _sited(ce, n, "fp32")
    want, logdet = ctx.condsim(z, 3, 7), ctx.info()["logdet"]
    ctx.set_wait_limit(0)
    _expires(ce, lambda: ctx.krige_weights(sites, "local", np_=2))
    ctx.set_wait_limit(1 << 22)
    ctx.sync()   # nothing left behind
    ctx.krige_weights(sites, "local", np_=2)
    assert ctx.info()["logdet"] == logdet and torch.equal(ctx.condsim(z, 3, 7), want)


def test_a_set_up_keeps_a_pending_status(ce):
    ctx, sites, z = _sited(ce, 200, "f16x3")
    ctx.set_wait_limit(0)
    ctx.condsim(z, 4, 3)
    torch.cuda.synchronize()
    ctx.set_wait_limit(1 << 22)
    ctx.krige_weights(sites, "local", np_=2, prec="f16x3")
    _expires(ce, ctx.sync)


def test_a_refused_set_up_leaves_no_status(ce):
    wl = workloads.workload("plain64").scaled(n=70, tau2=0.0)
    sites = workloads.make_sites(wl)
    sites[69] = sites[3]
    ctx = ce.Context.from_workload(wl)
    with pytest.raises(ce.CEError) as e:
        ctx.krige_weights(sites, "local", np_=2)
    assert e.value.status == ce.CE_ERR_NOT_SPD
    ctx.unconditional(2, 1)
    ctx.sync()
