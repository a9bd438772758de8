"""The one-launch application's bounded waits running out (a limit of 0 polls):
the solve returns an error, the next one applies sweep by sweep, a rebuild takes
the one launch up again.  Nothing hangs: with a limit of 0 no block waits."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DG_ERR_ARG, DG_ERR_TIMEOUT = -1, -7


@pytest.fixture(scope="module")
def dgl():
    import paper_2002_04222_gb300 as d
    return d


def launches(dgl, f):
    n0 = dgl.kernel_launches()
    out = f()
    return out, dgl.kernel_launches() - n0


@pytest.mark.parametrize("solver", ["gmres", "gmres_graphs", "gmres_noalloc"])
def test_a_wait_that_runs_out_is_an_error_and_a_rebuild_recovers(dgl, solver):
    c = w.vortex_case(n=6, P=2)
    m = dgl.Mesh.from_case(c)
    u = m.project()
    r = m.residual(u)
    b = torch.from_numpy(w.random_direction(u.cpu().numpy(), 3)).cuda()
    p = dgl.Precond(m).build(u, 0.0, 0.01)
    kw = dict(t=0.0, dt_a=0.01, precond=p, restart=8, max_cycles=2, rtol=1e-6)

    def solve():
        if solver == "gmres_noalloc":
            return m.gmres_noalloc(u, r, b, m.empty(), **kw)[0]
        return m.gmres(u, r, b, graphs=solver == "gmres_graphs", **kw)[0]

    x0, n0 = launches(dgl, solve)
    assert torch.isfinite(x0).all()
    # (a captured application is a chain of launches: no wait can run out there)
    one_launch = solver != "gmres_graphs"
    limit = dgl.lib().dg_precond_wait_limit
    assert limit(p.handle, -1) == DG_ERR_ARG and limit(None, 0) == DG_ERR_ARG
    former = limit(p.handle, 0)
    assert former > 1 << 20
    try:
        solve()
        failed = False
    except dgl._lib.DGError as e:
        assert e.code == DG_ERR_TIMEOUT
        failed = True
    assert failed or not one_launch
    x1, n1 = launches(dgl, solve)          # sweep by sweep: the same bits
    assert torch.equal(x1, x0) and (n1 > n0 or not one_launch)
    p.build(u, 0.0, 0.01)                  # up again, and out again
    if one_launch:
        with pytest.raises(dgl._lib.DGError):
            solve()
    assert limit(p.handle, former) == 0
    p.build(u, 0.0, 0.01)
    x2, n2 = launches(dgl, solve)
    assert torch.equal(x2, x0) and n2 == n0


def test_a_step_reports_the_wait_and_the_next_one_takes_the_sweeps(dgl):
    c = w.vortex_case(n=6, P=2)
    m = dgl.Mesh.from_case(c)
    u0 = m.project()
    p = dgl.Precond(m)
    ref = u0.clone()
    m.sdirk_step(ref, 0.0, 0.02, precond=p, restart=20)
    dgl.lib().dg_precond_wait_limit(p.handle, 0)
    u = u0.clone()
    with pytest.raises(dgl._lib.DGError) as e:
        m.sdirk_step(u, 0.0, 0.02, precond=p, restart=20)
    assert e.value.code == DG_ERR_TIMEOUT
    u = u0.clone()
    m.sdirk_step(u, 0.0, 0.02, precond=p, restart=20)
    assert torch.equal(u, ref)
