"""The solvers' one-launch forms on small meshes: the cooperative BRJ
application (every element's block resident at once) and the cluster kernels of
the norms and the Gram-Schmidt tail (up to 16,384 unknowns).

Per-kernel profiling keeps the sweeps of an application as separate launches,
so a solve under it is the reference of the same solve without: the same
arithmetic, hence the same bits.  The solution's true residual is held to the
stopping tolerance: GMRES stops on its estimate, which differs from the true
residual by the finite-difference product's error (1e-6 of ||A x||)."""
import numpy as np
import pytest

import workloads as w
from oracle.dg import DG

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def dgl():
    import paper_2002_04222_gb300 as d
    return d


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


MESHES = {"vortex_P2": lambda: w.vortex_case(n=5, P=2),
          "box_P2": lambda: w.small_tgv_case((3, 2, 4), P=2, stretch=True),
          "cylinder_P2": lambda: w.small_cylinder_case(2, 6, 2, P=2, wall_layer=0.1)}


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("J,omega", [(1, 1.0), (2, 0.8), (3, 1.0), (7, 0.9)])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_one_launch_apply_has_the_sweeps_bits(dgl, name, J, omega, precision):
    c = MESHES[name]()
    dg = DG(c.mesh, c.P, c.Q, c.phys)
    u = dg.project_exact()
    ud = dev(u + 0.01 * w.random_direction(u, 3))
    b = dev(w.random_direction(u, 4))
    m = dgl.Mesh.from_case(c)
    r = m.residual(ud)
    for fused in (False, True):
        pc = dgl.Precond(m).build(ud, 0.0, 0.01, J=J, omega=omega, precision=precision, fused=fused)
        kw = dict(t=0.0, dt_a=0.01, precond=pc, restart=6, max_cycles=2, rtol=1e-6)
        n0 = dgl.kernel_launches()
        x, st = m.gmres(ud, r, b, **kw)
        n = dgl.kernel_launches() - n0
        dgl.profile_enable(True)
        try:
            n0 = dgl.kernel_launches()
            x_ref, st_ref = m.gmres(ud, r, b, **kw)
            n_ref = dgl.kernel_launches() - n0
            dgl.profile_read()
        finally:
            dgl.profile_enable(False)
        assert torch.isfinite(x).all() and st == st_ref
        assert torch.equal(x, x_ref)
        if J > 1:
            assert n < n_ref


@pytest.mark.parametrize("nx,ny", [(1, 2), (16, 64), (27, 38), (41, 50)])
def test_solves_on_both_sides_of_the_cluster_limit(dgl, nx, ny):
    """16 unknowns an element: 32, 16,384 (the limit), 16,416 and 32,800."""
    c = w.poiseuille_case(1, nx=nx, ny=ny)
    m = dgl.Mesh.from_case(c)
    u = m.project()
    g = torch.Generator(device="cuda").manual_seed(1)
    b = torch.randn(u.shape, dtype=torch.float64, device="cuda", generator=g)
    r = m.residual(u)
    pc = dgl.Precond(m).build(u, 0.0, 0.005)
    x, st = m.gmres(u, r, b, 0.0, 0.005, precond=pc, restart=20, max_cycles=5, rtol=1e-4)
    assert st["converged"], st
    ax = m.jvp(u, r, x, 0.0, 1.0, -0.005)
    err = torch.linalg.norm(b - ax).item()
    bound = 1e-4 * torch.linalg.norm(b).item() + 1e-6 * torch.linalg.norm(ax).item()
    assert err < bound, (err, bound)


@pytest.mark.parametrize("nx,ny", [(16, 64), (27, 38)])
def test_a_full_basis_on_both_sides_of_the_cluster_limit(dgl, nx, ny):
    """16,384 unknowns and 16,416 with a basis of 64 vectors, none converged
    before it is full: the residual that the Hessenberg matrix tells (orthonormal
    vectors) is the true one, to the finite-difference product's 1e-6."""
    c = w.poiseuille_case(1, nx=nx, ny=ny)
    m = dgl.Mesh.from_case(c)
    u = m.project()
    g = torch.Generator(device="cuda").manual_seed(1)
    b = torch.randn(u.shape, dtype=torch.float64, device="cuda", generator=g)
    r = m.residual(u)
    dta = 0.05
    x, st = m.gmres(u, r, b, 0.0, dta, restart=64, max_cycles=1, rtol=1e-14)
    assert st["iters"] == 64 and 0.0 < st["res"] < st["res0"]
    ax = m.jvp(u, r, x, 0.0, 1.0, -dta)
    err = abs(torch.linalg.norm(b - ax).item() - st["res"])
    assert err < 1e-6 * torch.linalg.norm(ax).item() + 1e-10 * st["res0"], (err, st)
