"""Residual kernels whose contractions run in 64-bit fixed point: scale
invariance, degenerate inputs, and the axis-aligned kernels against the
general-geometry ones on the same elements.

Bounds: a contraction keeps 2^-53 of its largest value or better, so results
of two forms of the same residual differ by at most a multiple of the rounding
floor s, the oracle's relative change under a one-ulp relative perturbation of
u: 16 s for R, 64 s for the weak form L = M R (the parity tests' bounds; L
leaves out the rounding of the numerically inverted mass matrices of the
oracle and of the general kernels).  Scaling by an even power of two commutes
with every operation of the Euler residual, square roots included."""
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


def state(dg, seed=3, amp=0.02):
    u = dg.project_exact()
    return u + amp * w.random_direction(u, seed)


def floor(dg, u, R):
    s = np.sign(np.random.default_rng(0).standard_normal(u.shape))
    return np.linalg.norm(dg.residual(u * (1 + 2.0 ** -52 * s)) - R) / np.linalg.norm(R)


def weak(dg, R):
    return np.einsum("emn,evn->evm", np.einsum("qm,eq,qn->emn", dg.B, dg.wJ, dg.B), R)


def weak_floor(dg, u, L):
    s = np.sign(np.random.default_rng(0).standard_normal(u.shape))
    return np.linalg.norm(dg.rhs(u * (1 + 2.0 ** -52 * s)) - L) / np.linalg.norm(L)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def quadratic(mesh):
    """The same straight elements with (3)^dim geometry nodes: the mesh takes
    the general-geometry kernels."""
    d = mesh.dim
    lo, hi = mesh.nodes[:, 0], mesh.nodes[:, -1]
    a = np.stack(np.unravel_index(np.arange(3 ** d), (3,) * d)[::-1], -1) / 2.0
    nodes = lo[:, None] + (hi - lo)[:, None] * a[None]
    return w.Mesh(d, 2, nodes, mesh.faces, mesh.shape, mesh.periodic)


CASES = {
    "vortex_P2": lambda: w.vortex_case(n=5, P=2),
    "vortex_euler_P2": lambda: w.vortex_case(n=5, P=2, viscous=False),
    "channel_P3": lambda: w.poiseuille_case(3, nx=5, ny=4),
    "swbli_P3": lambda: w.swbli_case(nx=13, ny=7),
    "swbli_ducros_P3": lambda: w.swbli_case(nx=13, ny=7, av=2),
    "box_P1": lambda: w.small_tgv_case((3, 1, 2), P=1, stretch=True),
    "box_P2": lambda: w.small_tgv_case((3, 2, 2), P=2, stretch=True),
    "box_P3": lambda: w.small_tgv_case((2, 1, 3), P=3, stretch=True),
    "box_P4": lambda: w.small_tgv_case((1, 2, 2), P=4),
}


@pytest.mark.parametrize("riemann,mu_law", [(0, 0), (1, 1), (3, 0)])
@pytest.mark.parametrize("name", sorted(CASES))
def test_axis_aligned_and_general_kernels_agree(dgl, name, riemann, mu_law):
    c = CASES[name]()
    c.phys.riemann, c.phys.mu_law = riemann, mu_law
    dg = DG(c.mesh, c.P, c.Q, c.phys)
    u = state(dg)
    L = dg.rhs(u)
    tol = max(1e-12, 64 * weak_floor(dg, u, L))
    la = weak(dg, dgl.Mesh(c.mesh, c.P, c.Q, c.phys).residual(dev(u)).cpu().numpy())
    lg = weak(dg, dgl.Mesh(quadratic(c.mesh), c.P, c.Q, c.phys).residual(dev(u)).cpu().numpy())
    # (with the sensor on, the oracle's floor leaves out its own logarithm; the
    # general kernels take M^-1 as inverted in FP64, off by cond(M) 2^-53)
    inv = np.linalg.cond(np.einsum("qm,eq,qn->emn", dg.B, dg.wJ, dg.B)).max() * 2.0 ** -53
    if not c.phys.av:
        assert rel(la, L) < tol and rel(lg, L) < tol + inv
    assert rel(la, lg) < 2 * tol + inv


@pytest.mark.parametrize("general", [False, True])
def test_power_of_two_scaling_is_exact(dgl, general):
    """Euler: R(2^k u) = 2^k R(u) (the flux is homogeneous of degree one), bit
    for bit, over exponents far from one."""
    c = w.small_tgv_case((2, 3, 2), P=2)
    c.phys.viscous = False
    mesh = quadratic(c.mesh) if general else c.mesh
    u = state(DG(c.mesh, c.P, c.Q, c.phys))
    m = dgl.Mesh(mesh, c.P, c.Q, c.phys)
    r = m.residual(dev(u))
    for k in (-300, -40, 2, 50, 300):
        assert torch.equal(m.residual(dev(u * 2.0 ** k)), r * 2.0 ** k), k


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("general", [False, True])
def test_non_finite_input_reaches_the_element_and_its_neighbours_only(dgl, general, bad):
    c = w.small_tgv_case((5, 4, 4), P=2)
    mesh = quadratic(c.mesh) if general else c.mesh
    u = state(DG(c.mesh, c.P, c.Q, c.phys))
    m = dgl.Mesh(mesh, c.P, c.Q, c.phys)
    r0 = m.residual(dev(u)).cpu().numpy()
    e = 27
    u[e, 0, 5] = bad
    r = m.residual(dev(u)).cpu().numpy()
    near = {e}
    for eL, _, eR, _, _, _ in c.mesh.faces:
        if e in (eL, eR):
            near |= {int(eL), int(eR)}
    touched = {i for i in range(u.shape[0]) if not np.array_equal(r[i], r0[i])}
    assert touched <= near
    for i in near:
        assert not np.isfinite(r[i]).all()
    assert not np.isfinite(r[e]).any()


@pytest.mark.parametrize("general", [False, True])
def test_zero_components_stay_zero_and_tiny_ones_keep_their_scale(dgl, general):
    """A fluid at rest: no momentum, uniform pressure, energy a power of two (so
    that p = (gamma - 1) E is exact and p_R - p_L vanishes).  The mass residual
    is exactly zero; a cross flow of 1e-30 gives one of its own size, not of the
    pressure's."""
    c = w.small_tgv_case((3, 2, 2), P=2)
    mesh = quadratic(c.mesh) if general else c.mesh
    dg = DG(c.mesh, c.P, c.Q, c.phys)
    one = np.round(dg.one_coeffs(), 10)
    u = np.zeros((dg.E, 5, dg.nm))
    u[:, 0] = one
    u[:, 4] = 128.0 * one
    m = dgl.Mesh(mesh, c.P, c.Q, c.phys)
    r = m.residual(dev(u)).cpu().numpy()
    assert np.abs(r[:, 0]).max() == 0.0 and np.isfinite(r).all()
    u[:, 1] = 1e-30 * np.random.default_rng(1).standard_normal((dg.E, dg.nm))
    r = m.residual(dev(u)).cpu().numpy()
    # (the oracle's own pressure jumps round at 1e-15: only the scale is compared;
    # derivatives and M^-1 give factors of 1 to 1e3)
    assert 1e-31 < np.abs(r[:, 0]).max() < 1e-26


@pytest.mark.parametrize("beta_s", [0.0, -0.5, 2.0])
@pytest.mark.parametrize("general", [False, True])
def test_symmetric_flux_factor(dgl, general, beta_s):
    c = w.small_tgv_case((3, 2, 2), P=2, stretch=True)
    c.phys.beta_s = beta_s
    mesh = quadratic(c.mesh) if general else c.mesh
    dg = DG(c.mesh, c.P, c.Q, c.phys)
    u = state(dg)
    R = dg.residual(u)
    r = dgl.Mesh(mesh, c.P, c.Q, c.phys).residual(dev(u)).cpu().numpy()
    assert rel(r, R) < max(1e-12, 16 * floor(dg, u, R))


@pytest.mark.parametrize("name", ["vortex_P2", "box_P3"])
@pytest.mark.parametrize("general", [False, True])
def test_launch_shapes_give_the_same_bits(dgl, name, general):
    """Every candidate shape, odd groupings and a ragged last block included."""
    import ctypes
    from paper_2002_04222_gb300 import _lib
    c = CASES[name]()
    mesh = quadratic(c.mesh) if general else c.mesh
    m = dgl.Mesh(mesh, c.P, c.Q, c.phys)
    u = dev(state(DG(c.mesh, c.P, c.Q, c.phys)))
    r = m.residual(u)
    tried = 0
    for ve in (1, 2, 3, 4, 8, 16, 32):
        for vt, lt in ((64, 256), (96, 96), (128, 128), (160, 64), (224, 192), (256, 224)):
            t = _lib.TuneResult(ve, vt, ve, lt, 0, 0, 0, 0)
            if dgl.lib().dg_set_tune(m.handle, ctypes.byref(t)) == 0:
                tried += 1
                assert torch.equal(m.residual(u), r), (ve, vt, lt)
    assert tried > 4


@pytest.mark.parametrize("ratio", [1e4, 1e8])
@pytest.mark.parametrize("shape", [(4, 2), (4, 1, 2)])
@pytest.mark.parametrize("general", [False, True])
def test_a_side_keeps_its_digits_beside_a_much_larger_neighbour(dgl, general, shape, ratio):
    """Supersonic flow from light elements (i = 2, 3) into ones `ratio` times
    denser (i = 0, 1): the upwinded flux of the face between them is the light
    side's alone, so the weak form on the light elements beside it is as exact
    as without the jump.  Bound: 64 times those elements' own rounding floor
    (the parity tests'), for the general kernels plus cond(M) 2^-53."""
    P, d = 2, len(shape)
    c = (w.vortex_case(n=4, P=P) if d == 2 else w.small_tgv_case((4, 1, 2), P=P))
    mesh = w.box_mesh([np.linspace(0.0, 1.0, n + 1) for n in shape], (True,) * d)
    ph = c.phys
    ph.viscous, ph.riemann, ph.Ma = False, 1, 1.0
    dg = DG(mesh, P, c.Q, ph)
    rho, vel = 1.0, np.array([-3.0, 0.1, 0.05][:d])
    prim = np.concatenate([[rho], rho * vel, [rho / ph.gamma / (ph.gamma - 1.0) + 0.5 * rho * vel @ vel]])
    u = prim[None, :, None] * (dg.one_coeffs()[None, None, :]
                               + 0.02 * np.random.default_rng(2).standard_normal((dg.E, d + 2, dg.nm)))
    i = np.arange(dg.E) % shape[0]
    u[i < 2] *= ratio
    sel = i == 2
    L = dg.rhs(u)
    s = np.sign(np.random.default_rng(0).standard_normal(u.shape))
    tol = 64 * np.linalg.norm((dg.rhs(u * (1 + 2.0 ** -52 * s)) - L)[sel]) / np.linalg.norm(L[sel])
    if general:
        tol += np.linalg.cond(np.einsum("qm,eq,qn->emn", dg.B, dg.wJ, dg.B)).max() * 2.0 ** -53
    got = weak(dg, dgl.Mesh(quadratic(mesh) if general else mesh, P, c.Q, ph).residual(dev(u)).cpu().numpy())
    assert tol < 3e-10
    assert rel(got[sel], L[sel]) < tol
