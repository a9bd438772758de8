"""General elements: the off-diagonal product applies the dense inverse mass
matrix in one of three ways, chosen by precision, order and element count (the
separate kernels' line lies at 1064 elements for 64 modes); the sums are the
same, so the fused and the separate sweeps agree bit for bit on both sides."""
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,P,precision", [
    ((4, 3, 2), 1, "fp64"), ((4, 3, 2), 2, "fp64"), ((4, 3, 2), 2, "fp32"),
    ((4, 3, 2), 3, "fp32"), ((4, 3, 2), 3, "bf16"),
    ((8, 7, 19), 3, "fp32"), ((15, 71, 1), 3, "bf16"),     # 1064 and 1065 elements
    ((2, 1, 2), 4, "fp32"), ((2, 1, 2), 4, "bf16"),
])
def test_forms_of_the_inverse_mass_matrix_agree(shape, P, precision):
    import paper_2002_04222_gb300 as dgl
    c = w.wavy_box_case(shape, P=P)
    m = dgl.Mesh.from_case(c)
    u = m.project()
    g = torch.Generator(device="cuda").manual_seed(2)
    q = torch.randn(u.shape, dtype=torch.float64, device="cuda", generator=g)
    outs = [dgl.Precond(m).build(u, 0.0, 0.02, J=3, precision=precision, fused=f).apply(q)
            for f in (False, True)]
    assert torch.isfinite(outs[0]).all()
    assert torch.equal(*outs)
