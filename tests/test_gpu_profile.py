"""Per-kernel times: every family's time is that of its own kernels."""
import pytest

import workloads as w

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


@pytest.mark.parametrize("make", [lambda: w.small_tgv_case((3, 2, 2), P=2),
                                  lambda: w.wavy_box_case((3, 2, 2), P=2)])
def test_families_hold_their_own_kernels(make):
    import paper_2002_04222_gb300 as dgl
    m = dgl.Mesh.from_case(make())
    u = m.project()
    pc = dgl.Precond(m)
    dgl.profile_enable(True)
    try:
        dgl.profile_read()
        for _ in range(3):
            r = m.residual(u)
        res = dgl.profile_read()
        pc.build(u, 0.0, 0.02)
        build = dgl.profile_read()
    finally:
        dgl.profile_enable(False)
    assert r.shape == u.shape
    assert {k: v[0] for k, v in res.items()} == {"dg_vol": 3, "dg_face": 3, "dg_lift": 3}
    assert res["dg_lift"][1] == 0.0 and res["dg_vol"][1] > 0.0 and res["dg_face"][1] > 0.0
    # the build takes traces, and evaluates no residual
    assert build["dg_trace"][0] == 1 and not {"dg_vol", "dg_face", "dg_lift"} & set(build)
    assert not set(dgl.profile_read())
