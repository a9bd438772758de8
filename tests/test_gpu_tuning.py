"""The launch shapes the tuning admits, and which stored entry a mesh takes."""
import ctypes

import pytest

import workloads as w

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
DG_OK, DG_ERR_ARG = 0, -1


@pytest.fixture(scope="module")
def dgl():
    import paper_2002_04222_gb300 as d
    return d


@pytest.mark.parametrize("make,accepted,refused", [
    # 23 KB a face, three an element: up to three elements' faces a CTA; a volume
    # CTA holds two elements of 92 KB
    (lambda: w.tgv_case(n=2, P=4, Q=8), [(2, 3), (1, 2)], [(3, 1), (1, 4)]),
    # general elements: 32 KB a face
    (lambda: w.wavy_box_case((2, 2, 2), P=4, Q=8), [(2, 2)], [(3, 1), (1, 3)]),
    (lambda: w.vortex_case(n=6, P=6), [(32, 16)], [(32, 32)]),
])
def test_shapes_that_fit_the_launched_kernels_are_candidates(dgl, make, accepted, refused):
    from paper_2002_04222_gb300 import _lib
    c = make()
    m = dgl.Mesh.from_case(c)
    u = m.project()
    r = m.residual(u)

    def tune(ve, le):
        t = _lib.TuneResult(ve, 256, le, 256, 0, 0, 0, 0)
        return dgl.lib().dg_set_tune(m.handle, ctypes.byref(t))

    for ve, le in accepted:
        assert tune(ve, le) == DG_OK, (ve, le)
        assert torch.equal(m.residual(u), r), (ve, le)
    for ve, le in refused:
        assert tune(ve, le) == DG_ERR_ARG, (ve, le)


@pytest.mark.parametrize("make,general", [
    (lambda: w.small_tgv_case((2, 2, 2), P=2), False),
    (lambda: w.rotated_box_case((2, 2, 2), P=2), True),              # straight, not boxes
    (lambda: w.rotated_box_case((2, 2, 2), P=2, order=2), True),
    (lambda: w.wavy_box_case((2, 2, 2), P=2), True),
])
def test_a_mesh_takes_the_entry_of_its_own_kernels(dgl, tmp_path, make, general):
    import json
    c = make()
    m = dgl.Mesh.from_case(c)
    assert dgl.lib().dg_mesh_general(m.handle) == int(general)
    assert dgl.lib().dg_mesh_general(None) == DG_ERR_ARG
    entry = dict(vol_threads=128, lift_threads=128)
    table = tmp_path / "t.json"
    table.write_text(json.dumps({"3d_P2_Q5": dict(entry, vol_epb=1, lift_epb=1),
                                 "3d_P2_Q5_general": dict(entry, vol_epb=2, lift_epb=2)}))
    assert dgl.apply_tuning(m, str(table))["vol_epb"] == 1 + general
