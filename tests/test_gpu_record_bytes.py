"""The bytes of coefficient records that a simulation reports are those of the
records it keeps: one per column or per cell, FP32 records per cell short of
the values that the step forms from others, D3Q39's in groups of 32 cells."""
import pytest

from paper_2401_17183_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


@pytest.mark.parametrize("mesh,prec,per_record,group", [
    (lambda: W.channel_bump3d_mesh(5, 4, 11, stretch=0.5, bump=0.02), "F32", 320, 32),
    (lambda: W.channel_bump3d_mesh(5, 4, 11, stretch=0.5, bump=0.02), "F16", 4 * 136, 1),
    (lambda: W.channel_bump3d_mesh(5, 4, 11, stretch=0.5, bump=0.02), "F64", 8 * 136, 1),
    (lambda: W.periodic_sine_mesh(9, 0.02), "F32", 128, 32),
    (lambda: W.periodic_sine_mesh3d(5, 0.01, q=39), "F64", 8 * 193, 32)])
def test_record_bytes(V, mesh, prec, per_record, group):
    mesh = mesh()
    s = V.Sim(V.Mesh(mesh), W.params(0.8), *W.rest_fields(mesh), precision=getattr(V, "VLB_" + prec))
    lay = s.layout()
    assert not lay["plane"] and lay["records"] == W.ncell(mesh)
    assert lay["record_bytes"] == per_record * (-(-lay["records"] // group) * group)


def test_record_bytes_per_column(V):
    mesh = W.channel_mesh(5, 4, 11, stretch=0.5, bump=0.02)
    for prec, size in (("F32", 4), ("F64", 8), ("BF16", 4)):
        s = V.Sim(V.Mesh(mesh), W.params(0.8), *W.rest_fields(mesh), precision=getattr(V, "VLB_" + prec))
        lay = s.layout()
        assert lay["plane"] and lay["records"] == 20
        assert lay["record_bytes"] == size * lay["coef_per_cell"] * 20
