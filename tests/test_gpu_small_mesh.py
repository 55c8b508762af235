"""Many steps of a small mesh in one launch against the same steps launched one
by one: both parities at the start, sizes around whole blocks, every record
kind, walls at rest and moving. Both run the same arithmetic per cell; a
compiler may contract a product and a sum differently in the two kernels, so
the states agree to a few units of the last place of the largest population
per step, far below any addressing mistake."""
import numpy as np
import pytest

from paper_2401_17183_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "row_of_one_block": lambda: W.channel2d_mesh(2, 64, stretch=0.5),
    "box_33": lambda: W.periodic_sine_mesh(33, 0.02),
    "channel2d_plane": lambda: W.channel2d_mesh(31, 40, stretch=0.5),
    "channel2d_cells": lambda: W.channel2d_mesh(32, 64, stretch=0.5, bump=0.1),
    "channel_short_rows": lambda: W.channel_mesh(9, 8, 3, stretch=0.5, bump=0.02),
    "channel_plane": lambda: W.channel_mesh(16, 9, 50, stretch=0.5, bump=0.02),
    "channel_cells": lambda: W.channel_bump3d_mesh(16, 12, 17, stretch=0.5, bump=0.02),
    "limit": lambda: W.channel2d_mesh(150, 256, stretch=0.5, bump=0.05),
}


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


@pytest.mark.parametrize("name", sorted(MESHES))
@pytest.mark.parametrize("prec,ulp", [("F32", 2.0 ** -24), ("F64", 2.0 ** -53)])
def test_multi_step_launch_matches_single_steps(V, name, prec, ulp):
    mesh = MESHES[name]()
    prm = W.params(0.7, body_force=(1e-5, 2e-6, 0))
    rho, u = W.noise_fields(mesh, amp=0.01, seed=4)
    vm = V.Mesh(mesh)
    a, b = (V.Sim(vm, prm, rho, u, precision=getattr(V, "VLB_" + prec)) for _ in range(2))
    done = 0
    for n in (2, 1, 3, 10):      # the third call starts on odd parity
        a.step(n)
        for _ in range(n):
            b.step(1)
        done += n
        A, B = a.get_state(), b.get_state()
        assert np.abs(A - B).max() <= 8 * done * ulp * np.abs(B).max(), n
        assert a.time() == b.time() == done
    a.sync()


@pytest.mark.parametrize("prec,ulp", [("F32", 2.0 ** -24), ("F64", 2.0 ** -53)])
@pytest.mark.parametrize("bump", [0.0, 0.05])
def test_multi_step_moving_walls(V, prec, ulp, bump):
    mesh = W.channel2d_mesh(20, 36, stretch=0.5, bump=bump)
    wu = np.zeros((3, 2, 3))
    wu[0, 0, 1], wu[0, 1, 1] = 0.02, -0.01
    rho, u = W.noise_fields(mesh, amp=0.01, seed=4)
    vm = V.Mesh(mesh)
    a, b = (V.Sim(vm, W.params(0.8, wall_u=wu), rho, u, precision=getattr(V, "VLB_" + prec)) for _ in range(2))
    a.step(25)
    for _ in range(25):
        b.step(1)
    A, B = a.get_state(), b.get_state()
    assert np.abs(A - B).max() <= 8 * 25 * ulp * np.abs(B).max()


def test_multi_step_error_is_reported(V):
    """A cell that does not converge raises the sticky error from the multi-step launch."""
    mesh = W.periodic_sine_mesh(16, 0.02)
    rho, u = W.taylor_green_fields(mesh, L=16)
    s = V.Sim(V.Mesh(mesh), W.params(0.8, max_iter=1), rho, u)
    s.step(4)
    with pytest.raises(V.VlbError) as e:
        s.sync()
    assert e.value.code == "ENOCONV"
