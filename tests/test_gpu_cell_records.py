"""FP32 records per cell (the entries the step forms again in registers) and
tiles over the linear cell index: sizes around whole groups of 32 and 128
cells and around the narrow-tile limit, 16-bit storage, moving walls, against
the FP64 plane-record run of the same mesh."""
import numpy as np
import pytest

from paper_2401_17183_gb300 import workloads as W

from .helpers import rel_err

pytestmark = pytest.mark.gpu

# the FP32 bar of the parity tests (2e-5 of max |u|); 16-bit storage against the
# uniform reference stays below 1e-2 (FP16) over these few steps
SIZES = [(4, 3, 2), (5, 4, 3), (4, 4, 8), (7, 6, 37), (6, 5, 129), (16, 19, 64), (16, 19, 65), (32, 20, 96)]


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


def _compare(V, mesh, prm, prec, tol, steps=21):
    rho, u = W.noise_fields(mesh, amp=0.01, seed=4)
    vm = V.Mesh(mesh)
    ref = V.Sim(vm, prm, rho, u, precision=V.VLB_F64)
    g = V.Sim(vm, prm, rho, u, precision=prec, coef_mode=V.VLB_COEF_FULL)
    for n in (1, 2, steps - 3):
        ref.step(n)
        g.step(n)
        a, b = g.moments(), ref.moments()
        s = np.abs(b["u_tilde"]).max()
        assert rel_err(a["u_tilde"], b["u_tilde"], s) < tol, n
        assert rel_err(a["rho"], b["rho"], 1.0) < tol, n


@pytest.mark.parametrize("n", SIZES)
def test_sizes_f32(V, n):
    _compare(V, W.channel_mesh(*n, stretch=0.5, bump=0.02), W.params(0.8, body_force=(1e-5, 0, 0)), V.VLB_F32, 2e-5)


@pytest.mark.parametrize("n", [(7, 6, 37), (6, 5, 40), (16, 19, 65), (32, 20, 96)])
def test_sizes_f16(V, n):
    _compare(V, W.channel_mesh(*n, stretch=0.5, bump=0.02), W.params(0.8, body_force=(1e-5, 0, 0)), V.VLB_F16, 1e-2)


@pytest.mark.parametrize("n", [(3, 5), (8, 16), (33, 31), (150, 140)])
@pytest.mark.parametrize("tau", [0.51, 0.8, 30.0])
def test_sizes_2d(V, n, tau):
    _compare(V, W.channel2d_mesh(*n, stretch=0.5, bump=0.02), W.params(tau, body_force=(0, 1e-5, 0)), V.VLB_F32, 2e-5)


@pytest.mark.parametrize("n", [(6, 5, 16), (9, 21, 107)])
def test_moving_walls(V, n):
    wu = np.zeros((3, 2, 3))
    wu[1, 0, 0], wu[1, 1, 2] = 0.02, -0.01
    _compare(V, W.channel_mesh(*n, stretch=0.5, bump=0.02), W.params(0.8, wall_u=wu), V.VLB_F32, 2e-5)


def test_batch_of_ragged_members_is_bitwise(V):
    """Linear tiles cut a batch's members anywhere in a row: the populations
    are those of the members stepped alone."""
    def make():
        out = []
        for k, n in enumerate([(3, 5), (17, 40), (33, 31), (64, 129)]):
            mesh = W.channel2d_mesh(*n, stretch=0.5, bump=0.03)
            rho, u = W.noise_fields(mesh, amp=0.01, seed=k)
            out.append(V.Sim(V.Mesh(mesh), W.params(0.8, body_force=(0, 1e-5, 0)), rho, u, precision=V.VLB_F32))
        return out
    alone, members = make(), make()
    b = V.Batch(members)
    for shape in range(4):
        b.set_shape(shape)
        b.step(35)
        for s in alone:
            s.step(35)
        for s, t in zip(alone, members):
            assert np.array_equal(s.get_state(), t.get_state()), shape
