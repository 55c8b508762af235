"""D3Q39 simulations without their records (the form taken where device memory
does not hold them): against the oracle at the bounds of the form with records,
and on a device that is nearly full."""
import numpy as np
import pytest

from oracle import OracleSim
from oracle import lattice as olat
from paper_2401_17183_gb300 import workloads as W

from .helpers import oracle_state_in_lib_order, rel_err

pytestmark = pytest.mark.gpu

FORM = W.params(0.8, body_force=(1e-5, 3e-6, 2e-6))


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


def _compact(V, sim):
    assert V.load().vlb_internal_q39_compact(sim.h) == 0
    assert sim.layout()["coef_per_cell"] == 12


@pytest.mark.parametrize("L,amp,tau", [(3, 0.004, 0.8), (5, 0.01, 0.8), (7, 0.02, 1.7), (13, 0.02, 0.8)])
def test_without_records_against_oracle(V, L, amp, tau):
    mesh = W.periodic_sine_mesh3d(L, amp, q=39)
    prm = W.params(tau, body_force=(1e-5, 3e-6, 2e-6))
    rho, u = W.noise_fields(mesh, amp=0.02, seed=7, rho_amp=0.01)
    g = V.Sim(V.Mesh(mesh), prm, rho, u, precision=V.VLB_F64)
    _compact(V, g)
    o = OracleSim(mesh, prm)
    o.init(rho, u)
    co, _, _ = olat(39)
    cl, _ = V.lattice(39)
    done = 0
    for s in (1, 2, 3, 10):
        g.step(s - done)
        o.step(s - done)
        done = s
        assert rel_err(g.get_state(), oracle_state_in_lib_order(o.get_state(), co, cl)) < (1e-13 if s <= 3 else 1e-12), s
        gm, om = g.moments(), o.moments()
        su = np.abs(om["u"]).max()
        assert rel_err(gm["rho"], om["rho"], 1.0) < 1e-12
        assert rel_err(gm["u_tilde"], om["u_tilde"], su) < 1e-12
        assert abs(gm["mass"] - om["mass"]) <= 1e-13 * om["mass"]


def test_records_leave_room_for_the_fields_and_the_state(V):
    """Room for the records, but not for the staging of the state after them."""
    torch = pytest.importorskip("torch")
    mesh = W.periodic_sine_mesh3d(64, 0.01, q=39)
    rho, u = W.noise_fields(mesh, amp=0.02, seed=7, rho_amp=0.01)
    n = W.ncell(mesh)
    small = W.periodic_sine_mesh3d(8, 0.01, q=39)
    warm = V.Sim(V.Mesh(small), FORM, *W.noise_fields(small, amp=0.02, seed=7))
    for form in (None, _compact):     # (the kernels' own memory is there before the device is full)
        if form:
            form(V, warm)
        warm.step(2)
        warm.moments()
        warm.get_state()
    vm = V.Mesh(mesh)
    torch.cuda.empty_cache()
    # populations and records, and 40 MB more: the fields' staging (15 MB) fits, the state's (82 MB) does not
    room = (39 * 8 + 1544) * n + (40 << 20)
    fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    try:
        s = V.Sim(vm, FORM, rho, u)
        s.step(2)
        s.moments()
        N = s.get_state()
        s.set_state(N)
        form = s.layout()["coef_per_cell"]
        s.close()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert form == 12
    s = V.Sim(vm, FORM, rho, u)       # room again: with records
    assert s.layout()["coef_per_cell"] == 193
    s.step(2)
    assert rel_err(s.get_state(), N) < 1e-13
