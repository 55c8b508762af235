"""The polynomial force map of the D3Q39 step at sizes where its records and
addressing can go wrong: the shortest axes (links of length 3 wrap onto their
own cell), cell counts that are not whole groups of 32 or 128."""
import numpy as np
import pytest

from oracle import OracleSim
from oracle import lattice as olat
from paper_2401_17183_gb300 import workloads as W

from .helpers import oracle_state_in_lib_order, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


@pytest.mark.parametrize("L,amp,tau", [(3, 0.004, 0.8), (4, 0.01, 0.6), (5, 0.01, 0.8), (7, 0.02, 1.7), (13, 0.02, 0.8)])
def test_d3q39_sizes_against_oracle(V, L, amp, tau):
    mesh = W.periodic_sine_mesh3d(L, amp, q=39)
    prm = W.params(tau, body_force=(1e-5, 3e-6, 2e-6))
    rho, u = W.noise_fields(mesh, amp=0.02, seed=7, rho_amp=0.01)
    g = V.Sim(V.Mesh(mesh), prm, rho, u, precision=V.VLB_F64)
    o = OracleSim(mesh, prm)
    o.init(rho, u)
    co, _, _ = olat(39)
    cl, _ = V.lattice(39)
    done = 0
    for s in (1, 2, 3, 10):
        g.step(s - done)
        o.step(s - done)
        done = s
        # the bounds of the D3Q39 parity test
        assert rel_err(g.get_state(), oracle_state_in_lib_order(o.get_state(), co, cl)) < (1e-13 if s <= 3 else 1e-12), s
        gm, om = g.moments(), o.moments()   # both parities
        su = np.abs(om["u"]).max()
        assert rel_err(gm["rho"], om["rho"], 1.0) < 1e-12
        assert rel_err(gm["u_tilde"], om["u_tilde"], su) < 1e-12
        assert abs(gm["mass"] - om["mass"]) <= 1e-13 * om["mass"]
        assert np.abs(gm["M"] - om["M"]).max() <= 1e-12 * np.abs(om["M"]).max() + 1e-14
        assert np.abs(gm["P"] - om["P"]).max() <= 1e-12 * np.abs(om["P"]).max() + 1e-14
