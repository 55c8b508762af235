"""FP64 runs at densities beyond FP32's range: every relation of the method is
homogeneous of degree one in the populations, so a run at 2^130 (D3Q39, whose
populations are stored as they are, at 2^-130 too) times the density is that
run scaled, to FP64 rounding."""
import numpy as np
import pytest

from paper_2401_17183_gb300 import workloads as W

from .helpers import rel_err

pytestmark = pytest.mark.gpu

MESHES = {
    "box2d": lambda: W.periodic_sine_mesh(16, 0.02),
    "channel": lambda: W.channel_mesh(11, 9, 20, stretch=0.5, bump=0.02),
    "channel_cells": lambda: W.channel_bump3d_mesh(11, 9, 12, stretch=0.5, bump=0.02),
    "d3q39": lambda: W.periodic_sine_mesh3d(8, 0.01, q=39),
}


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


@pytest.mark.parametrize("name,power", [(n, 130) for n in sorted(MESHES)] + [("d3q39", -130)])
def test_scaled_densities(V, name, power):
    mesh = MESHES[name]()
    prm = W.params(0.8, body_force=(1e-5, 2e-6, 0.0))
    rho, u = W.noise_fields(mesh, amp=0.01, seed=3, rho_amp=0.01)
    scale = 2.0 ** power
    vm = V.Mesh(mesh)
    a, b = (V.Sim(vm, prm, rho * f, u) for f in (1.0, scale))
    for n in (1, 1, 8):          # single steps, both parities, and (small meshes) one launch of eight
        a.step(n)
        b.step(n)
        assert rel_err(b.get_state() / scale, a.get_state()) < 1e-13
        ma, mb = a.moments(), b.moments()
        assert rel_err(mb["rho"] / scale, ma["rho"]) < 1e-13
        assert rel_err(mb["u_tilde"], ma["u_tilde"]) < 1e-12
