"""The FP64 force solve takes its last change to first order in FP32 instead of
evaluating the map once more. A step's populations are those of a solve that
goes on until nothing changes (tol = 1e-30: to 64 units of the last place, with
the same correction after that), but for last bits: what is left of the force
is below 1e-19 of m, and a population of 1e-3 to 1e-1 keeps 2e-19 to 1.4e-17,
so that less than one in 30 rounds the other way."""
import numpy as np
import pytest

from paper_2401_17183_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "extruded": lambda: W.channel_mesh(20, 12, 24, stretch=0.7, bump=0.05),
    "cells": lambda: W.channel_bump3d_mesh(20, 16, 24, stretch=0.7, bump=0.05),
    "channel2d": lambda: W.channel2d_mesh(31, 40, stretch=0.7),
    "channel2d_cells": lambda: W.channel2d_mesh(64, 100, stretch=0.7, bump=0.1),
    "box2d": lambda: W.periodic_sine_mesh(64, 0.02),
}


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


@pytest.mark.parametrize("name", sorted(MESHES))
@pytest.mark.parametrize("amp", [0.01, 0.04])
def test_step_as_solved_to_the_end(V, name, amp):
    mesh = MESHES[name]()
    force = (1e-5, -4e-6, 6e-6) if mesh["dim"] == 3 else (2e-6, 1e-5, 0)
    rho, u = W.noise_fields(mesh, amp=amp, seed=5)
    vm, states = V.Mesh(mesh), []
    for tol in (0.0, 1e-30):
        s = V.Sim(vm, W.params(0.8, body_force=force, tol=tol), rho, u)
        s.step(1)
        states.append(s.get_state())
    a, b = states
    assert np.mean(a != b) < 1.0 / 30.0
    assert np.abs(a - b).max() <= 2.0 ** -53      # one unit of the last place of N below 1
