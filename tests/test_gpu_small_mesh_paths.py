"""Which launch a small mesh's steps take, and calls longer than one launch holds
(1024 steps): the split, its odd starts and its remainder of one step. The
populations are those of single steps bit for bit, in every form of record,
mesh, precision and launch."""
import numpy as np
import pytest

from paper_2401_17183_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEP, CLUSTER, COOPERATIVE = 1, 2, 3


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


def _sheared(*n):
    mesh = dict(W.channel_mesh(*n, stretch=0.5, bump=0.02))
    x = np.array(mesh["x"], dtype=np.float64).reshape(n + (3,))
    shift = np.array(mesh["shift"], dtype=np.float64)
    x[..., 2] += 0.0625 * x[..., 0]
    shift[0][2] = 0.0625 * n[0]
    mesh["x"], mesh["shift"] = x.reshape(np.asarray(mesh["x"]).shape), shift
    return mesh


# mesh, launch of FP32 runs (FP64: always cooperative)
MESHES = {
    "one_block": (lambda: W.channel2d_mesh(2, 64, stretch=0.5), CLUSTER),
    "box": (lambda: W.periodic_sine_mesh(33, 0.02), CLUSTER),
    "plane2d": (lambda: W.channel2d_mesh(31, 40, stretch=0.5), CLUSTER),
    "cells2d": (lambda: W.channel2d_mesh(32, 64, stretch=0.5, bump=0.1), CLUSTER),
    "cluster_limit": (lambda: W.channel2d_mesh(64, 64, stretch=0.5, bump=0.1), CLUSTER),
    "past_cluster": (lambda: W.channel2d_mesh(65, 64, stretch=0.5, bump=0.1), COOPERATIVE),
    "extruded": (lambda: W.channel_mesh(16, 9, 25, stretch=0.5, bump=0.02), CLUSTER),
    "extruded_large": (lambda: W.channel_mesh(16, 19, 25, stretch=0.5, bump=0.02), COOPERATIVE),
    "sheared": (lambda: _sheared(11, 9, 40), CLUSTER),
    "cells": (lambda: W.channel_bump3d_mesh(16, 12, 17, stretch=0.5, bump=0.02), CLUSTER),
    "cells_large": (lambda: W.channel_bump3d_mesh(16, 22, 17, stretch=0.5, bump=0.02), COOPERATIVE),
}


def _pair(V, mesh, prec, **kw):
    force = (1e-5, 2e-6, 3e-6) if mesh["dim"] == 3 else (2e-6, 1e-5, 0)
    rho, u = W.noise_fields(mesh, amp=0.01, seed=4)
    vm = V.Mesh(mesh)
    return [V.Sim(vm, W.params(0.7, body_force=force, **kw), rho, u, precision=getattr(V, "VLB_" + prec)) for _ in range(2)]


@pytest.mark.parametrize("prec", ["F32", "F64"])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_launch_taken_and_populations(V, name, prec):
    make, launch = MESHES[name]
    a, b = _pair(V, make(), prec)
    path = V.load().vlb_internal_step_path
    for n in (2, 1, 3, 40):        # the third call starts on odd parity
        a.step(n)
        assert path(a.h) == (STEP if n == 1 else launch if prec == "F32" else COOPERATIVE)
        for _ in range(n):
            b.step(1)
        assert path(b.h) == STEP
        assert np.array_equal(a.get_state(), b.get_state()), n


@pytest.mark.parametrize("prec", ["F32", "F64"])
@pytest.mark.parametrize("bump", [0.0, 0.05])
def test_moving_walls(V, prec, bump):
    wu = np.zeros((3, 2, 3))
    wu[0, 0, 1], wu[0, 1, 1] = 0.02, -0.01
    a, b = _pair(V, W.channel2d_mesh(20, 36, stretch=0.5, bump=bump), prec, wall_u=wu)
    a.step(25)
    for _ in range(25):
        b.step(1)
    assert np.array_equal(a.get_state(), b.get_state())


@pytest.mark.parametrize("prec", ["F32", "F64"])
def test_calls_longer_than_a_launch(V, prec):
    a, b = _pair(V, W.channel2d_mesh(12, 24, stretch=0.5, bump=0.05), prec)
    path = V.load().vlb_internal_step_path
    for n, last in ((1, STEP), (1025, STEP), (2049, STEP), (1026, None)):
        a.step(n)
        assert path(a.h) == (last or (CLUSTER if prec == "F32" else COOPERATIVE))
    for _ in range(a.time()):
        b.step(1)
    assert a.time() == b.time() == 4101
    assert np.array_equal(a.get_state(), b.get_state())
    a.sync()
