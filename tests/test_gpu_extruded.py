"""Extruded meshes (the first two coordinates do not depend on the fastest
axis, the third on nothing else) take a shorter form of the collision; meshes
that are merely invariant along the fastest axis do not. Both forms against
the FP64 oracle, with a spanwise spacing other than one, a body force along
every axis, moving walls, and rows that are whole tiles, ragged, or so short
that tiles lie along them. Bounds as elsewhere in the suite: FP64 1e-12 after
40 steps, FP32 2e-5 after 100. The members of a batch, extruded or not, give
their own steps bit for bit.
"""
import numpy as np
import pytest

from oracle import OracleSim
from paper_2401_17183_gb300 import workloads as W

from .helpers import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


def _mesh(n0, n1, n2, kind):
    mesh = dict(W.channel_mesh(n0, n1, n2, stretch=0.5, bump=0.02))
    x = np.array(mesh["x"], dtype=np.float64).reshape(n0, n1, n2, 3)
    shift = np.array(mesh["shift"], dtype=np.float64)
    if kind == "spacing":          # extruded, g^zz = (32/31)^2
        x[..., 2] *= 31.0 / 32.0
        shift[2] *= 31.0 / 32.0
    elif kind == "sheared":        # invariant along the fastest axis, g^02 != 0
        x[..., 2] += 0.0625 * x[..., 0]
        shift[0][2] = 0.0625 * n0
    mesh["x"], mesh["shift"] = x.reshape(np.asarray(mesh["x"]).shape), shift
    return mesh


def _params(moving):
    wall_u = None
    if moving:
        wall_u = np.zeros((3, 2, 3))
        wall_u[1, 1] = (0.02, 0.0, 0.01)
    return W.params(0.8, body_force=(1e-5, -4e-6, 6e-6), wall_u=wall_u)


@pytest.mark.parametrize("kind", ["spacing", "sheared"])
@pytest.mark.parametrize("n2,moving", [(128, False), (40, True), (7, True)])
def test_extruded_and_sheared_against_oracle(V, kind, n2, moving):
    mesh, prm = _mesh(11, 9, n2, kind), _params(moving)
    rho, u = W.noise_fields(mesh, amp=0.01, seed=5)
    o = OracleSim(mesh, prm)
    o.init(rho, u)
    # 41 steps: one call of 40 (small meshes: one launch) and one of one step
    o.step(41)
    m41 = o.moments()
    o.step(59)
    m100 = o.moments()
    for prec, steps, want, tol in ((V.VLB_F64, 41, m41, 1e-12), (V.VLB_F32, 100, m100, 2e-5)):
        g = V.Sim(V.Mesh(mesh), prm, rho, u, precision=prec)
        assert g.layout()["plane"]
        g.step(steps - 1)
        g.step(1)
        m = g.moments()
        su = np.abs(want["u"]).max()
        assert rel_err(m["rho"], want["rho"], 1.0) < tol
        assert rel_err(m["u"], want["u"], su) < tol
        assert rel_err(m["u_tilde"], want["u_tilde"], su) < tol


@pytest.mark.parametrize("prec", ["VLB_F32", "VLB_F64"])
def test_batch_of_extruded_and_other_members(V, prec):
    def sims():
        out = []
        for i, (kind, n2) in enumerate((("spacing", 40), ("sheared", 24), ("spacing", 130))):
            mesh = _mesh(11, 9, n2, kind)
            rho, u = W.noise_fields(mesh, amp=0.01, seed=7 + i)
            out.append(V.Sim(V.Mesh(mesh), _params(False), rho, u, precision=getattr(V, prec)))
        return out

    alone, members = sims(), sims()
    b = V.Batch(members)
    b.step(35)
    for s, t in zip(alone, members):
        s.step(35)
        t.sync()
        assert np.array_equal(s.get_state(), t.get_state())


@pytest.mark.parametrize("prec", ["VLB_F32", "VLB_F16", "VLB_BF16"])
@pytest.mark.parametrize("kind", ["spacing", "sheared"])
@pytest.mark.parametrize("n2,copies", [(64, 2), (96, 4)])
def test_rows_of_whole_tiles_repeat_a_narrower_mesh(V, prec, kind, n2, copies):
    """A flow that repeats along the fastest axis, on rows of whole tiles (the
    block copies the neighbouring rows' segments on odd steps, with wrap-around
    pieces at their ends and, in 16 bits, values one half-word to the side)
    and on rows of one period (copied value by value): the same populations."""
    precision = getattr(V, prec)
    got = []
    for k in (1, copies):
        mesh = _mesh(11, 9, n2 * k, kind)
        rho, u = W.noise_fields(_mesh(11, 9, n2, kind), amp=0.01, seed=5)
        rho = np.tile(rho.reshape(99, n2), (1, k)).reshape(-1)
        u = np.tile(u.reshape(99, n2, 3), (1, k, 1)).reshape(-1, 3)
        g = V.Sim(V.Mesh(mesh), _params(True), rho, u, precision=precision,
                  reference=V.VLB_REF_UNIFORM if prec == "VLB_F32" else V.VLB_REF_REST)
        for _ in range(13):
            g.step(1)
        got.append(g.get_state().reshape(19, 99, k, n2))
    for k in range(copies):
        assert np.array_equal(got[1][:, :, k], got[0][:, :, 0])
