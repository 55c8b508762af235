"""Runs with 16-bit population storage, bit for bit. Every step rounds each
population to 16 bits, and a last bit of the FP32 or FP64 arithmetic before it
decides which way: another order of a sum gives another sequence of roundings,
1e-4 to 1e-2 of the velocity away after a hundred steps, although neither is
more exact. So the geometry's link sums, the initial state, the step and the
moments of such runs are pinned by digests of their values."""
import zlib

import numpy as np
import pytest

from paper_2401_17183_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MESHES = {
    "even_rows": lambda: W.channel_mesh(16, 12, 8, stretch=0.7, bump=0.05),
    "odd_rows": lambda: W.channel_mesh(9, 7, 37, stretch=0.5, bump=0.02),
    "whole_tiles": lambda: W.channel_mesh(11, 9, 128, stretch=0.5, bump=0.02),
    "general": lambda: W.channel_bump3d_mesh(12, 10, 16, stretch=0.7, bump=0.05),
    "channel2d": lambda: W.channel2d_mesh(31, 40, stretch=0.5),
}


def _mesh(name):
    """The mesh with its positions rounded to 2^-20, so that no host's sin or tanh shows."""
    mesh = dict(MESHES[name]())
    mesh["x"] = np.round(np.asarray(mesh["x"], dtype=np.float64) * 2.0 ** 20) / 2.0 ** 20
    return mesh


@pytest.fixture(scope="module")
def V():
    from paper_2401_17183_gb300 import build as B
    B.build()
    from paper_2401_17183_gb300 import vlb
    vlb.load()
    return vlb


def _digest(*arrays):
    crc = 0
    for a in arrays:
        crc = zlib.crc32(np.ascontiguousarray(a, dtype=np.float64).tobytes(), crc)
    return "%08x" % crc


def _run(V, mesh, prec, mode, ref):
    """A simulation, and the same flow's initial state as the FP64 path gives it."""
    force = (1e-5, -4e-6, 6e-6) if mesh["dim"] == 3 else (2e-6, 1e-5, 0)
    rho, u = W.noise_fields(mesh, amp=0.01, seed=5)
    vm, prm = V.Mesh(mesh), W.params(0.8, body_force=force)
    s = V.Sim(vm, prm, rho, u, precision=getattr(V, "VLB_" + prec), coef_mode=getattr(V, "VLB_COEF_" + mode),
              reference=getattr(V, "VLB_REF_" + ref))
    return s, V.Sim(vm, prm, rho, u).get_state()


LINK_SUMS = {
    "channel2d": "5c538014", "even_rows": "a2332909", "general": "d1ec4710", "odd_rows": "4a8a0037",
    "whole_tiles": "51a7261e",
}


@pytest.mark.parametrize("name", sorted(MESHES))
def test_link_sums(V, name):
    assert _digest(V.Mesh(_mesh(name)).geometry()["K"]) == LINK_SUMS[name]


PLANE = [(m, p, "AUTO", r) for m in ("even_rows", "odd_rows", "whole_tiles", "channel2d") for p in ("F16", "BF16")
         for r in ("REST", "UNIFORM")]
STEPS = {
    "even_rows-F16-AUTO-REST": "0bd544d8", "even_rows-F16-AUTO-UNIFORM": "8589fcc8",
    "even_rows-BF16-AUTO-REST": "32f09459", "even_rows-BF16-AUTO-UNIFORM": "e0160812",
    "odd_rows-F16-AUTO-REST": "6cd6f8a7", "odd_rows-F16-AUTO-UNIFORM": "4a8e93b9",
    "odd_rows-BF16-AUTO-REST": "2681e163", "odd_rows-BF16-AUTO-UNIFORM": "c25ef3f7",
    "whole_tiles-F16-AUTO-REST": "b57a875d", "whole_tiles-F16-AUTO-UNIFORM": "d5477769",
    "whole_tiles-BF16-AUTO-REST": "3321055e", "whole_tiles-BF16-AUTO-UNIFORM": "942b356d",
    "channel2d-F16-AUTO-REST": "d68da9c7", "channel2d-F16-AUTO-UNIFORM": "f9221850",
    "channel2d-BF16-AUTO-REST": "b811683f", "channel2d-BF16-AUTO-UNIFORM": "7bc9ad7d",
}


def _step_digest(V, case):
    name, prec, mode, ref = case
    s, N = _run(V, _mesh(name), prec, mode, ref)
    s.set_state(N)
    states = []
    for n in (1, 1, 19):
        for _ in range(n):
            s.step(1)
        states.append(s.get_state())
    return _digest(*states)


@pytest.mark.parametrize("case", PLANE, ids="-".join)
def test_steps(V, case):
    assert _step_digest(V, case) == STEPS["-".join(case)]


INITIAL = {
    "even_rows-F16-AUTO-REST": "c11e6111", "even_rows-F16-AUTO-UNIFORM": "a61eaeeb",
    "even_rows-BF16-AUTO-REST": "9c1d1680", "even_rows-BF16-AUTO-UNIFORM": "fa6fdaf4",
    "odd_rows-F16-AUTO-REST": "202c6631", "odd_rows-F16-AUTO-UNIFORM": "54361136",
    "odd_rows-BF16-AUTO-REST": "8a10b247", "odd_rows-BF16-AUTO-UNIFORM": "7cf77f39",
    "whole_tiles-F16-AUTO-REST": "2a16aa7a", "whole_tiles-F16-AUTO-UNIFORM": "f526ed1d",
    "whole_tiles-BF16-AUTO-REST": "e7813a84", "whole_tiles-BF16-AUTO-UNIFORM": "e4b8a683",
    "channel2d-F16-AUTO-REST": "204812f6", "channel2d-F16-AUTO-UNIFORM": "84e64455",
    "channel2d-BF16-AUTO-REST": "8790d7b7", "channel2d-BF16-AUTO-UNIFORM": "bcadea85",
}


@pytest.mark.parametrize("case", PLANE, ids="-".join)
def test_initial_state(V, case):
    name, prec, mode, ref = case
    s, _ = _run(V, _mesh(name), prec, mode, ref)
    assert _digest(s.get_state()) == INITIAL["-".join(case)]


MOMENTS = {
    "even_rows-F16-AUTO-REST": "d5af4d01", "even_rows-F16-AUTO-UNIFORM": "8d691d28",
    "even_rows-BF16-AUTO-REST": "89466f16", "even_rows-BF16-AUTO-UNIFORM": "1b099365",
    "odd_rows-F16-AUTO-REST": "2f09d30c", "odd_rows-F16-AUTO-UNIFORM": "14dcef6f",
    "odd_rows-BF16-AUTO-REST": "8ed0ac40", "odd_rows-BF16-AUTO-UNIFORM": "6ad3dddf",
    "whole_tiles-F16-AUTO-REST": "6ede362d", "whole_tiles-F16-AUTO-UNIFORM": "f17179c4",
    "whole_tiles-BF16-AUTO-REST": "0ac4eb9d", "whole_tiles-BF16-AUTO-UNIFORM": "f92f426b",
    "channel2d-F16-AUTO-REST": "04ea3ebd", "channel2d-F16-AUTO-UNIFORM": "1d546fc5",
    "channel2d-BF16-AUTO-REST": "ba2f99f5", "channel2d-BF16-AUTO-UNIFORM": "d97f521a",
}


def _moments_digest(V, case):
    name, prec, mode, ref = case
    s, N = _run(V, _mesh(name), prec, mode, ref)
    s.set_state(N)
    out = []
    for n in (1, 1, 19):      # both parities
        s.step(n)
        m = s.moments()
        out += [m["rho"], m["u"], m["u_tilde"]]
    return _digest(*out)


@pytest.mark.parametrize("case", PLANE, ids="-".join)
def test_moments(V, case):
    assert _moments_digest(V, case) == MOMENTS["-".join(case)]


GENERAL = [(m, p, "FULL", "UNIFORM") for m in ("odd_rows", "general", "channel2d") for p in ("F16", "BF16")]
RECORD_PER_CELL = {
    "odd_rows-F16-FULL-UNIFORM": ["f4136f97", "13a2aa24"], "odd_rows-BF16-FULL-UNIFORM": ["7c7c1d94", "7dde50ed"],
    "general-F16-FULL-UNIFORM": ["430a5077", "5e41db62"], "general-BF16-FULL-UNIFORM": ["984d3000", "a580c551"],
    "channel2d-F16-FULL-UNIFORM": ["5cfdf266", "ab0ec671"], "channel2d-BF16-FULL-UNIFORM": ["d7a804c9", "9b2f1d0c"],
}


@pytest.mark.parametrize("case", GENERAL, ids="-".join)
def test_one_record_per_cell(V, case):
    assert [_step_digest(V, case), _moments_digest(V, case)] == RECORD_PER_CELL["-".join(case)]
