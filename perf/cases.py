"""The work a user of this library has it do, as measurable cases.

Each case is one pass of a program that uses the public entry points
(vlb.Sim / vlb.Mesh / vlb.Batch / nn.Net): a run of time steps between two
looks at the fields, a batch of runs, the set-up of a simulation on a new
mesh, or a pass of the warm-start network. The kinds:

  flow    vlb_reset from host fields, vlb_step(steps), vlb_moments into host
          buffers. mesh "channel" (plane coefficient records, walls), "bump3d"
          (a geometry that varies along every axis: one record per cell),
          "channel2d" (D2Q9), "box2d" (D2Q9, periodic curved box), "sine3d"
          (periodic curved box; D3Q39)
  batch   many uneven D2Q9 channels advanced by one launch per step, then the
          fields of every member
  setup   vlb.Mesh (geometry precompute) and vlb.Sim (coefficient records,
          initial populations) on new node positions, then the fields
  nn      the warm-start network: a forward pass, or the forward pass, the
          loss and the gradients of a training iteration

Fields come back in the type the populations are stored in (FP64, FP32, FP16
or BF16); the network's FP32 interface comes back as it is.

exact() is the same method, written from its equations with torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2401_17183_gb300 import nn, vlb
from paper_2401_17183_gb300 import workloads as W

STORAGE = {"f64": (vlb.VLB_F64, torch.float64), "f32": (vlb.VLB_F32, torch.float32),
           "f16": (vlb.VLB_F16, torch.float16), "bf16": (vlb.VLB_BF16, torch.bfloat16)}
NN_CI, NN_CO = 8, 3          # channels of the warm-start network


def listed():
    return [
        # the headline workload: a channel with a bumped wall, 16.8 M cells, FP32
        # (100 steps between two looks at the fields, as the warm start's residual
        # checks, or 200)
        flow("channel_f32_256", "channel", 256, 256, 256, "f32", 200),
        # the same channel family with 16-bit populations relative to the rest state
        flow("channel_f16_128", "channel", 128, 128, 128, "f16", 100),
        # a mesh that varies along every axis: one coefficient record per cell
        flow("general_f32_160x96x128", "bump3d", 160, 96, 128, "f32", 100),
        # odd sizes: ragged tiles, rows that start off every alignment
        flow("channel_f32_ragged", "channel", 75, 67, 101, "f32", 100),
        # FP64 reference run of the storage-precision comparison (64^3)
        flow("channel_f64_64", "channel", 64, 64, 64, "f64", 100),
        # the smallest calls: the 64 x 64 mapped box in FP64 and one 2D channel of the
        # warm start's size, where launches and latency count
        flow("box2d_f64_64", "box2d", 64, 64, 1, "f64", 200),
        flow("channel2d_f32_32x64", "channel2d", 32, 64, 1, "f32", 100),
        # the 6th-order isotropic velocity set
        flow("d3q39_f64_64", "sine3d", 64, 64, 64, "f64", 10),
        # uneven 2D channels in one launch per step, fields of every member after 320 steps
        {"name": "batch_f32_64", "kind": "batch", "members": 64, "lo": 64, "hi": 512, "steps": 320, "tune": False},
        # a new mesh: geometry precompute, records, initial fields
        {"name": "setup_general_f32", "kind": "setup", "mesh": "bump3d", "n0": 96, "n1": 64, "n2": 80,
         "storage": "f32", "steps": 0},
        # serving the warm start: one batch through the network
        net("nn_forward_bf16_b32", "forward", 64, 32, 64, 32, "bf16"),
        # one training iteration's gradients at the training batch
        net("nn_grad_bf16_b32", "grad", 64, 32, 64, 32, "bf16"),
    ]


def flow(name, mesh, n0, n1, n2, storage, steps, reference="rest"):
    c = {"kind": "flow", "mesh": mesh, "n0": n0, "n1": n1, "n2": n2, "storage": storage, "steps": steps}
    if storage in ("f16", "bf16"):
        c["reference"] = reference
    return dict(c, name=name) if name else c


def net(name, what, width, H, Wd, batch, storage):
    c = {"kind": "nn", "what": what, "width": width, "H": H, "W": Wd, "batch": batch, "storage": storage}
    return dict(c, name=name) if name else c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plane", "plane", "general", "storage16", "f64", "flow2d", "flow2d", "q39", "batch", "setup",
                       "forward", "grad"])
    if kind in ("plane", "storage16", "general", "f64"):
        # wall-normal size from the log range; the streamwise and spanwise sizes at
        # least that (the bump's slope grows with their ratio)
        n1 = _log(rng, 12, {"plane": 176, "storage16": 128, "general": 96, "f64": 48}[kind])
        n0, n2 = (int(n1 * rng.uniform(1.0, 1.6)) for _ in range(2))
        storage = {"plane": "f32", "general": "f32", "f64": "f64", "storage16": rng.choice(["f16", "bf16"])}[kind]
        mesh = "bump3d" if kind == "general" else "channel"
        if kind == "f64":
            mesh = rng.choice(["channel", "channel", "bump3d"])
        ref = rng.choice(["rest", "rest", "uniform"])
        return flow(None, mesh, n0, n1, n2, storage, rng.choice([50, 100, 101, 200]) if n1 < 96 else 100, ref)
    if kind == "flow2d":
        mesh = rng.choice(["channel2d", "channel2d", "box2d"])
        n0 = _log(rng, 16, 384)
        n1 = n0 if mesh == "box2d" else int(n0 * rng.uniform(1.0, 2.5))
        return flow(None, mesh, n0, n1, 1, rng.choice(["f32", "f32", "f64"]), rng.choice([100, 101, 320]))
    if kind == "q39":
        L = _log(rng, 12, 60)
        return flow(None, "sine3d", L, L, L, "f64", rng.choice([5, 10]))
    if kind == "batch":
        hi = rng.choice([128, 256, 384])
        return {"kind": "batch", "members": _log(rng, 8, 96), "lo": 64, "hi": hi, "steps": rng.choice([100, 200, 320]),
                "tune": rng.random() < 0.5}
    if kind == "setup":
        n1 = _log(rng, 16, 64)
        n0, n2 = (int(n1 * rng.uniform(1.0, 1.6)) for _ in range(2))
        return {"kind": "setup", "mesh": rng.choice(["bump3d", "channel"]), "n0": n0, "n1": n1, "n2": n2,
                "storage": rng.choice(["f32", "f32", "f64"]), "steps": 0}
    # the network: the warm start's width and grid and their neighbours
    storage = rng.choice(["bf16", "bf16", "bf16", "f32"])
    width = rng.choice([16, 32, 64, 64])
    H, Wd = rng.choice([(32, 64), (32, 64), (32, 96), (64, 64), (64, 128)])
    return net(None, kind, width, H, Wd, _log(rng, 1, 32 * 2048 // (H * Wd) if width == 64 else 32), storage)


# ------------------------------------------------------------------- inputs

def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed) + 1)


def _noise(seed, n, dim, amp):
    return amp * (2.0 * torch.rand((n, dim), generator=_gen(seed), dtype=torch.float64, device="cuda") - 1.0)


def _mesh(c):
    n = (c["n0"], c["n1"], c["n2"])
    if c["mesh"] == "channel":
        return W.channel_mesh(*n, stretch=0.7, bump=0.05)
    if c["mesh"] == "bump3d":
        return W.channel_bump3d_mesh(*n, stretch=0.7, bump=0.05)
    if c["mesh"] == "channel2d":
        return W.channel2d_mesh(n[0], n[1], stretch=0.7, bump=0.1)
    if c["mesh"] == "box2d":
        return W.periodic_sine_mesh(n[0], amp_frac=0.02)
    return W.periodic_sine_mesh3d(n[0], 0.01, q=39)


# tau and body force of each mesh family (as the repository's workloads)
def _params(c):
    G = {"channel": (1e-6, 0.0, 0.0), "bump3d": (1e-6, 0.0, 0.0), "channel2d": (0.0, 1e-5, 0.0),
         "box2d": (0.0, 0.0, 0.0), "sine3d": (1e-5, 0.0, 2e-6)}[c["mesh"]]
    return W.params(0.8, body_force=G)


def _fields(c, mesh, seed):
    """rho = 1 and seeded 1% velocity noise; the mapped box: Taylor-Green flow
    plus 1e-4 noise. Device tensors."""
    nc, dim = W.ncell(mesh), mesh["dim"]
    rho = torch.ones(nc, dtype=torch.float64, device="cuda")
    if c["mesh"] == "box2d":
        k = 2.0 * math.pi / c["n0"]
        X = torch.from_numpy(W.node_positions(mesh)).cuda() * k
        u = 0.01 * torch.stack([torch.sin(X[:, 0]) * torch.cos(X[:, 1]), -torch.cos(X[:, 0]) * torch.sin(X[:, 1])], -1)
        return rho, u + _noise(seed, nc, dim, 1e-4)
    return rho, _noise(seed, nc, dim, 0.01)


def _pinned(*shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True)


def _host(t):
    p = _pinned(*t.shape)
    p.copy_(t)
    return p


def _batch_members(c, seed):
    """(mesh, params) of a batch: channels of log-uniform length in [lo, hi]
    and half as high, with seeded stretching, bump and force; the sizes do not
    depend on the seed, so that every seed is the same amount of work."""
    sizes = np.exp(np.linspace(math.log(c["lo"]), math.log(c["hi"]), c["members"]))
    r = torch.rand((c["members"], 3), generator=_gen(seed, "cpu"), dtype=torch.float64).tolist()
    out = []
    for n, (a, b, g) in zip(sizes, r):
        n = int(n)
        mesh = W.channel2d_mesh(n // 2, n, stretch=0.3 + 0.5 * a, bump=0.1 * b)
        out.append((mesh, W.params(0.8, body_force=(0.0, (1.0 + g) * 1e-6, 0.0))))
    return out


def _batch_fields(nc, seed):
    return torch.ones(nc, dtype=torch.float64, device="cuda"), _noise(seed, nc, 2, 0.01)


def _nn_inputs(c, seed):
    """Parameters (He-uniform weights, small biases), inputs and targets."""
    g = _gen(seed)
    r = lambda *s: 2.0 * torch.rand(s, generator=g, device="cuda") - 1.0  # noqa: E731
    layers = [(r(co, ci, k, k) * math.sqrt(6.0 / (ci * k * k)), 0.05 * r(co))
              for co, ci, k in nn.layer_shapes(NN_CI, NN_CO, c["width"])]
    x, t = r(c["batch"], NN_CI, c["H"], c["W"]), r(c["batch"], NN_CO, c["H"], c["W"])
    return layers, x, t


# ---------------------------------------------------------------- the passes

def prepare(case, seed):
    c, k = case, case["kind"]
    s = {"case": c}
    if k == "flow":
        mesh = _mesh(c)
        rho, u = _fields(c, mesh, seed)
        s["rho"], s["u"] = _host(rho), _host(u)
        prec, dt = STORAGE[c["storage"]]
        ref = vlb.VLB_REF_REST if c.get("reference") == "rest" else vlb.VLB_REF_UNIFORM
        s["sim"] = vlb.Sim(vlb.Mesh(mesh), _params(c), s["rho"].numpy(), s["u"].numpy(), precision=prec, reference=ref)
        s.update(_outputs(W.ncell(mesh), mesh["dim"], dt))
    elif k == "batch":
        members = _batch_members(c, seed)
        s["off"] = np.concatenate([[0], np.cumsum([W.ncell(m) for m, _ in members])]).tolist()
        rho, u = (t.cpu().numpy() for t in _batch_fields(s["off"][-1], seed))
        part = [slice(a, b) for a, b in zip(s["off"], s["off"][1:])]
        sims = [vlb.Sim(vlb.Mesh(mesh), prm, rho[k], u[k], precision=vlb.VLB_F32)
                for (mesh, prm), k in zip(members, part)]
        s["batch"] = vlb.Batch(sims)
        if c["tune"]:
            s["batch"].tune(4)
            for sim, k in zip(sims, part):   # back at the start, time 0
                sim.reset(rho[k], u[k])
        s.update(_outputs(s["off"][-1], 2, torch.float32, c["members"]))
    elif k == "setup":
        s["mesh"] = _mesh(c)
        rho, u = _fields(c, s["mesh"], seed)
        s["rho"], s["u"] = _host(rho), _host(u)
        s.update(_outputs(W.ncell(s["mesh"]), s["mesh"]["dim"], STORAGE[c["storage"]][1]))
    else:
        layers, s["x"], s["t"] = _nn_inputs(c, seed)
        s["net"] = nn.Net(NN_CI, NN_CO, c["width"], c["H"], c["W"], c["batch"],
                          storage=nn.VLB_NN_BF16 if c["storage"] == "bf16" else nn.VLB_NN_F32)
        s["net"].set_params(torch.cat([v.reshape(-1) for l in layers for v in l]).cpu().numpy())
        s["y"] = torch.zeros_like(s["t"])
        s["dy"] = torch.zeros_like(s["t"])
        s["grads"] = torch.zeros(s["net"].nparams, dtype=torch.float32, pin_memory=True)
    return s


def _outputs(nc, dim, dt, members=1):
    """Host buffers for the fields in FP64 (as vlb_moments gives them) and in
    the type of the populations."""
    o = {"rho64": _pinned(nc), "ut64": _pinned(nc, dim), "tot64": _pinned(members, 7)}
    if dt != torch.float64:
        o["rho_out"], o["ut_out"] = torch.zeros(nc, dtype=dt), torch.zeros((nc, dim), dtype=dt)
    return o


def _look(sims, o):
    """Density, fluid velocity and the conservation totals of simulations, one
    after another in the host buffers."""
    cell = 0
    for k, sim in enumerate(sims):
        sim.moments_ptr(o["rho64"].data_ptr() + 8 * cell, 0, o["ut64"].data_ptr() + 8 * cell * sim.mesh.dim,
                        o["tot64"].data_ptr() + 56 * k)
        cell += sim.mesh.ncell
    if "rho_out" not in o:
        return [o["rho64"], o["ut64"], o["tot64"]]
    o["rho_out"].copy_(o["rho64"])
    o["ut_out"].copy_(o["ut64"])
    return [o["rho_out"], o["ut_out"], o["tot64"].float()]


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "flow":
        s["sim"].reset_ptr(s["rho"].data_ptr(), s["u"].data_ptr())
        s["sim"].step(c["steps"])
        return _look([s["sim"]], s)
    if c["kind"] == "batch":
        s["batch"].step(c["steps"])
        return _look(s["batch"].sims, s)
    if c["kind"] == "setup":
        mesh = vlb.Mesh(s["mesh"])
        sim = vlb.Sim(mesh, _params(c), s["rho"].numpy(), s["u"].numpy(), precision=STORAGE[c["storage"]][0])
        out = _look([sim], s)
        sim.close()
        mesh.close()
        return out
    B, n = c["batch"], s["net"]
    n.forward(s["x"].data_ptr(), s["y"].data_ptr(), B)
    if c["what"] == "forward":
        return s["y"]
    loss = n.mse(s["y"].data_ptr(), s["t"].data_ptr(), s["dy"].data_ptr(), B)
    n.backward(s["dy"].data_ptr(), B)
    nn.load().vlb_nn_get_grads(n.h, s["grads"].data_ptr())
    return {"y": s["y"], "loss": loss, "grads": s["grads"]}


def work(case):
    """Bytes: the populations read and written once per step (and, on a mesh
    that varies along every axis, its node positions read), the fields in and out; the
    set-up: positions and fields in, populations and fields out; the network:
    parameters, inputs and outputs. Operations: about 40 per population and
    step (moments, equilibrium, relaxation, force); the network's products."""
    c = case
    if c["kind"] == "nn":
        px, mac, npar = c["H"] * c["W"], 0, 0
        for i, (co, ci, k) in enumerate(nn.layer_shapes(NN_CI, NN_CO, c["width"])):
            mac += co * ci * k * k * px // {2: 4, 3: 4, 6: 4, 7: 4, 4: 16, 5: 16}.get(i, 1)
            npar += co * ci * k * k + co
        f = 2.0 * mac * c["batch"] * (3 if c["what"] == "grad" else 1)
        io = c["batch"] * px * (NN_CI + NN_CO) * 4
        return {"bytes": io + npar * (8 if c["what"] == "grad" else 2), "flops": f}
    es = {"f64": 8, "f32": 4}.get(c.get("storage", "f32"), 2)
    if c["kind"] == "batch":
        nc = sum((int(n) // 2) * int(n) for n in np.exp(np.linspace(math.log(c["lo"]), math.log(c["hi"]), c["members"])))
        return {"bytes": nc * (c["steps"] * 2 * 9 * 4 + 24), "flops": 40.0 * 9 * nc * c["steps"]}
    nc = c["n0"] * c["n1"] * c["n2"]
    dim = 2 if c["n2"] == 1 else 3
    q = 9 if dim == 2 else 39 if c["mesh"] == "sine3d" else 19
    if c["kind"] == "setup":
        return {"bytes": nc * (8 * dim + 16 * (1 + dim) + q * es), "flops": 200.0 * q * nc}
    per = 2 * q * es + (8 * dim if c["mesh"] in ("bump3d", "box2d") else 0)
    return {"bytes": nc * (c["steps"] * per + 16 * (1 + dim)), "flops": 40.0 * q * nc * c["steps"]}


# --------------------------------------------- the method in 64 bits, with torch

def _velocities(q):
    """c [q, D], w [q], T0 of D2Q9, D3Q19 and D3Q39."""
    D = 2 if q == 9 else 3
    reach = 3 if q == 39 else 1
    wt = {9: {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}, 19: {0: 1 / 3, 1: 1 / 18, 2: 1 / 36},
          39: {0: 1 / 12, 1: 1 / 12, 3: 1 / 27, 4: 2 / 135, 8: 1 / 432, 9: 1 / 1620}}[q]
    c, w = [], []
    for v in np.ndindex(*(2 * reach + 1,) * D):
        v = [i - reach for i in v]
        c2, m = sum(i * i for i in v), [abs(i) for i in v if i]
        if c2 not in wt or (q == 39 and (len(set(m)) > 1 or (c2 == 9 and len(m) > 1))):
            continue
        c.append(v)
        w.append(wt[c2])
    assert len(c) == q
    return torch.tensor(c, dtype=torch.float64, device="cuda"), torch.tensor(w, dtype=torch.float64, device="cuda"), \
        2 / 3 if q == 39 else 1 / 3


def _geometry(mesh, c):
    """J, g_i, g^i, the link sums K_a^i = sum_j c_a^j Theta^i_j(q + c_a, q)
    (zero through a wall), e_a(q - c_a), the source of each arriving
    population and whether it comes back from a wall; cells flattened."""
    D, n = mesh["dim"], list(mesh["n"][:mesh["dim"]])
    P = int(c.abs().max()) + 1
    x = torch.from_numpy(mesh["x"]).cuda().reshape(n + [D])
    wall = [mesh["bc"][a] == W.WALL for a in range(D)]
    for a in range(D):       # node positions beyond the ends of axis a
        m = x.shape[a]
        if wall[a]:
            lo, hi = [x.narrow(a, 0, 1), x.narrow(a, 1, 1)], [x.narrow(a, m - 1, 1), x.narrow(a, m - 2, 1)]
            below = [lo[0] + k * (lo[0] - lo[1]) for k in range(P, 0, -1)]
            above = [hi[0] + k * (hi[0] - hi[1]) for k in range(1, P + 1)]
        else:
            sh = torch.from_numpy(mesh["shift"][a, :D]).cuda()
            idx = torch.arange(-P, m + P, device="cuda")
            wrap = torch.div(idx, m, rounding_mode="floor")
            shape = [1] * D + [D]
            shape[a] = m + 2 * P
            x = x.index_select(a, idx - wrap * m) + (wrap[:, None] * sh[None, :]).reshape(shape)
            continue
        x = torch.cat(below + [x] + above, a)
    cut = lambda t, a, o: t.narrow(a, 1 + o, t.shape[a] - 2)  # noqa: E731
    g = []
    for i in range(D):       # tangents on the mesh and P - 1 cells around it
        y = x
        for a in range(D):
            if a != i:
                y = cut(y, a, 0)
        x0, dp, dm = cut(y, i, 0), cut(y, i, 1), cut(y, i, -1)
        dp, dm = dp - x0, dm - x0
        d = dp - dm
        beta = (dp.norm(dim=-1) + dm.norm(dim=-1)) / d.norm(dim=-1)
        g.append(0.5 * beta[..., None] * d / mesh["dx"])
    g = torch.stack(g, -2)   # [..., i, d]
    R = P - 1

    def at(v):               # tangents of q + v
        t = g
        for a in range(D):
            t = t.narrow(a, R + int(v[a]), n[a])
        return t.reshape(-1, D, D)

    gl = at([0] * D)
    J = torch.linalg.det(gl)
    gu = torch.linalg.inv(gl).transpose(1, 2).contiguous()
    ic = torch.stack([t.reshape(-1) for t in torch.meshgrid(*[torch.arange(k, device="cuda") for k in n], indexing="ij")])
    nt = torch.tensor(n, device="cuda")[:, None]
    wl = torch.tensor(wall, device="cuda")[:, None]
    st = [int(np.prod(n[a + 1:])) for a in range(D)]
    K, eb, src, back = [], [], [], []
    for v in c.long().cpu().tolist():
        vt = torch.tensor(v, device="cuda")[:, None]
        ve = torch.tensor(v, dtype=torch.float64, device="cuda")
        out = (((ic + vt < 0) | (ic + vt >= nt)) & wl).any(0)
        k = torch.einsum("j,njd,nid->ni", ve, at(v) - gl, gu)
        K.append(torch.where(out[:, None], torch.zeros_like(k), k))
        p = ic - vt
        b = (((p < 0) | (p >= nt)) & wl).any(0)
        p = p % nt
        back.append(b)
        src.append(sum(p[a] * st[a] for a in range(D)))
        e = torch.einsum("i,nid->nd", ve, gl)
        eb.append(torch.where(b[:, None], e, torch.einsum("i,nid->nd", ve, at([-t for t in v]))))
    return {"J": J, "gl": gl, "gu": gu, "K": torch.stack(K), "eb": torch.stack(eb), "src": torch.stack(src),
            "back": torch.stack(back)}


def _solve(meshes, params, rho, u, steps):
    """rho, u~ of every cell and [mass, P, M] of every mesh after `steps`
    steps from (rho, u); meshes of one velocity set, cells one after another."""
    q, D = meshes[0]["q"], meshes[0]["dim"]
    c, w, T0 = _velocities(q)
    geo = [_geometry(m, c) for m in meshes]
    nc = [g["J"].shape[0] for g in geo]
    off = np.concatenate([[0], np.cumsum(nc)])
    cat = lambda k, d: torch.cat([g[k] for g in geo], d)  # noqa: E731
    J, gl, gu, K, eb, back = cat("J", 0), cat("gl", 0), cat("gu", 0), cat("K", 1), cat("eb", 1), cat("back", 1)
    src = torch.cat([g["src"] + int(o) for g, o in zip(geo, off)], 1)
    G = torch.cat([gu[o:o + k] @ torch.tensor(p["body_force"][:D], dtype=torch.float64, device="cuda")
                   for p, o, k in zip(params, off, nc)]).T.contiguous()
    tau, n = params[0]["tau"], int(off[-1])
    del geo
    opp = [int(((c + v).abs().sum(1) == 0).nonzero()[0, 0]) for v in c]
    row = torch.arange(q, device="cuda")[:, None]
    gather = torch.where(back, torch.tensor(opp, device="cuda")[:, None] * n + torch.arange(n, device="cuda")[None],
                         row * n + src)
    del src, back
    K = K.permute(2, 0, 1).contiguous()                  # [i, a, cell]
    Kb = K[:, opp]
    M = K + Kb
    ginv = torch.einsum("nid,njd->ijn", gu, gu)
    eye = torch.eye(D, dtype=torch.float64, device="cuda")
    gd = ginv - eye[:, :, None]
    s2 = [(i, j) for i in range(D) for j in range(i, D)]
    s3 = [(i, j, k) for i in range(D) for j in range(i, D) for k in range(j, D)]
    perms = {2: lambda t: len({t, t[::-1]}), 3: lambda t: {1: 1, 2: 3, 3: 6}[len(set(t))]}
    h2 = torch.stack([perms[2](t) * (c[:, t[0]] * c[:, t[1]] / T0 - eye[t[0], t[1]]) / (2 * T0) for t in s2], 1)
    h3 = torch.stack([perms[3](t) * (c[:, t[0]] * c[:, t[1]] * c[:, t[2]] - T0 * (
        c[:, t[0]] * eye[t[1], t[2]] + c[:, t[1]] * eye[t[2], t[0]] + c[:, t[2]] * eye[t[0], t[1]])) / (6 * T0 ** 3)
        for t in s3], 1)
    basis = w[:, None] * torch.cat([c / T0, h2, h3], 1)
    hp = w[:, None] * ((c[:, :, None] * c[:, None, :] / T0 - eye) / T0).reshape(q, D * D)
    cw = w[:, None] * c / T0

    def feq(r, U, Ut):
        B = [gd[i, j] * T0 + Ut[i] * Ut[j] for i, j in s2]
        d = Ut - U
        t = lambda i, j, k: gd[i, j] * Ut[k] + (d[k] if i == j else 0.0)  # noqa: E731
        C = [T0 * (t(i, j, k) + t(j, k, i) + t(k, i, j)) + Ut[i] * Ut[j] * Ut[k] for i, j, k in s3]
        return r * (w[:, None] + basis @ torch.stack(list(U) + B + C))

    def collide(N, F):
        r = N.sum(0) / J
        U = (c.T @ N) / (J * r)
        for _ in range(200):
            f = feq(r, U, U + 0.5 * F / r)
            dP = torch.stack([c.T @ (M[j] * f) for j in range(D)], 1) * (-0.5 * (1.0 - 0.5 / tau))
            Np = N - (N - J * f) / tau + J * (cw @ F + hp @ dP.reshape(D * D, n))
            Fn = torch.stack([-0.5 * (K[i] * Np + Kb[i] * N).sum(0) for i in range(D)]) / J + r * G
            done = bool(((Fn - F).abs().amax(0) <= 1e-14 * torch.maximum(r, Fn.abs().amax(0))).all())
            F = Fn
            if done:
                break
        return r, U, F, Np

    U0 = torch.einsum("nd,nid->in", u, gu)
    N, F = J * feq(rho, U0, U0), torch.zeros((D, n), dtype=torch.float64, device="cuda")
    for _ in range(steps):
        _, _, F, Np = collide(N, F)
        N = Np.reshape(-1)[gather]
    r, U, F, _ = collide(N, F)
    ut = torch.einsum("in,nid->nd", U + 0.5 * F / r, gl)
    tot = []
    for o, k in zip(off, nc):
        Nk, s = N[:, o:o + k], slice(int(o), int(o + k))
        e = torch.einsum("ai,nid->and", c, gl[s])
        z = torch.zeros(3 - D, dtype=torch.float64, device="cuda")
        Pm, Mm = torch.einsum("and,an->d", e, Nk), 0.5 * torch.einsum("and,an->d", e + eb[:, s], Nk)
        tot.append(torch.cat([Nk.sum()[None], Pm, z, Mm, z]))
    return r, ut, torch.stack(tot)


def exact(case, seed):
    c = case
    if c["kind"] == "nn":
        return _exact_nn(c, seed)
    if c["kind"] == "batch":
        mem = _batch_members(c, seed)
        nc = sum(W.ncell(m) for m, _ in mem)
        r, ut, tot = _solve([m for m, _ in mem], [p for _, p in mem], *_batch_fields(nc, seed), c["steps"])
        return [r, ut, tot]
    if c["n0"] * c["n1"] * c["n2"] > 1 << 22:
        return None      # over about 20 seconds
    mesh = _mesh(c)
    rho, u = _fields(c, mesh, seed)
    r, ut, tot = _solve([mesh], [_params(c)], rho, u, c["steps"])
    return [r, ut, tot]


def _exact_nn(c, seed):
    import torch.nn.functional as F
    layers, x, t = _nn_inputs(c, seed)
    p = [v.double().requires_grad_(c["what"] == "grad") for l in layers for v in l]

    def conv(h, i, relu=True):
        # the taps as one matrix product each way (cuDNN has no fast 64-bit form)
        k = p[2 * i].shape[-1]
        y = F.unfold(h, k, padding=k // 2).transpose(1, 2) @ p[2 * i].reshape(p[2 * i].shape[0], -1).T + p[2 * i + 1]
        y = y.transpose(1, 2).reshape(h.shape[0], -1, h.shape[2], h.shape[3])
        return F.relu(y) if relu else y

    up = lambda h: F.interpolate(h, scale_factor=2, mode="nearest")  # noqa: E731
    s1 = conv(conv(x.double(), 0), 1)
    s2 = conv(conv(F.avg_pool2d(s1, 2), 2), 3)
    b = conv(conv(F.avg_pool2d(s2, 2), 4), 5)
    t2 = conv(conv(torch.cat([up(b), s2], 1), 6), 7)
    t1 = conv(conv(torch.cat([up(t2), s1], 1), 8), 9)
    y = conv(t1, 10, relu=False)
    if c["what"] == "forward":
        return y
    loss = ((y - t.double()) ** 2).mean()
    loss.backward()
    return {"y": y.detach(), "loss": float(loss.detach()), "grads": torch.cat([v.grad.reshape(-1) for v in p])}
