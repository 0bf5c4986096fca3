"""The work that users of this framework have it do, as cases to be timed.

The wave path through the public entry points: a batch of shots advanced
over a nested simplex mesh (forward traces), the sensitivity of the traces
to the permittivity of a coarse level (J v, J^T w, both beside the traces in
one pass), several problems at once, the flux form with its absorbing layer,
and a whole reconstruction.  Meshes, permittivity fields, shot geometry and
step counts are those of ``workloads.configs`` and of the tests: the square
of 4,225 nodes, the asteroid on refinement levels 1 to 4 (3,997 to 249,697
nodes), the ellipsoid on levels 1 and 2 (30,525 and 232,505 nodes), 1 to 256
shots, a few hundred to a few thousand steps.

Every case is one dict: ``call`` (what is called), ``mesh`` and ``level``
(which mesh), ``shots``, ``steps``, and where they apply ``ckpt``
(checkpoint spacing of J^T), ``tuned`` (the handle autotuned first) and
``instances``.
"""
import functools
import math

import numpy as np
import torch

import paper_1707_04605_gb300 as mg
from paper_1707_04605_gb300.autograd import level_traces
from workloads import configs, fields, meshes, shots as shot_geometry

NODES = {("square", 3): 4225, ("asteroid", 1): 3997, ("asteroid", 2): 15769,
         ("asteroid", 3): 62641, ("asteroid", 4): 249697, ("ellipsoid", 1): 30525,
         ("ellipsoid", 2): 232505}
# fields advanced per step, for the cost of a drawn case
FIELDS = {"forward": 1.0, "tangent": 2.0, "gradient": 3.0, "fused": 3.0, "batch": 1.0,
          "pml_forward": 4.0, "pml_gradient": 14.0, "tv": 60.0}
LARGEST = 249697 * 256 * 256.0


def listed():
    return [
        # one source, 16 receivers, a small mesh: the smallest problem of the
        # configurations, where the latency of a step is all there is
        dict(name="forward_square", call="forward", mesh="square", level=3, shots=1, steps=2000),
        # the backscatter survey of the asteroid with an autotuned handle, as
        # the README's first example runs it
        dict(name="forward_asteroid", call="forward", mesh="asteroid", level=3, shots=128,
             steps=1024, tuned=True),
        # the largest two-dimensional instance of the uneven batch
        dict(name="forward_asteroid_fine", call="forward", mesh="asteroid", level=4, shots=256,
             steps=256),
        # three dimensions: longer rows, states that exceed L2
        dict(name="forward_ellipsoid", call="forward", mesh="ellipsoid", level=2, shots=128,
             steps=256),
        # one tangent column set on a mid-sized mesh, a ragged shot count
        dict(name="tangent_ragged", call="tangent", mesh="asteroid", level=2, shots=37,
             steps=900),
        # least-squares misfit and its gradient through autograd, forward
        # checkpoints every 256 steps: one step of a gradient-based inversion
        dict(name="gradient_asteroid", call="gradient", mesh="asteroid", level=3, shots=128,
             steps=512, ckpt=256),
        # the same on a three-dimensional mesh with few shots
        dict(name="gradient_ellipsoid", call="gradient", mesh="ellipsoid", level=1, shots=24,
             steps=256, ckpt=64),
        # traces and J v in one pass that keeps the forward history, then
        # J^T w on it: the step of the repository's benchmark
        dict(name="fused_asteroid", call="fused", mesh="asteroid", level=3, shots=128, steps=384),
        # independent problems of different sizes advanced together
        dict(name="batch_uneven", call="batch", mesh="asteroid", level=3, shots=64, steps=500,
             instances=6),
        # the flux form with the absorbing layer: traces, and a gradient on a
        # mid-sized mesh at the default checkpoint spacing
        dict(name="pml_forward", call="pml_forward", mesh="asteroid", level=3, shots=128,
             steps=256),
        dict(name="pml_gradient", call="pml_gradient", mesh="asteroid", level=2, shots=32,
             steps=300, ckpt=64),
        # a whole coarse-to-fine reconstruction with total variation: many
        # short J and J^T calls on a small mesh
        dict(name="tv_asteroid", call="tv", mesh="asteroid", level=1, shots=12, steps=300,
             ckpt=64),
    ]


def _padded(shots):
    """Shot columns that are advanced: a power of two from 4 to 128, above it
    a multiple of 128."""
    return max(4, 1 << (shots - 1).bit_length()) if shots <= 128 else -(-shots // 128) * 128


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["forward", "forward", "tangent", "gradient", "fused", "batch",
                       "pml_forward", "pml_gradient", "tv"])
    if call == "tv":
        return dict(call=call, mesh="asteroid", level=1, shots=rng.randint(4, 24),
                    steps=rng.randint(150, 400), ckpt=rng.choice([32, 64, 100]))
    if call == "batch":
        return dict(call=call, mesh="asteroid", level=rng.randint(2, 3),
                    shots=_log_int(rng, 8, 96), steps=rng.randint(200, 600),
                    instances=rng.randint(2, 6))
    mesh = "asteroid" if call.startswith("pml") else rng.choice(
        ["asteroid", "asteroid", "asteroid", "ellipsoid", "square"])
    level = {"asteroid": rng.randint(1, 4 if call == "forward" else 3),
             "ellipsoid": rng.randint(1, 2 if call == "forward" else 1),
             "square": 3}[mesh]
    shots = _log_int(rng, 1, 256)
    if call == "pml_gradient":   # whole or ragged groups of 4, 8, 16, 32 or 64 shots
        shots = 4 * rng.choice([1, 2, 4, 8, 16]) - rng.randint(0, 3)
    if mesh == "square":
        shots = 1
    n = NODES[mesh, level]
    columns = _padded(shots) * (2.0 if mesh == "ellipsoid" else 1.0)
    most = LARGEST / (FIELDS[call] * n * columns)
    if call == "fused":   # the kept history of three states fits the card
        most = min(most, 16e9 / (4.0 * n * columns))
    steps = _log_int(rng, 150, 2000 if mesh == "square" else 1200)
    case = dict(call=call, mesh=mesh, level=level, shots=shots,
                steps=int(max(60, min(steps, most))))
    if call in ("gradient", "pml_gradient"):
        case["ckpt"] = rng.choice([32, 64, 100, 256])
    return case


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=32)
def _geometry(mesh, level, shots, rotation=0.0, scale=1.0):
    """Mesh, shots and centre frequency: the same for every seed."""
    if mesh == "square":
        m = meshes.square_mesh(8, level)
        sh = shot_geometry.square_shots(m, 16)
    elif mesh == "asteroid":
        m = meshes.asteroid_mesh(level, 18, rotation, scale)
        sh = shot_geometry.asteroid_shots(m, shots, rotation, scale)
    else:
        m = meshes.ellipsoid_mesh(level)
        sh = shot_geometry.ellipsoid_shots(m, shots)
    f = shot_geometry.ricker_frequency(m.mean_edge_length(), 8.0 if mesh == "ellipsoid" else 10.0)
    return m, sh, f


def _eps(case, m, seed, instance=0, rotation=0.0, scale=1.0):
    if case["mesh"] == "square":
        r = fields.rng_for(seed + 100)
        return fields.square_disc_eps(m, centre=r.uniform(-0.4, 0.4, 2), radius=0.3)
    if case["mesh"] == "asteroid":
        return fields.asteroid_eps(m, seed + 100, instance, rotation, scale)
    return fields.ellipsoid_eps(m, seed + 100)


def _layer(m, dt):
    """Square absorbing layer over the outer 15% of the half-width."""
    c = np.abs(m.coords[m.cells].mean(axis=1))
    half, vs = float(np.abs(m.coords).max()), 0.25 / dt
    xi = np.where(c.max(axis=1) >= 0.85 * half, vs, 0.0)
    return xi, np.ascontiguousarray(np.where(c >= 0.85 * half, vs, 0.0))


def _instances(case):
    """Levels, shot counts, rotations and scales of a batch, largest first in
    the case's own sizes."""
    r = np.random.default_rng(case["shots"] * 1000 + case["instances"])
    out = [(case["level"], case["shots"], 0.3, 1.0)]
    for _ in range(case["instances"] - 1):
        out.append((int(r.integers(1, case["level"] + 1)),
                    int(max(1, round(case["shots"] * r.uniform(0.15, 1.0)))),
                    float(r.uniform(0, 2 * math.pi)), float(r.uniform(0.75, 1.25))))
    return out


def _noise(case, seed, m, sh):
    """Random parts of the inputs (numpy FP64): direction, weights, data."""
    r = np.random.default_rng([seed, 7])
    v = r.standard_normal(m.n_cells[min(1, m.n_levels - 1)])
    w = r.standard_normal((sh.n_traces, case["steps"])).astype(np.float32)
    return v, w


def _handle(m):
    return mg.mesh_create(m.dim, m.coords, m.cells, m.cell_parent, m.n_cells, m.bnd)


def prepare(case, seed):
    dev = torch.device("cuda")
    cu = lambda x, t=torch.float64: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device=dev)
    st = dict(case=case)
    if case["call"] == "batch":
        st.update(meshes=[], eps=[], shots=[], wav=[], dt=[])
        for i, (level, S, rot, scale) in enumerate(_instances(case)):
            m, sh, f = _geometry("asteroid", level, S, rot, scale)
            h = _handle(m)
            eps = cu(_eps(case, m, seed, i, rot, scale))
            dt = 0.5 * mg.cfl_dt(h, eps)
            st["meshes"].append(h)
            st["eps"].append(eps)
            st["shots"].append(mg.Shots.of(sh))
            st["wav"].append(cu(shot_geometry.ricker(f, dt, case["steps"])))
            st["dt"].append(dt)
        return st
    m, sh, f = _geometry(case["mesh"], case["level"], case["shots"])
    h = _handle(m)
    eps = cu(_eps(case, m, seed))
    dt = 0.5 * mg.cfl_dt(h, eps)
    wav = cu(shot_geometry.ricker(f, dt, case["steps"]))
    v, w = _noise(case, seed, m, sh)
    st.update(mesh=h, eps=eps, shots=mg.Shots.of(sh), wav=wav, dt=dt,
              level=min(1, m.n_levels - 1))
    if case.get("tuned"):
        h.autotune(eps, st["shots"], wav, dt)
    call = case["call"]
    if call in ("tangent", "fused"):
        st["v"] = cu(v)
    if call in ("fused", "pml_gradient"):
        st["w"] = cu(w, torch.float32)
    if call == "gradient":   # recorded data: noise of the size of the traces
        st["obs"] = cu(1e-3 * w, torch.float32)
        st["dc"] = cu(0.01 * v).requires_grad_()
    if call == "tv":
        st["dy"] = cu(1e-3 * w, torch.float32)
    if call.startswith("pml"):
        xi, zeta = _layer(m, dt)
        st.update(xi=cu(xi), zeta=cu(zeta))
    return st


# ---------------------------------------------------------------- the calls
def run(st):
    case, call = st["case"], st["case"]["call"]
    if call == "batch":
        return mg.forward_batch(st["meshes"], st["eps"], st["shots"], st["wav"], st["dt"])
    h, eps, sh, wav, dt, level = (st[k] for k in ("mesh", "eps", "shots", "wav", "dt", "level"))
    if call == "forward":
        return mg.forward(h, eps, sh, wav, dt)
    if call == "tangent":
        return mg.jacobian_apply(h, level, eps, sh, wav, dt, st["v"])
    if call == "gradient":
        st["dc"].grad = None
        y = level_traces(st["dc"], h, level, eps, sh, wav, dt, ckpt_every=case["ckpt"])
        (0.5 * (y - st["obs"]).square().sum()).backward()
        return y.detach(), st["dc"].grad
    if call == "fused":
        y, jv = mg.forward_jacobian_apply(h, level, eps, sh, wav, dt, st["v"], keep_states=True)
        g = mg.jacobian_T_apply(h, level, eps, sh, wav, dt, st["w"], ckpt_every=case["steps"],
                                reuse_checkpoints=True)
        return y, jv, g
    if call == "pml_forward":
        return mg.forward_pml(h, eps, sh, wav, dt, st["xi"], st["zeta"])
    if call == "pml_gradient":
        return mg.jacobian_T_apply_pml(h, level, eps, sh, wav, dt, st["w"], st["xi"], st["zeta"],
                                       ckpt_every=case["ckpt"])
    x, hist = mg.tv_reconstruct(h, 0, eps, sh, wav, dt, st["dy"], level_f=level, alpha=1e-2,
                                beta=1.0, n_outer=2, n_cg=6, ckpt_every=case["ckpt"])
    return x, hist


def work(case):
    """Inputs read once, outputs written once (and the kept history, which
    the caller asks for, written and read once); the multiplications and
    additions of the updates.  The states of the steps are neither."""
    def one(mesh, level, S, rot=0.0, scale=1.0):
        m, sh, _ = _geometry(mesh, level, S, rot, scale)
        n, d = m.coords.shape
        edges = m.cells.shape[0] * 3 / 2 if d == 2 else 1.19 * m.cells.shape[0]
        rows = n + 2.0 * edges                      # stored entries of the stiffness
        io = 8.0 * m.cells.shape[0] + 8.0 * case["steps"] + 4.0 * sh.n_traces * case["steps"]
        return n, m.cells.shape[0], d, sh.n_shots * case["steps"], rows, io

    if case["call"] == "batch":
        parts = [one("asteroid", *i) for i in _instances(case)]
    else:
        parts = [one(case["mesh"], case["level"], case["shots"])]
    b = f = 0.0
    for n, m, d, ss, rows, io in parts:
        step = (2.0 * rows + 5.0 * n) * ss          # one field, all shots and steps
        pml = (2.0 * m * (d + 1) * d * 2 + 4.0 * m * d + 6.0 * n) * ss
        call = case["call"]
        b += io * (2.0 if call in ("tangent", "gradient", "fused", "pml_gradient") else 1.0)
        if call == "fused":
            b += 8.0 * n * ss
        f += {"forward": step, "batch": step, "tangent": 2 * step, "gradient": 2 * step,
              "fused": 3 * step, "pml_forward": pml, "pml_gradient": 2 * pml,
              "tv": step * (1 + 2 * 2 * 2 * 6)}[call]
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- in 64 bits
class _System:
    """Lumped P1 matrices of one mesh in FP64 (torch): stiffness, mass and
    boundary damping as functions of eps."""

    def __init__(self, m, dev):
        self.dev = dev
        t = lambda x, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(x), device=dev).to(dt)
        x, cells = np.asarray(m.coords, np.float64), np.asarray(m.cells, np.int64)
        n, d = x.shape
        E = np.transpose(x[cells[:, 1:]] - x[cells[:, :1]], (0, 2, 1))
        inv = np.linalg.inv(E)
        self.n, self.d, k = n, d, d + 1
        vol = np.abs(np.linalg.det(E)) / math.factorial(d)
        g = np.concatenate([-inv.sum(1, keepdims=True), inv], axis=1)
        self.vol, self.grads, self.cells = t(vol), t(g), t(cells, torch.int64)
        Ke = vol[:, None, None] * np.einsum("eak,ebk->eab", g, g)
        ij = np.stack([np.repeat(cells, k, axis=1).ravel(), np.tile(cells, (1, k)).ravel()])
        self.K = torch.sparse_coo_tensor(t(ij, torch.int64), t(Ke.ravel()), (n, n)).coalesce()
        self.rowabs = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(
            0, self.K.indices()[0], self.K.values().abs())
        self.K = self.K.to_sparse_csr()
        # the cell of each boundary facet
        faces = np.sort(np.concatenate([np.delete(cells, j, 1) for j in range(k)]), 1)
        bnd = np.sort(np.asarray(m.bnd, np.int64), 1)
        key = lambda a: functools.reduce(lambda s, c: s * n + c, a.T)
        kf = key(faces)
        order = np.argsort(kf, kind="stable")
        self.owner = t((order[np.searchsorted(kf[order], key(bnd))]) % len(cells), torch.int64)
        xb = x[bnd]
        area = (np.linalg.norm(xb[:, 1] - xb[:, 0], axis=1) if d == 2 else
                0.5 * np.linalg.norm(np.cross(xb[:, 1] - xb[:, 0], xb[:, 2] - xb[:, 0]), axis=1))
        self.bnd, self.area = t(bnd, torch.int64), t(area)

    def to_nodes(self, per_cell, cells=None):
        """out_i = sum of per_cell over the cells (or facets) of node i."""
        cells = self.cells if cells is None else cells
        out = torch.zeros(self.n, dtype=torch.float64, device=self.dev)
        for a in range(cells.shape[1]):
            out = out.index_add(0, cells[:, a], per_cell)
        return out

    def mass(self, eps):
        return self.to_nodes(eps * self.vol / (self.d + 1))

    def damping(self, eps):
        return self.to_nodes(eps[self.owner].sqrt() * self.area / self.d, self.bnd)

    def damping_along(self, eps, v):
        return self.to_nodes(v[self.owner] / (2 * eps[self.owner].sqrt()) * self.area / self.d,
                             self.bnd)

    def dt(self, eps):
        return float(2.0 / (self.rowabs / self.mass(eps)).max().sqrt())


def _events(sh, dev):
    src = torch.as_tensor(np.asarray(sh.src, np.int64), device=dev)
    rec = torch.as_tensor(np.asarray(sh.rec, np.int64), device=dev)
    shot = torch.as_tensor(np.repeat(np.arange(sh.n_shots), np.diff(sh.rec_ptr)), device=dev)
    return src, rec, shot


def _leapfrog(s, eps, dt, wav, sh, deps=None, keep=False):
    """Traces, their derivative along deps, and all states p_0 .. p_nt."""
    src, rec, shot = _events(sh, s.dev)
    M, D = s.mass(eps), s.damping(eps)
    W, V = (M + dt / 2 * D)[:, None], (M - dt / 2 * D)[:, None]
    M2, cols, nt = 2 * M[:, None], torch.arange(len(src), device=s.dev), len(wav)
    p = torch.zeros((s.n, len(src)), dtype=torch.float64, device=s.dev)
    pm, q, qm = p.clone(), p.clone(), p.clone()
    y = torch.zeros((len(rec), nt), dtype=torch.float64, device=s.dev)
    jy, states = torch.zeros_like(y), [p.clone()] if keep else None
    if deps is not None:
        dM, dD = s.mass(deps)[:, None], s.damping_along(eps, deps)[:, None]
    for l in range(nt):
        r = M2 * p - V * pm - dt * dt * (s.K @ p)
        r[src, cols] += dt * dt * float(wav[l])
        pn = r / W
        if deps is not None:
            qn = (M2 * q - V * qm - dt * dt * (s.K @ q) - dM * (pn - 2 * p + pm) -
                  dt / 2 * dD * (pn - pm)) / W
            jy[:, l] = qn[rec, shot]
            q, qm = qn, q
        y[:, l] = pn[rec, shot]
        p, pm = pn, p
        if keep:
            states.append(p)
    return y, jy, states


def _gradient(s, eps, dt, sh, w, states):
    """Derivative of sum w y with respect to eps of every cell, from the
    transposed recursion over the stored states."""
    src, rec, shot = _events(sh, s.dev)
    M, D = s.mass(eps), s.damping(eps)
    W, V, M2 = (M + dt / 2 * D)[:, None], (M - dt / 2 * D)[:, None], 2 * M[:, None]
    a = torch.zeros_like(states[0])
    b, zero = a.clone(), a
    G = torch.zeros(s.n, dtype=torch.float64, device=s.dev)
    H = G.clone()
    for l in range(w.shape[1] - 1, -1, -1):
        r = M2 * a - V * b - dt * dt * (s.K @ a)
        r.index_put_((rec, shot), w[:, l].double(), accumulate=True)
        lam = r / W
        pm = states[l - 1] if l else zero
        G -= (lam * (states[l + 1] - 2 * states[l] + pm)).sum(1)
        H -= dt / 2 * (lam * (states[l + 1] - pm)).sum(1)
        a, b = lam, a
    g = s.vol / (s.d + 1) * G[s.cells].sum(1)
    f = s.area / s.d * H[s.bnd].sum(1) / (2 * eps[s.owner].sqrt())
    return g.index_add(0, s.owner, f)


def _to_level(m, level, g):
    anc = torch.as_tensor(m.ancestor(level), device=g.device)
    return torch.zeros(m.n_cells[level], dtype=g.dtype, device=g.device).index_add(0, anc, g)


def _flux_traces(s, C, dt, wav, sh, xi, zeta, with_grad):
    """The flux form: differentiable in the lumped mass C."""
    src, rec, shot = _events(sh, s.dev)
    S, nt = len(src), len(wav)
    B = []                                  # per direction: cells x nodes, |e| dphi/dx_k
    e = torch.arange(s.cells.shape[0], device=s.dev).repeat_interleave(s.d + 1)
    for k in range(s.d):
        v = (s.vol[:, None] * s.grads[:, :, k]).reshape(-1)
        B.append(torch.sparse_coo_tensor(torch.stack([e, s.cells.reshape(-1)]), v,
                                         (s.cells.shape[0], s.n)).coalesce())
    BT = [b.t().coalesce().to_sparse_csr() for b in B]
    B = [b.to_sparse_csr() for b in B]
    R = s.mass(xi)[:, None]
    one = torch.zeros((s.n, S), dtype=torch.float64, device=s.dev)
    one[src, torch.arange(S, device=s.dev)] = 1.0
    p = torch.zeros_like(one)
    q = [torch.zeros((len(s.vol), S), dtype=torch.float64, device=s.dev) for _ in range(s.d)]
    y, f, vol, back = [], 0.0, s.vol[:, None], []
    for l in range(nt):
        f += dt * float(wav[l])
        q = [(1 - dt * zeta[:, k, None]) * q[k] + dt * (B[k] @ p) / vol for k in range(s.d)]
        rhs = f * one - R * p - sum(BT[k] @ q[k] for k in range(s.d))
        if with_grad:
            back.append(dt * rhs / C[:, None])      # p_{l+1} - p_l
        p = p + dt * rhs / C[:, None]
        y.append(p[rec, shot])
    return torch.stack(y, 1), back, B, BT, R


def _flux_gradient(s, C, dt, sh, w, xi, zeta, wav):
    src, rec, shot = _events(sh, s.dev)
    _, diff, B, BT, R = _flux_traces(s, C, dt, wav, sh, xi, zeta, True)
    a = torch.zeros_like(diff[0])
    Q = [torch.zeros((len(s.vol), a.shape[1]), dtype=torch.float64, device=s.dev)
         for _ in range(s.d)]
    gC, vol = torch.zeros(s.n, dtype=torch.float64, device=s.dev), s.vol[:, None]
    for l in range(len(wav) - 1, -1, -1):
        a.index_put_((rec, shot), w[:, l].double(), accumulate=True)
        gC -= (a * diff[l]).sum(1) / C
        r = dt * a / C[:, None]
        Q = [Q[k] - B[k] @ r for k in range(s.d)]           # adjoint of q_{l+1/2}
        a = a - R * r + sum(BT[k] @ (dt * Q[k] / vol) for k in range(s.d))
        Q = [(1 - dt * zeta[:, k, None]) * Q[k] for k in range(s.d)]
    return s.vol / (s.d + 1) * gC[s.cells].sum(1)


def exact(case, seed):
    call = case["call"]
    if call == "tv":
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    t = lambda x: torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device=dev)
    if call == "batch":
        out = []
        for i, (level, S, rot, scale) in enumerate(_instances(case)):
            m, sh, f = _geometry("asteroid", level, S, rot, scale)
            s, eps = _System(m, dev), t(_eps(case, m, seed, i, rot, scale))
            dt = 0.5 * s.dt(eps)
            out.append(_leapfrog(s, eps, dt, shot_geometry.ricker(f, dt, case["steps"]), sh)[0])
        return out
    m, sh, f = _geometry(case["mesh"], case["level"], case["shots"])
    if call in ("gradient", "fused", "pml_gradient") and \
            8.0 * len(m.coords) * sh.n_shots * case["steps"] > 60e9:
        return None
    s, eps, level = _System(m, dev), t(_eps(case, m, seed)), min(1, m.n_levels - 1)
    dt = 0.5 * s.dt(eps)
    wav = shot_geometry.ricker(f, dt, case["steps"])
    v, w = _noise(case, seed, m, sh)
    anc = torch.as_tensor(m.ancestor(level), device=dev)
    if call == "forward":
        return _leapfrog(s, eps, dt, wav, sh)[0]
    if call == "tangent":
        return _leapfrog(s, eps, dt, wav, sh, t(v)[anc])[1]
    if call == "gradient":
        eps = eps + t(0.01 * v)[anc]
        y, _, states = _leapfrog(s, eps, dt, wav, sh, keep=True)
        obs = t((1e-3 * w).astype(np.float32))
        return y, _to_level(m, level, _gradient(s, eps, dt, sh, y - obs, states))
    if call == "fused":
        y, jv, states = _leapfrog(s, eps, dt, wav, sh, t(v)[anc], keep=True)
        return y, jv, _to_level(m, level, _gradient(s, eps, dt, sh, t(w), states))
    xi, zeta = (t(x) for x in _layer(m, dt))
    if call == "pml_forward":
        return _flux_traces(s, s.mass(eps), dt, wav, sh, xi, zeta, False)[0]
    return _to_level(m, level, _flux_gradient(s, s.mass(eps), dt, sh, t(w), xi, zeta, wav))
