"""Performance cases of the wedge Stokes library: what a user's program has it do.

Every case goes through the public entry points (paper_2609_21633_gb300, include/terra_wedge.h) on one
mesh of the shell 0.55 <= r <= 1.  Kinds:

  step     A u, B u, B^T p and diag(A) on the finest level: the operator step of bench.py
  apply    A u alone: the smoother's and the Krylov solver's operator
  saddle   B u and B^T p: the off-diagonal blocks of one Krylov iteration
  vcycle   one multigrid V-cycle: the preconditioner of every solve and served request
  energy   Heun substeps of the energy equation with the SUPG term: the other half of a time step
  stokes   one time step's Stokes part: viscosity and load from the temperature, then FGMRES(10) for ten
           iterations (the paper's setting), multigrid set-up included

Options: dtype (f64 | f32), kappa (hourglass control), quad (radial quadrature points), eta (storage of the
FP32 path's viscosity: 0 FP32, 1 BF16), noslip (1: no-slip at r_in, else free-slip on both surfaces).

Velocities and pressures of the operator kinds are N(0, 1) per node, as in bench.py: a Krylov vector holds
every wavelength.  The viscosity is that of bench.py's shell, 30^(r < 0.9) exp(ln(contrast) (1/2 - T)) with T
the conductive profile plus a degree-3 perturbation and nodal noise.
"""
import functools
import math

import torch

import paper_2609_21633_gb300 as tn

R_IN, R_OUT = 0.55, 1.0
JUMP_R, JUMP_F = 0.9, 30.0
DEVICE = "cuda"


# ------------------------------------------------------------------------------------------- cases
def _case(kind, level, n_r, dtype="f64", kappa=0.0, quad=1, eta=0, noslip=0, contrast=1e3, steps=1):
    return dict(kind=kind, level=level, n_r=n_r, dtype=dtype, kappa=kappa, quad=quad, eta=eta, noslip=noslip,
                contrast=contrast, steps=steps)


def listed():
    return [
        # the FP64 operator step of bench.py at its own size: 63.4 M velocity unknowns
        dict(_case("step", 7, 129), name="step_f64_l7_n129"),
        # the smallest FP64 operator apply in use: the convergence configuration at level 4, 17 layers
        dict(_case("apply", 4, 17, contrast=10.0), name="apply_f64_l4_n17"),
        # FP64 operator of the solves with hourglass control, 8.3 M unknowns, viscosity contrast 1e4
        dict(_case("apply", 6, 65, kappa=0.3, contrast=1e4), name="apply_f64_hg_l6_n65"),
        # the smoother's operator of the fast solves on a large shell: FP32, hourglass control, BF16 viscosity
        dict(_case("apply", 7, 129, "f32", kappa=0.3, eta=1), name="apply_f32_hg_bf16_l7_n129"),
        # divergence and gradient of a shell with a ragged number of layers, no-slip at the inner surface
        dict(_case("saddle", 5, 101, noslip=1), name="saddle_f64_l5_n101"),
        # divergence and gradient of the FP32 inner solves
        dict(_case("saddle", 6, 65, "f32"), name="saddle_f32_l6_n65"),
        # preconditioner of a small served request: launches and latency
        dict(_case("vcycle", 4, 17, "f32", kappa=0.3, eta=1), name="vcycle_f32_l4_n17"),
        # preconditioner of the 8.3 M-unknown solve in its fastest setting
        dict(_case("vcycle", 6, 65, "f32", kappa=0.3, eta=1, contrast=1e4), name="vcycle_f32_l6_n65"),
        # the same preconditioner with the second radial quadrature point, the other hourglass remedy
        dict(_case("vcycle", 5, 33, "f32", quad=2, eta=1, contrast=1e4), name="vcycle_f32_q2_l5_n33"),
        # FP64 preconditioner of the plain one-point operator
        dict(_case("vcycle", 5, 33, contrast=1e4), name="vcycle_f64_l5_n33"),
        # energy update of a time step: ten Heun substeps
        dict(_case("energy", 6, 65, steps=10), name="energy_f64_l6_n65"),
        # Stokes part of a time step in FP64, ten FGMRES iterations
        dict(_case("stokes", 5, 33, contrast=100.0, steps=10), name="stokes_f64_l5_n33"),
    ]


def draw(rng):
    kind = rng.choice(["step", "apply", "apply", "apply", "saddle", "saddle", "vcycle", "vcycle", "energy", "stokes"])
    contrast = round(10.0 ** rng.uniform(1.0, 4.0), 2)
    noslip = int(rng.random() < 0.2)
    if kind in ("step", "apply", "saddle"):  # levels 3 to 7, 9 to 129 layers, over the logarithm of the size
        level = rng.choice([3, 4, 5, 6, 7])
        n_r = 2 * int(round(4 * 16 ** rng.random())) + 1
        dtype = rng.choice(["f64", "f32"])
        kappa = rng.choice([0.0, 0.3]) if kind != "saddle" and (kind, level) != ("step", 7) else 0.0
        eta = rng.choice([0, 1]) if dtype == "f32" and kind != "saddle" and level >= 4 else 0
        return _case(kind, level, n_r, dtype, kappa, 1, eta, noslip, contrast)
    if kind == "vcycle":
        level = rng.choice([3, 4, 5, 6])
        n_r = 8 * int(round(8 ** rng.random())) + 1
        dtype = rng.choice(["f32", "f32", "f64"])
        kappa, quad = rng.choice([(0.3, 1), (0.3, 1), (0.0, 2), (0.0, 1)])
        eta = rng.choice([0, 1]) if dtype == "f32" else 0
        return _case(kind, level, n_r, dtype, kappa, quad, eta, noslip, contrast)
    if kind == "energy":
        return _case(kind, rng.choice([3, 4, 5, 6]), 2 * int(round(4 * 8 ** rng.random())) + 1, steps=rng.choice([3, 5, 10]))
    return _case(kind, rng.choice([3, 4, 5]), rng.choice([9, 17, 25, 33]), noslip=noslip,
                 contrast=round(10.0 ** rng.uniform(1.0, 2.0), 2), steps=10)


# ------------------------------------------------------------------------------------------- lattice
def _normsum(p, q):
    v = p + q
    x, y, z = v[..., 0], v[..., 1], v[..., 2]
    xx, yy, zz = x * x, y * y, z * z
    s = xx + yy
    s = s + zz
    return v / torch.sqrt(s)[..., None]


@functools.lru_cache(maxsize=None)
def _lattice(level):
    """(points (n_lat, 3), id (10, N+1, N+1)): unit-sphere lattice points of the ten diamonds, copies of one
    point on several diamonds under one id (the mesh of include/terra_wedge.h)."""
    n, lat = 1 << level, math.atan(0.5)
    up = [(math.cos(lat) * math.cos(2 * math.pi * k / 5), math.cos(lat) * math.sin(2 * math.pi * k / 5), math.sin(lat))
          for k in range(5)]
    lo = [(math.cos(lat) * math.cos(math.pi / 5 + 2 * math.pi * k / 5),
           math.cos(lat) * math.sin(math.pi / 5 + 2 * math.pi * k / 5), -math.sin(lat)) for k in range(5)]
    north, south = (0.0, 0.0, 1.0), (0.0, 0.0, -1.0)
    corners = [(north, up[k], up[(k + 1) % 5], lo[k]) for k in range(5)]
    corners += [(up[(k + 1) % 5], lo[k], lo[(k + 1) % 5], south) for k in range(5)]
    c = torch.tensor(corners, dtype=torch.float64)
    p = torch.zeros((10, n + 1, n + 1, 3), dtype=torch.float64)
    p[:, 0, 0], p[:, n, 0], p[:, 0, n], p[:, n, n] = c[:, 0], c[:, 1], c[:, 2], c[:, 3]
    s = n
    while s > 1:
        h = s // 2
        p[:, h::s, 0::s] = _normsum(p[:, 0:n:s, 0::s], p[:, s::s, 0::s])
        p[:, 0::s, h::s] = _normsum(p[:, 0::s, 0:n:s], p[:, 0::s, s::s])
        p[:, h::s, h::s] = _normsum(p[:, s::s, 0:n:s], p[:, 0:n:s, s::s])
        s = h
    flat = p.reshape(-1, 3).to(DEVICE)
    grid = torch.round((flat + 1.5) * 2.0 ** 19).to(torch.int64)  # far finer than the lattice; copies are bitwise equal
    _, ids = torch.unique((grid[:, 0] << 42) + (grid[:, 1] << 21) + grid[:, 2], return_inverse=True)
    n_lat = 10 * 4 ** level + 2
    assert int(ids.max()) + 1 == n_lat
    pts = torch.empty((n_lat, 3), dtype=torch.float64, device=DEVICE)
    pts[ids] = flat
    return pts, ids.reshape(10, n + 1, n + 1)


def _radii(n_r):
    return R_IN + ((R_OUT - R_IN) * torch.arange(n_r, dtype=torch.float64, device=DEVICE)) / (n_r - 1)


@functools.lru_cache(maxsize=None)
def _triangles(level):
    """Point ids (10, N, N, 2, 3) of the two lateral triangles of every cell, in the wedge layout's order."""
    ids = _lattice(level)[1]
    a, b, c, d = ids[:, :-1, :-1], ids[:, 1:, :-1], ids[:, :-1, 1:], ids[:, 1:, 1:]
    return torch.stack([torch.stack([a, b, c], -1), torch.stack([d, c, b], -1)], -2)


def _to_layout(v, level):
    """(n_r, n_lat) values -> the node layout (padding 0)."""
    ids = _lattice(level)[1]
    m = (1 << level) + 1
    pitch = (m + 3) // 4 * 4
    out = torch.zeros((10, v.shape[0], m, pitch), dtype=v.dtype, device=v.device)
    for d in range(10):
        out[d, :, :, :m] = v[:, ids[d].reshape(-1)].reshape(-1, m, m)
    return out.reshape(-1)


# ------------------------------------------------------------------------------------------- inputs
def _gen(seed, which):
    g = torch.Generator(device=DEVICE)
    g.manual_seed((seed * 1000003 + which) % (1 << 62))
    return g


def _normal(seed, which, n_r, level):
    n_lat = 10 * 4 ** level + 2
    return torch.randn((n_r, n_lat), generator=_gen(seed, which), dtype=torch.float64, device=DEVICE)


def _temperature(case, seed, noise=0.01):
    """T (n_r, n_lat): conductive profile, a degree-3 order-2 perturbation of random amplitude and phase, noise
    inside the shell."""
    level, n_r = case["level"], case["n_r"]
    s, r = _lattice(level)[0], _radii(n_r)[:, None]
    a = torch.rand(2, generator=_gen(seed, 1), dtype=torch.float64, device=DEVICE)
    ang = torch.cos(2 * torch.atan2(s[:, 1], s[:, 0]) + 2 * math.pi * a[1]) * 15 * s[:, 2] * (1 - s[:, 2] ** 2)
    shape = torch.sin(math.pi * (r - R_IN) / (R_OUT - R_IN))
    t = R_IN * (r - R_OUT) / (r * (R_IN - R_OUT)) + (0.01 + 0.02 * a[0]) * ang[None] * shape
    if noise:
        t[1:-1] += noise * _normal(seed, 2, n_r, level)[1:-1]
    return t


def _viscosity(case, seed):
    """One value per wedge in the wedge layout."""
    level, n_r = case["level"], case["n_r"]
    t, tri = _temperature(case, seed), _triangles(level)
    lat = torch.stack([t[k][tri].sum(-1) for k in range(n_r)])  # (n_r, 10, N, N, 2)
    e = torch.exp(math.log(case["contrast"]) * (0.5 - (lat[:-1] + lat[1:]) / 6.0))
    r = _radii(n_r)
    e *= torch.where(0.5 * (r[:-1] + r[1:]) < JUMP_R, JUMP_F, 1.0).to(e)[:, None, None, None, None]
    return e.permute(1, 0, 2, 3, 4).contiguous().reshape(-1)


def _flow(case, seed):
    """Smooth velocity (3 x (n_r, n_lat)) of an overturning cell pattern, |u| about 100 (an advective Peclet
    number of order 1 per cell)."""
    level, n_r = case["level"], case["n_r"]
    s, r = _lattice(level)[0], _radii(n_r)[:, None]
    a = 2 * math.pi * torch.rand(3, generator=_gen(seed, 3), dtype=torch.float64, device=DEVICE)
    shape = torch.sin(math.pi * (r - R_IN) / (R_OUT - R_IN))
    return [100.0 * (shape * torch.sin(3 * s[:, c] + a[c])[None] + 0.3 * torch.cos(4 * s[:, (c + 1) % 3] + a[c])[None])
            for c in range(3)]


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


class _State:
    """A mesh with its inputs and output buffers; the mesh is freed with the object."""

    def __init__(self, case):
        self.case = case
        self.mesh = tn.tn_mesh_create(case["level"], case["n_r"], R_IN, R_OUT, case["noslip"], 0,
                                      eta_storage=case["eta"], hg_kappa=case["kappa"], radial_quad_points=case["quad"])
        self.n0 = tn.tn_mesh_info(self.mesh, 0)["n_layout"]
        self.n1 = tn.tn_mesh_info(self.mesh, 1)["n_layout"]

    def zeros(self, n, count=None, dtype=None):
        dtype = dtype or _dtype(self.case)
        if count is None:
            return torch.zeros(n, dtype=dtype, device=DEVICE)
        return [torch.zeros(n, dtype=dtype, device=DEVICE) for _ in range(count)]

    def __del__(self):
        mesh, self.mesh = getattr(self, "mesh", None), None
        if mesh is not None:
            torch.cuda.synchronize()
            tn.tn_mesh_destroy(mesh)


def prepare(case, seed):
    case = dict(case)
    level, n_r, kind = case["level"], case["n_r"], case["kind"]
    st = _State(case)
    if kind in ("step", "apply", "saddle"):
        if kind != "saddle":
            tn.tn_set_viscosity(st.mesh, _viscosity(case, seed))
        st.u = [_to_layout(_normal(seed, 10 + c, n_r, level).to(_dtype(case)), level) for c in range(3)]
        if kind != "apply":
            st.p = _to_layout(_normal(seed, 20, (n_r - 1) // 2 + 1, level - 1).to(_dtype(case)), level - 1)
            st.q, st.g = st.zeros(st.n1), st.zeros(st.n0, 3)
        if kind != "saddle":
            st.y = st.zeros(st.n0, 3)
        if kind == "step":
            st.d = st.zeros(st.n0, 3)
    elif kind == "vcycle":
        T = _to_layout(_temperature(case, seed), level)
        tn.tn_set_temperature(st.mesh, T, math.log(case["contrast"]), JUMP_R, JUMP_F)
        tn.tn_mg_setup(st.mesh, _dtype(case))
        st.r = [_to_layout(_normal(seed, 10 + c, n_r, level).to(_dtype(case)), level) for c in range(3)]
        st.z = st.zeros(st.n0, 3)
    elif kind == "energy":
        st.T0 = _to_layout(_temperature(case, seed), level)
        st.u = [_to_layout(v, level) for v in _flow(case, seed)]
        st.T = torch.zeros_like(st.T0)
        st.dt = _substep(case)
    else:
        st.T = _to_layout(_temperature(case, seed), level)
        st.f, st.u, st.p = st.zeros(st.n0, 3), st.zeros(st.n0, 3), st.zeros(st.n1)
        st.opts = tn.tn_solve_default_opts(mode=tn.TN_SOLVE_F64, restart=10, max_iters=case["steps"])
    return st


def _substep(case):
    """A stable Heun substep: a fixed share of the squared smallest cell edge."""
    h = min((R_OUT - R_IN) / (case["n_r"] - 1), 0.9 * R_IN / (1 << case["level"]))
    return 0.04 * h * h


def run(st):
    case, kind = st.case, st.case["kind"]
    if kind == "step":
        tn.tn_apply_A(st.mesh, 0, st.u, st.y)
        tn.tn_apply_B(st.mesh, 0, st.u, st.q)
        tn.tn_apply_BT(st.mesh, 0, st.p, st.g)
        tn.tn_diag_A(st.mesh, 0, st.d)
        return {"A": st.y, "B": st.q, "BT": st.g, "diag": st.d}
    if kind == "apply":
        tn.tn_apply_A(st.mesh, 0, st.u, st.y)
        return {"A": st.y}
    if kind == "saddle":
        tn.tn_apply_B(st.mesh, 0, st.u, st.q)
        tn.tn_apply_BT(st.mesh, 0, st.p, st.g)
        return {"B": st.q, "BT": st.g}
    if kind == "vcycle":
        tn.tn_vcycle(st.mesh, st.r, st.z)
        return {"z": st.z}
    if kind == "energy":
        st.T.copy_(st.T0)
        tn.tn_energy_steps(st.mesh, st.T, st.u, st.dt, case["steps"])
        return {"T": st.T}
    tn.tn_set_temperature(st.mesh, st.T, math.log(case["contrast"]))
    tn.tn_buoyancy(st.mesh, st.T, 7e3, st.f)
    tn.tn_stokes_solve(st.mesh, st.f, None, st.u, st.p, st.opts, check=False)
    return {"u": st.u, "p": st.p}


# ------------------------------------------------------------------------------------------- work
def work(case):
    """Bytes and operations of one pass at the least: every input read and every output written once; the
    element arithmetic of both wedges of a cell (FMA = 2)."""
    level, n_r, kind = case["level"], case["n_r"], case["kind"]
    word = 8 if case["dtype"] == "f64" else 4
    nodes = (10 * 4 ** level + 2) * n_r
    cells = 10 * 4 ** level * (n_r - 1)
    pnodes = (10 * 4 ** (level - 1) + 2) * ((n_r - 1) // 2 + 1)
    eta = 2 * cells * (word if not case["eta"] else 2)
    flops_a = 480 if case["quad"] == 1 and not case["kappa"] else 620 if case["quad"] == 1 else 840
    a_bytes, a_flops = 6 * nodes * word + eta, flops_a * cells
    b_bytes, b_flops = (3 * nodes + pnodes) * word, 80 * cells
    d_bytes, d_flops = 3 * nodes * word + eta, 130 * cells
    if kind == "apply":
        return {"bytes": a_bytes, "flops": a_flops}
    if kind == "saddle":
        return {"bytes": 2 * b_bytes, "flops": 2 * b_flops}
    if kind == "step":
        return {"bytes": a_bytes + 2 * b_bytes + d_bytes, "flops": a_flops + 2 * b_flops + d_flops}
    # the finest level's eight operator applications and its updates (node blocks: six words), coarser levels 1/7
    v_bytes, v_flops = 6 * nodes * word + eta + 6 * nodes * word, 8 * a_flops * 8 / 7
    if kind == "vcycle":
        return {"bytes": v_bytes, "flops": v_flops}
    if kind == "energy":
        return {"bytes": 5 * nodes * 8, "flops": 2 * case["steps"] * 200 * cells}
    it = case["steps"]
    return {"bytes": nodes * 8 + (3 * nodes + pnodes) * 8, "flops": it * (v_flops + a_flops + 3 * b_flops)}


# ------------------------------------------------------------------------------------------- exact
def _unit_wedges(level):
    """Per lateral triangle: ids (n, 3), rows of M^-1 (n, 3, 3) and |det M|, M = [s1 - s0, s2 - s0, mean s]."""
    s = _lattice(level)[0]
    tri = _triangles(level).reshape(-1, 3)
    s0, s1, s2 = s[tri[:, 0]], s[tri[:, 1]], s[tri[:, 2]]
    a, b, c = s1 - s0, s2 - s0, (s0 + s1 + s2) / 3.0
    det = (a * torch.linalg.cross(b, c)).sum(-1)
    inv = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], 1) / det[:, None, None]
    return tri, inv, det.abs()


def _gradients(inv, rho, h, zeta=0.0):
    """grad N_j (n, 6, 3) at the lateral barycentre and radial coordinate zeta of the wedges between the radii
    rho -/+ h; nodes: three at the bottom, three at the top."""
    lat = torch.stack([-(inv[:, 0] + inv[:, 1]), inv[:, 0], inv[:, 1]], 1) / (rho + zeta * h)
    rad = (inv[:, 2] / (3.0 * 2.0 * h))[:, None, :]
    return torch.cat([lat * (0.5 * (1 - zeta)) - rad, lat * (0.5 * (1 + zeta)) + rad], 1)


class _Exact:
    """The operators in 64 bits on unique nodes: fields (n_r, n_lat, ...), one cell layer at a time."""

    def __init__(self, case, seed):
        self.case, self.level, self.n_r = case, case["level"], case["n_r"]
        self.tri, self.inv, self.det = _unit_wedges(self.level)
        self.s, self.r = _lattice(self.level)[0], _radii(self.n_r)
        self.eta = None
        if case["kind"] in ("step", "apply"):
            e = _viscosity(case, seed).reshape(10, self.n_r - 1, -1).permute(1, 0, 2).reshape(self.n_r - 1, -1)
            if case["dtype"] == "f32":
                if case["eta"]:  # stored as 16-bit values over one FP32 factor per radial column
                    c = torch.sqrt(e.amin(0) * e.amax(0)).float().double()
                    e = (e / c).float().bfloat16().double() * c
                else:
                    e = e.float().double()
            self.eta = e

    def layer(self, k):
        rho, h = float(self.r[k] + self.r[k + 1]) / 2, float(self.r[k + 1] - self.r[k]) / 2
        return rho, h, rho * rho * h * self.det

    def project(self, u):
        """Boundary projector on a velocity (n_r, n_lat, 3): free-slip, or no-slip at r_in."""
        u = u.clone()
        for k in (0, self.n_r - 1):
            if k == 0 and self.case["noslip"]:
                u[k] = 0
            else:
                u[k] -= (u[k] * self.s).sum(-1, keepdim=True) * self.s
        return u

    def add(self, y, k, v):
        """v (n_tri, 6, ...): contributions to the six nodes of the wedges of cell layer k."""
        ids = self.tri.reshape(-1)
        y[k].index_add_(0, ids, v[:, :3].reshape((-1,) + v.shape[2:]))
        y[k + 1].index_add_(0, ids, v[:, 3:].reshape((-1,) + v.shape[2:]))

    def nodes(self, f, k):
        return torch.cat([f[k][self.tri], f[k + 1][self.tri]], 1)

    def apply_A(self, u):
        case, pu = self.case, self.project(u)
        y = torch.zeros_like(u)
        eye = torch.eye(3, dtype=u.dtype, device=u.device)
        for k in range(self.n_r - 1):
            rho, h, _ = self.layer(k)
            ue = self.nodes(pu, k)
            ye = 0
            for zeta, wgt in ([(0.0, 1.0)] if case["quad"] == 1 else [(-1 / math.sqrt(3), 0.5), (1 / math.sqrt(3), 0.5)]):
                g = _gradients(self.inv, rho, h, zeta)
                v = wgt * (rho + zeta * h) ** 2 * h * self.det * self.eta[k]
                du = ue.transpose(1, 2) @ g
                s = du + du.transpose(1, 2) - (2.0 / 3.0) * (du[:, 0, 0] + du[:, 1, 1] + du[:, 2, 2])[:, None, None] * eye
                ye = ye + g @ (v[:, None, None] * s)
            if case["kappa"]:
                w = torch.tensor([[1., -2, 1, -1, 2, -1], [1., 1, -2, -1, -1, 2]], dtype=u.dtype, device=u.device) / 3.0
                xs = self.s[self.tri]
                x = torch.cat([float(self.r[k]) * xs, float(self.r[k + 1]) * xs], 1)
                gm = w[None] - (w @ x) @ g.transpose(1, 2)
                eps = case["kappa"] / 18.0 * (3.0 + 1.0 / 3.0) * v * (g * g).sum((1, 2))
                ye = ye + eps[:, None, None] * (gm.transpose(1, 2) @ (gm @ ue))
            self.add(y, k, ye)
        return self.project(y) + (u - pu)

    def diag_A(self):
        """diag(P A P + I - P) from the node blocks sum V eta (|g|^2 I + g g^T / 3) and the hourglass terms."""
        case = self.case
        n_lat = self.s.shape[0]
        blk = torch.zeros((self.n_r, n_lat, 6), dtype=torch.float64, device=DEVICE)
        for k in range(self.n_r - 1):
            rho, h, vol = self.layer(k)
            g = _gradients(self.inv, rho, h)
            v = (vol * self.eta[k])[:, None, None]
            sq = (g * g).sum(-1, keepdim=True)
            off = torch.stack([g[..., 0] * g[..., 1], g[..., 0] * g[..., 2], g[..., 1] * g[..., 2]], -1) / 3.0
            dia = sq + g * g / 3.0
            out = v * torch.cat([dia, off], -1)
            if case["kappa"]:
                w = torch.tensor([[1., -2, 1, -1, 2, -1], [1., 1, -2, -1, -1, 2]], dtype=g.dtype, device=g.device) / 3.0
                xs = self.s[self.tri]
                x = torch.cat([float(self.r[k]) * xs, float(self.r[k + 1]) * xs], 1)
                gm = w[None] - (w @ x) @ g.transpose(1, 2)
                eps = case["kappa"] / 18.0 * (3.0 + 1.0 / 3.0) * vol * self.eta[k] * sq.sum((1, 2))
                out[..., :3] += (eps[:, None] * (gm * gm).sum(1))[..., None]
            self.add(blk, k, out)
        d = blk[..., :3].clone()
        for k in (0, self.n_r - 1):
            if k == 0 and case["noslip"]:
                d[k] = 1.0
                continue
            b, s = blk[k], self.s
            full = torch.stack([b[:, 0], b[:, 3], b[:, 4], b[:, 3], b[:, 1], b[:, 5], b[:, 4], b[:, 5], b[:, 2]], -1).reshape(-1, 3, 3)
            p = torch.eye(3, dtype=s.dtype, device=s.device) - s[:, :, None] * s[:, None, :]
            d[k] = torch.diagonal(p @ full @ p, dim1=1, dim2=2) + s * s
        return d

    def parents(self):
        """Coarse lateral ids (n_lat, 2) whose mean is the nested interpolation at a fine lateral point."""
        fine, coarse = _lattice(self.level)[1], _lattice(self.level - 1)[1]
        n = 1 << self.level
        i, j = torch.meshgrid(torch.arange(n + 1, device=DEVICE), torch.arange(n + 1, device=DEVICE), indexing="ij")
        oi, oj = i & 1, j & 1
        i0, j0 = (i + oi * (2 * oj - 1)) // 2, (j - oj) // 2
        i1, j1 = (i + oi * (1 - 2 * oj)) // 2, (j + oj) // 2
        out = torch.empty((self.s.shape[0], 2), dtype=torch.int64, device=DEVICE)
        out[fine.reshape(-1)] = torch.stack([coarse[:, i0, j0].reshape(-1), coarse[:, i1, j1].reshape(-1)], -1)
        return out

    def apply_B(self, u):
        pu = self.project(u)
        q = torch.zeros(u.shape[:2], dtype=u.dtype, device=u.device)
        for k in range(self.n_r - 1):
            rho, h, vol = self.layer(k)
            div = (self.nodes(pu, k) * _gradients(self.inv, rho, h)).sum((1, 2))
            self.add(q, k, (-vol * div / 6.0)[:, None].expand(-1, 6))
        rad = q[0::2].clone()  # radial, then lateral transpose of the nested interpolation
        rad[:-1] += 0.5 * q[1::2]
        rad[1:] += 0.5 * q[1::2]
        par = self.parents()
        out = torch.zeros((rad.shape[0], 10 * 4 ** (self.level - 1) + 2), dtype=u.dtype, device=u.device)
        out.index_add_(1, par[:, 0], 0.5 * rad)
        out.index_add_(1, par[:, 1], 0.5 * rad)
        return out

    def apply_BT(self, p):
        par = self.parents()
        lat = 0.5 * (p[:, par[:, 0]] + p[:, par[:, 1]])
        f = torch.empty((self.n_r, lat.shape[1]), dtype=p.dtype, device=p.device)
        f[0::2] = lat
        f[1::2] = 0.5 * (lat[:-1] + lat[1:])
        y = torch.zeros(f.shape + (3,), dtype=p.dtype, device=p.device)
        for k in range(self.n_r - 1):
            rho, h, vol = self.layer(k)
            pc = self.nodes(f, k).sum(1) / 6.0
            self.add(y, k, (-vol * pc)[:, None, None] * _gradients(self.inv, rho, h))
        return self.project(y)

    def energy(self, T, u, dt, steps):
        m = torch.zeros_like(T)
        for k in range(self.n_r - 1):
            self.add(m, k, (self.layer(k)[2] / 6.0)[:, None].expand(-1, 6))

        def residual(t):
            R = torch.zeros_like(t)
            for k in range(self.n_r - 1):
                rho, h, vol = self.layer(k)
                g = _gradients(self.inv, rho, h)
                gt = (self.nodes(t, k)[..., None] * g).sum(1)
                ub = self.nodes(u, k).sum(1) / 6.0
                adv = (ub * gt).sum(-1)
                un, hh = torch.linalg.norm(ub, dim=1), (2 * vol) ** (1.0 / 3.0)
                pe = un * hh / 2
                big = pe > 1e-3
                pb, ubig = torch.where(big, pe, 1.0), torch.where(big, un, 1.0)
                tau = torch.where(big, hh / (2 * ubig) * (1 / torch.tanh(pb) - 1 / pb), hh ** 2 / 12 * (1 - pe ** 2 / 15))
                flux = gt + (tau * adv)[:, None] * ub
                self.add(R, k, vol[:, None] * ((g * flux[:, None, :]).sum(-1) + adv[:, None] / 6.0))
            return R

        for _ in range(steps):
            a = dt * residual(T) / m
            t1 = T - a
            t1[0], t1[-1] = T[0], T[-1]
            b = 0.5 * ((T + t1) - dt * residual(t1) / m)
            b[0], b[-1] = T[0], T[-1]
            T = b
        return T


def exact(case, seed):
    kind, level, n_r = case["kind"], case["level"], case["n_r"]
    if kind in ("vcycle", "stokes"):
        return None
    ex = _Exact(case, seed)

    def vec(y):
        return [_to_layout(y[..., c].contiguous(), level) for c in range(3)]

    if kind == "energy":
        u = torch.stack(_flow(case, seed), -1)
        return {"T": _to_layout(ex.energy(_temperature(case, seed), u, _substep(case), case["steps"]), level)}
    u = torch.stack([_normal(seed, 10 + c, n_r, level).to(_dtype(case)).double() for c in range(3)], -1)
    out = {}
    if kind in ("step", "apply"):
        out["A"] = vec(ex.apply_A(u))
    if kind in ("step", "saddle"):
        p = _normal(seed, 20, (n_r - 1) // 2 + 1, level - 1).to(_dtype(case)).double()
        out["B"] = _to_layout(ex.apply_B(u), level - 1)
        out["BT"] = vec(ex.apply_BT(p))
    if kind == "step":
        out["diag"] = vec(ex.diag_A())
    return out
