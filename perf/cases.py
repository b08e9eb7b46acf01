"""What the library is timed on: solves and monitoring as a user's program
runs them, through the public entry points of paper_1503_03337_gb300.lbm.

A pass of a solve queues a run of fused steps and hands back the updated
populations (the domain's own buffer, canonical layout because every pass has
an even number of steps).  `exact` is the same flow in 64-bit torch: its own
velocity sets, moment matrix, boundary links and extrapolation faces.
"""
import math
import weakref

import numpy as np
import torch

from paper_1503_03337_gb300 import lbm

PERIODIC, WALL, LID, SYMMETRY, NEQ_U, NEQ_P = range(6)
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
FLOPS = {14: 200, 18: 270, 26: 620}  # of one cell update
DUCT_K = 0.2946854131  # centre velocity of a square duct: u = K F a^2 / nu


# ---- the cases ---------------------------------------------------------------

def listed():
    return [
        # the duct validation run: small, FP64 storage, thousands of steps from rest
        dict(name="duct_16x16x32_q18_f64", flow="duct", Q=18, nx=16, ny=16, nz=32, storage="f64",
             sr=0, steps=200),
        # a small request of the serving loop, odd side, one check interval
        dict(name="cavity_33_q14_f32", flow="cavity", Q=14, nx=33, ny=33, nz=33, storage="f32",
             sr=0, steps=100),
        # oscillating channel, reduced-precision storage with unbiased rounding
        dict(name="pulsatile_64x64x8_q18_f16sr", flow="pulsatile", Q=18, nx=64, ny=64, nz=8,
             storage="f16", sr=1, steps=200),
        # pressure-driven duct with nodes on the walls (spacing 1/32), FP64
        dict(name="pressure_duct_65x33x33_q14_f64", flow="pressure_duct", Q=14, nx=65, ny=33,
             nz=33, storage="f64", sr=0, steps=100),
        # half cavity on the 97-node grid: symmetry plane, lid corner velocities, odd rows
        dict(name="half_cavity_97x97x49_q18_f32", flow="half_cavity", Q=18, nx=97, ny=97, nz=49,
             storage="f32", sr=0, steps=100),
        # the benchmark's cavity: 1000 steps between convergence checks
        dict(name="cavity_128_q18_f32", flow="cavity", Q=18, nx=128, ny=128, nz=128,
             storage="f32", sr=0, steps=1000),
        # a large cavity, FP16 storage rounded to nearest
        dict(name="cavity_256_q18_f16", flow="cavity", Q=18, nx=256, ny=256, nz=256,
             storage="f16", sr=0, steps=100),
        # a large duct as the serving loop stores it at loose tolerance
        dict(name="duct_250x250x62_q14_f16sr", flow="duct", Q=14, nx=250, ny=250, nz=62,
             storage="f16", sr=1, steps=100),
        # porous medium: random spheres, 30 % solid nodes
        dict(name="porous_192_q18_f32", flow="porous", Q=18, nx=192, ny=192, nz=192,
             storage="f32", sr=0, steps=50),
        # the 26-velocity model
        dict(name="cavity_160_q26_f32", flow="cavity", Q=26, nx=160, ny=160, nz=160,
             storage="f32", sr=0, steps=50),
        # uneven cavities and ducts stepped together, one check interval
        dict(name="batch_24_domains", flow="batch", domains=24, mix=0, lmin=24, lmax=160,
             steps=100),
        # restart from a checkpoint and monitor: restore, statistics, fields, a few steps, residual
        dict(name="monitor_160_q18_f32", flow="monitor", Q=18, nx=160, ny=160, nz=160,
             storage="f32", sr=0, steps=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    flow = rng.choice(["cavity", "cavity", "cavity", "duct", "duct", "pulsatile", "half_cavity",
                       "pressure_duct", "porous", "batch", "monitor"])
    if flow == "batch":
        return dict(flow="batch", domains=rng.randint(8, 24), mix=rng.randint(1, 10 ** 6),
                    lmin=24, lmax=rng.randint(60, 160), steps=2 * rng.randint(20, 50))
    Q = rng.choice([14, 18])
    storage, sr = rng.choice([("f32", 0), ("f32", 0), ("f16", 0), ("f16", 1), ("bf16", 1)])
    if flow == "cavity":
        nx = _log(rng, 24, 256)
        ny, nz = nx, nx
        if rng.random() < 0.3:  # a box that is not a cube
            ny, nz = (max(8, int(nx * rng.uniform(0.5, 1.0))) for _ in range(2))
        if rng.random() < 0.2 and nx <= 192:
            Q, storage, sr = 26, rng.choice(["f32", "f16"]), 0
    elif flow == "duct":
        nx = _log(rng, 16, 256)
        ny, nz = nx, max(4, nx // 4)
        if nx <= 48 and rng.random() < 0.5:
            storage, sr = "f64", 0
    elif flow == "pulsatile":
        nx = _log(rng, 32, 256)
        ny, nz = nx, max(4, nx // 4) if rng.random() < 0.5 else 8
    elif flow == "half_cavity":
        nx = _log(rng, 25, 129)
        ny, nz = nx, (nx + 1) // 2
        storage, sr = rng.choice([("f32", 0), ("f16", 1)])
    elif flow == "pressure_duct":
        k = rng.randint(6, 40)
        nx, ny, nz = 2 * k + 1, k + 1, k + 1
        storage, sr = rng.choice([("f64", 0), ("f32", 0)])
    elif flow == "porous":
        nx = ny = nz = _log(rng, 64, 192)
        storage, sr = rng.choice([("f32", 0), ("f16", 1)])
    else:
        nx = ny = nz = _log(rng, 32, 160)
        storage, sr = rng.choice([("f32", 0), ("f16", 0)])
    cells = nx * ny * nz
    most = max(20, min(400, int(1.5e9 / cells)))
    steps = 10 if flow == "monitor" else 2 * rng.randint(10, most // 2)
    return dict(flow=flow, Q=Q, nx=nx, ny=ny, nz=nz, storage=storage, sr=sr, steps=steps)


def work(case):
    """State in and state out once; the arithmetic of every update."""
    if case["flow"] == "batch":
        ds = _domains(case)
        return {"bytes": sum(2 * d["Q"] * BYTES[d["storage"]] * _cells(d) + 12 * _cells(d)
                             for d in ds),
                "flops": sum(FLOPS[d["Q"]] * _cells(d) * case["steps"] for d in ds)}
    N, v = _cells(case), case["Q"] * BYTES[case["storage"]]
    moved = 2 * v * N
    if case["flow"] == "porous":
        moved += N
    if case["flow"] == "monitor":  # 64-bit populations in, u and p out, state written and read
        moved = case["Q"] * 8 * N + 32 * N + 2 * v * N
    return {"bytes": moved, "flops": FLOPS[case["Q"]] * N * case["steps"]}


def _cells(d):
    return d["nx"] * d["ny"] * d["nz"]


# ---- flows -------------------------------------------------------------------

def _setup(case):
    """Faces, wall velocities, viscosity, force and pressures of a flow."""
    nx, ny, nz, flow = case["nx"], case["ny"], case["nz"], case["flow"]
    s = dict(faces=[WALL] * 6, uw=np.zeros((6, 3)), nu=0.05, force=(0.0, 0.0, 0.0), period=0.0,
             edge=None, p_face=[0.0] * 6, p_ref=0.0, U=0.02)
    if flow in ("cavity", "half_cavity", "monitor"):
        s["faces"][3] = LID
        s["U"] = 0.05
        s["uw"][3] = (0.05, 0.0, 0.0)
        s["nu"] = 0.05 * nx / case.get("Re", 400.0)
        if flow == "half_cavity":
            s["faces"][5] = SYMMETRY
            s["edge"] = {3: (0, 0.3, 1.0)}
    elif flow == "duct":
        a = nx / 2.0
        s["nu"] = case.get("nu", 0.1)
        s["faces"][4] = s["faces"][5] = PERIODIC
        s["force"] = (0.0, 0.0, 0.02 * s["nu"] / (DUCT_K * a * a))
    elif flow == "pulsatile":  # period 1000 steps, Womersley number 4
        b = nx / 2.0
        s["nu"] = b * b * (2.0 * math.pi / 1000.0) / 16.0
        s["faces"][4] = s["faces"][5] = PERIODIC
        s["force"] = (0.0, 0.0, 0.02 * s["nu"] / (DUCT_K * b * b))
        s["period"] = 1000.0
    elif flow == "pressure_duct":  # physical spacing 2 / (nx - 1), viscosity 0.03, 1/tau = 1
        dx = 2.0 / (nx - 1)
        c = dx / (0.5 / 3.0 * dx * dx / 0.03)
        s["faces"] = [NEQ_P, NEQ_P, NEQ_U, NEQ_U, NEQ_U, NEQ_U]
        s["nu"] = 0.5 / 3.0
        s["p_face"][0], s["p_face"][1] = 1.1 / c ** 2, 1.0 / c ** 2
        s["p_ref"] = 1.05 / c ** 2
        s["U"] = 0.2 / c
    elif flow == "porous":
        s["faces"] = [PERIODIC] * 6
        s["force"] = (1e-6, 0.0, 0.0)
        s["U"] = 1e-3
    return s


def _fields(case, s, seed):
    """A smooth seeded initial state: a few long waves in u (3, N) and p (N)."""
    g = torch.Generator().manual_seed(int(seed))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) / nx
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny
    z = (torch.arange(nz, device="cuda", dtype=torch.float64) + 0.5) / nz
    out = []
    for k in range(4):
        f = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.float64)
        for _ in range(3):
            m = torch.randint(0, 3, (3,), generator=g).tolist()
            ph = (2 * math.pi * torch.rand(3, generator=g)).tolist()
            a = float(torch.rand(1, generator=g)) - 0.5
            f += a * (torch.cos(2 * math.pi * m[2] * z + ph[2])[:, None, None]
                      * torch.cos(2 * math.pi * m[1] * y + ph[1])[None, :, None]
                      * torch.cos(2 * math.pi * m[0] * x + ph[0])[None, None, :])
        out.append(f * s["U"] * (0.5 if k < 3 else 0.02) + (s["p_ref"] if k == 3 else 0.0))
    u, p = torch.stack(out[:3]), out[3]
    if case["flow"] == "pressure_duct":
        p[:, :, 0], p[:, :, -1] = s["p_face"][0], s["p_face"][1]
    return u.reshape(3, -1).contiguous(), p.reshape(-1).contiguous()


def _solid(case, seed):
    """Overlapping random spheres of radius 6, 30 % solid, periodic."""
    n = case["nx"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    o = torch.arange(-6, 7, device="cuda")
    dz, dy, dx = torch.meshgrid(o, o, o, indexing="ij")
    ball = dx * dx + dy * dy + dz * dz <= 36
    bz, by, bx = dz[ball], dy[ball], dx[ball]
    solid = torch.zeros(n ** 3, dtype=torch.uint8, device="cuda")
    part = 0.0
    while part < 0.3:
        k = max(1, int((0.3 - part) * n ** 3 / bx.numel() * 0.5) + 1)
        c = torch.randint(0, n, (3, k, 1), device="cuda", generator=g)
        solid[(((c[0] + bz) % n) * n + (c[1] + by) % n) * n + (c[2] + bx) % n] = 1
        part = float(solid.float().mean())
    return solid


def _domains(case):
    """The uneven domains of a batch: cavity or duct, Q, side, Re, storage."""
    r = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["domains"]):
        flow = "cavity" if r.random() < 0.5 else "duct"
        d = dict(flow=flow, Q=14 if r.random() < 0.5 else 18, storage="f32", sr=0)
        n = int(r.integers(case["lmin"], case["lmax"] + 1))
        Re = float(r.uniform(100.0, 1000.0))
        d.update(nx=n, ny=n, nz=n, Re=Re, nu=0.02 * n / Re)
        d["storage"] = "f32" if r.random() < 0.5 else "f16"
        out.append(d)
    return out


# ---- the library's side --------------------------------------------------------

def _stream():
    return torch.cuda.current_stream().cuda_stream


class _Owner:
    """A handle, destroyed with the last object that needs it."""

    def __init__(self, handle, destroy):
        self.handle = handle
        weakref.finalize(self, destroy, handle).atexit = False


class _Buffer:
    """A domain's device populations, as an array for torch; a tensor made of
    it keeps the domain alive."""

    def __init__(self, owner, address, count, storage):
        kind = {"f64": "<f8", "f32": "<f4", "f16": "<f2", "bf16": "<i2"}[storage]
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": kind,
                                         "data": (address, False), "version": 2}


def prepare(case, seed):
    if case["flow"] == "batch":
        return _prepare_batch(case, seed)
    s = _setup(case)
    Q, nx, ny, nz = case["Q"], case["nx"], case["ny"], case["nz"]
    h = lbm.lbm_create(Q, nx, ny, nz, case["storage"], _stream())
    state = dict(case=case, owner=_Owner(h, lbm.lbm_destroy))
    lbm.lbm_set_geometry(h, s["faces"], s["uw"], s["edge"])
    # a solve of this length checks convergence once, at its end
    every = case["steps"] if case["flow"] == "cavity" and case["steps"] >= 1000 else 0
    lbm.lbm_set_params(h, nu=s["nu"], force=s["force"], force_period=s["period"],
                       p_ref=s["p_ref"], p_face=s["p_face"], rounding=case["sr"],
                       residual_interval=every)
    if case["flow"] == "porous":
        lbm.lbm_set_solid(h, _solid(case, seed))
    if nx * ny * nz >= 1 << 20 and case["flow"] != "monitor":  # a long run on a large grid tunes
        lbm.lbm_autotune(h, 0)
    u, p = _fields(case, s, seed)
    if case["flow"] == "monitor":
        f = torch.empty(Q * _cells(case), device="cuda", dtype=torch.float64)
        T = _tables(Q)
        _equilibrium(T, u, p, f.view(Q, -1))
        state.update(f0=f, up=torch.empty(4 * _cells(case), device="cuda", dtype=torch.float64))
        return state
    lbm.lbm_init_equilibrium(h, u, p)
    if every:
        lbm.lbm_reductions(h)
    state["every"] = every
    address, nbytes = lbm.lbm_device_populations(h)
    f = torch.as_tensor(_Buffer(state["owner"], address, nbytes // BYTES[case["storage"]],
                                case["storage"]), device="cuda")
    state["f"] = f.view(torch.bfloat16) if case["storage"] == "bf16" else f
    return state


def _prepare_batch(case, seed):
    ds = _domains(case)
    b = lbm.lbm_batch_create(len(ds), 0, _stream())
    state = dict(case=case, owner=_Owner(b, lbm.lbm_batch_destroy), slots=[])
    lbm.lbm_batch_set_launch(b, 64, 2, 0)  # the serving loop's launch
    total = {"f32": 0, "f16": 0}
    for k, d in enumerate(ds):
        s = _setup(d)
        slot = lbm.lbm_batch_add(b, d["Q"], d["nx"], d["ny"], d["nz"], d["storage"], s["faces"],
                                 s["uw"], nu=s["nu"], force=s["force"])
        u, p = _fields(d, s, seed * 1000 + k)
        lbm.lbm_batch_init_equilibrium(b, slot, u, p)
        state["slots"].append((slot, d["storage"], total[d["storage"]], 3 * _cells(d)))
        total[d["storage"]] += 3 * _cells(d)
    for storage, n in total.items():
        state[storage] = torch.empty(n, device="cuda", dtype=torch.float32)
    torch.cuda.synchronize()
    return state


def run(state):
    case, h = state["case"], state["owner"].handle
    if case["flow"] == "batch":
        lbm.lbm_batch_step(h, case["steps"], 50)
        stats = lbm.lbm_batch_reductions_all(h, case["domains"])
        for slot, storage, at, n in state["slots"]:
            lbm.lbm_batch_read_fields(h, slot, lbm.LBM_FIELD_U, state[storage][at:at + n],
                                      lbm.LBM_DTYPE_F32)
        flux = np.array([list(stats[slot[0]].sum_u) for slot in state["slots"]], dtype=np.float32)
        return {"u_f32": state["f32"], "u_f16": state["f16"], "flux": flux}
    if case["flow"] == "monitor":
        lbm.lbm_set_step(h, 0)
        lbm.lbm_write_populations(h, state["f0"])
        s = lbm.lbm_reductions(h)
        lbm.lbm_read_fields(h, lbm.LBM_FIELD_U | lbm.LBM_FIELD_P, state["up"])
        lbm.lbm_step(h, case["steps"])
        lbm.lbm_reductions(h)
        r = lbm.lbm_residual(h, lbm.LBM_RESIDUAL_CAVITY)
        sums = np.array(list(s.sum_abs_u) + list(s.sum_u) + [s.sum_P, s.max_abs_u])
        return {"up": state["up"], "sums": sums, "residual": np.float32(r)}
    lbm.lbm_step(h, case["steps"])
    out = {"f": state["f"]}
    if state["every"]:
        out["residual"] = np.float32(lbm.lbm_residual(h, lbm.LBM_RESIDUAL_CAVITY))
    return out


# ---- the same flows in 64-bit torch ----------------------------------------------

_AXES = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
_EDGES = [(1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1),
          (-1, 0, -1), (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)]
_CUBE = [(1, 1, 1), (-1, 1, 1), (1, -1, 1), (-1, -1, 1), (1, 1, -1), (-1, 1, -1), (1, -1, -1),
         (-1, -1, -1)]


def _tables(Q):
    """Velocities, weights, w0 and the orthogonal moment rows (Gram-Schmidt of
    the monomials in order) with the class of each row's rate."""
    if Q == 14:
        c, w, w0 = _AXES + _CUBE, [1 / 9] * 6 + [1 / 72] * 8, 2 / 9
    elif Q == 18:
        c, w, w0 = _AXES + _EDGES, [1 / 18] * 6 + [1 / 36] * 12, 1 / 3
    else:
        c = _AXES + _EDGES + _CUBE
        w, w0 = [2 / 27] * 6 + [1 / 54] * 12 + [1 / 216] * 8, 8 / 27
    c, w = np.array(c, dtype=np.float64), np.array(w)
    x, y, z = c.T
    n2 = x * x + y * y + z * z
    rows = [(np.ones(Q), "c"), (n2, "e")]
    for v in (x, y, z):
        rows += [(v, "c"), (n2 * v, "q")]
    pxx, pww = 3 * x * x - n2, y * y - z * z
    if Q == 14:
        rows += [(pxx, "nu"), (pww, "nu"), (x * y, "nu"), (y * z, "nu"), (x * z, "nu"),
                 (x * y * z, "t")]
    else:
        rows += [(pxx, "nu"), (n2 * pxx, "pi"), (pww, "nu"), (n2 * pww, "pi"), (x * y, "nu"),
                 (y * z, "nu"), (x * z, "nu"), (pww * x, "t"), ((z * z - x * x) * y, "t"),
                 ((x * x - y * y) * z, "t")]
    if Q == 26:
        rows += [(n2 * n2, "e")] + [(n2 * n2 * v, "q") for v in (x, y, z)]
        rows += [(n2 * x * y, "pi"), (n2 * y * z, "pi"), (n2 * x * z, "pi"), (x * y * z, "t")]
    T = []
    for r, _ in rows:
        r = r.copy()
        for _ in range(2):
            for t in T:
                r -= (r @ t) / (t @ t) * t
        T.append(r)
    opp = [int(np.where((c == -v).all(1))[0][0]) for v in c]
    return dict(Q=Q, c=c, w=w, w0=w0, T=np.array(T), cls=[k for _, k in rows], opp=opp)


def _equilibrium(T, u, p, out):
    """f_eq of velocity u and pressure p into out (Q, N)."""
    u2 = (u * u).sum(0)
    for a in range(T["Q"]):
        cu = u[0] * T["c"][a, 0] + u[1] * T["c"][a, 1] + u[2] * T["c"][a, 2]
        out[a] = T["w"][a] * (3 * p + 3 * cu + 4.5 * cu * cu - 1.5 * u2)
    return out


def _dev(v):
    return torch.tensor(np.ascontiguousarray(v), device="cuda", dtype=torch.float64)


class _Exact:
    def __init__(self, case, seed):
        self.case, self.s = case, _setup(case)
        s, T = self.s, _tables(case["Q"])
        self.T, Q, c, w = T, T["Q"], T["c"], T["w"]
        self.n = (case["nx"], case["ny"], case["nz"])
        self.N = _cells(case)
        self.solid = _solid(case, seed).bool() if case["flow"] == "porous" else None
        rate = dict(c=1.0, e=1.19, q=1.2, nu=1.0 / (3.0 * s["nu"] + 0.5), pi=1.19, t=0.98)
        S = np.diag([rate[k] for k in T["cls"]])
        inv = T["T"].T @ np.diag(1.0 / (T["T"] ** 2).sum(1))
        K = inv @ S @ T["T"]
        # f_eq as a matrix on (3p - 3/2 u^2, u, u u)
        A = np.zeros((Q, 10))
        A[:, 0] = w
        A[:, 1:4] = 3 * w[:, None] * c
        for k, (i, j) in enumerate([(0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)]):
            A[:, 4 + k] = 4.5 * w * c[:, i] * c[:, j] * (1 if i == j else 2)
        Z = np.eye(Q)
        Z[0, 0] = 0.0
        G = inv @ (np.eye(Q) - 0.5 * S) @ Z @ T["T"]
        self.keep, self.relax, self.guo = _dev(np.eye(Q) - K), _dev(K @ A), G
        self.moments = _dev(np.vstack([np.ones(Q), c.T]))
        self._links()
        u, p = _fields(case, s, seed)
        self.f = torch.empty((Q, self.N), device="cuda", dtype=torch.float64)
        _equilibrium(T, u, p - s["p_ref"], self.f)
        if self.solid is not None:
            self.f[:, self.solid] = 0.0
        self.t = 0

    def force(self, t):
        P = self.s["period"]
        k = math.cos(2 * math.pi * t / P) if P > 0 else 1.0
        return [v * k for v in self.s["force"]]

    def _links(self):
        """Where each population of each node comes from, and the lid's terms."""
        T, s, n = self.T, self.s, self.n
        i = torch.arange(self.N, device="cuda")
        xyz = [i % n[0], (i // n[0]) % n[1], i // (n[0] * n[1])]
        self.src = torch.empty((T["Q"], self.N), device="cuda", dtype=torch.int64)
        self.lid = []
        for a in range(T["Q"]):
            c = [int(v) for v in T["c"][a]]
            wall = torch.zeros(self.N, dtype=torch.bool, device="cuda")
            flip = torch.zeros(self.N, dtype=torch.int64, device="cuda")
            at, lid = [], None
            for k in range(3):
                v = xyz[k] - c[k]
                for face, out in ((2 * k, v < 0), (2 * k + 1, v >= n[k])):
                    if (c[k] > 0) != (face % 2 == 0) or c[k] == 0:
                        continue
                    kind = s["faces"][face]
                    if kind == PERIODIC:
                        v = v % n[k]
                    elif kind == SYMMETRY:
                        v = torch.where(out, xyz[k], v)
                        flip = torch.where(out, flip | (1 << k), flip)
                    else:
                        v = torch.where(out, xyz[k], v)
                        wall = wall | out
                        if kind == LID:
                            lid = (face, out)
                at.append(v)
            j = at[0] + n[0] * (at[1] + n[1] * at[2])
            if self.solid is not None:
                wall = wall | self.solid[j]
            b = torch.full((self.N,), a, device="cuda", dtype=torch.int64)
            for m in range(1, 8):
                hit = flip == m
                if bool(hit.any()):
                    want = [-v if (m >> k) & 1 else v for k, v in enumerate(c)]
                    b[hit] = int(np.where((T["c"] == np.array(want)).all(1))[0][0])
            self.src[a] = torch.where(wall, T["opp"][a] * self.N + i, b * self.N + j)
            if lid:
                face, out = lid
                at = torch.nonzero(out).reshape(-1)
                val = torch.full((at.numel(),), 6 * T["w"][a] * float(T["c"][a] @ s["uw"][face]),
                                 device="cuda", dtype=torch.float64)
                if s["edge"]:
                    axis, first, last = s["edge"][face]
                    val[xyz[axis][at] == 0] *= first
                    val[xyz[axis][at] == n[axis] - 1] *= last
                self.lid.append((a, at, val))
        self.rim = None
        if any(k in (NEQ_U, NEQ_P) for k in s["faces"]):
            to = [v.clone() for v in xyz]
            on = torch.zeros(self.N, dtype=torch.bool, device="cuda")
            still = torch.zeros(self.N, dtype=torch.bool, device="cuda")
            pres = torch.full((self.N,), math.nan, device="cuda", dtype=torch.float64)
            for face in range(6):
                k, last = face // 2, face % 2
                here = xyz[k] == (n[k] - 1 if last else 0)
                on |= here
                to[k] = torch.where(here, torch.full_like(to[k], n[k] - 2 if last else 1), to[k])
                if s["faces"][face] == NEQ_U:
                    still |= here
                else:
                    pres = torch.where(here & pres.isnan(),
                                       torch.full_like(pres, s["p_face"][face] - s["p_ref"]), pres)
            at = torch.nonzero(on).reshape(-1)
            j = to[0] + n[0] * (to[1] + n[1] * to[2])
            self.rim = (at, j[at], still[at], pres[at])

    def macro(self, f, t):
        """u (3, N) and the pressure of the stored deviations."""
        m = self.moments @ f
        F = self.force(t)
        u = m[1:]
        for k in range(3):
            if F[k]:
                u[k] += 0.5 * F[k]
        u2 = (u * u).sum(0)
        w0 = self.T["w0"]
        return u, (m[0] - 1.5 * w0 * u2) / (3.0 * (1.0 - w0)), u2

    def step(self):
        T, F = self.T, self.force(self.t)
        u, p, u2 = self.macro(self.f, self.t)
        g = torch.empty((10, self.N), device="cuda", dtype=torch.float64)
        g[0] = 3 * p - 1.5 * u2
        g[1:4] = u
        for k, (i, j) in enumerate([(0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)]):
            torch.mul(u[i], u[j], out=g[4 + k])
        mix, const = self.relax, None
        if any(self.s["force"]):
            c, w, Fv = T["c"], T["w"], np.array(F)
            cF = c @ Fv
            mix = mix.clone()
            mix[:, 1:4] += _dev(self.guo @ (w[:, None] * (9 * c * cF[:, None] - 3 * Fv)))
            const = _dev(self.guo @ (3 * w * cF))
        post = torch.addmm(mix @ g, self.keep, self.f)
        if const is not None:
            post += const[:, None]
        self.f = torch.take(post, self.src)
        for a, at, val in self.lid:
            self.f[a, at] += val
        if self.solid is not None:
            self.f[:, self.solid] = 0.0
        self.t += 1
        if self.rim is not None:
            at, j, still, pres = self.rim
            fj = self.f[:, j]
            uf, pf, _ = self.macro(fj, self.t)
            ub = torch.where(still, torch.zeros_like(uf), uf)
            pb = torch.where(pres.isnan(), pf, pres)
            self.f[:, at] = (_equilibrium(T, ub, pb, torch.empty_like(fj)) + fj
                             - _equilibrium(T, uf, pf, torch.empty_like(fj)))

    def run(self, steps):
        for _ in range(steps):
            self.step()


def _change(u, v):
    return np.float64(float((u - v).abs().sum() / u.abs().sum()))


def exact(case, seed):
    if case["flow"] == "batch":
        u, flux = {"f32": [], "f16": []}, []
        for k, d in enumerate(_domains(case)):
            e = _Exact(d, seed * 1000 + k)
            e.run(case["steps"])
            v = e.macro(e.f, e.t)[0]
            u[d["storage"]].append(v.reshape(-1))
            flux.append(v.sum(1).tolist())
        none = torch.empty(0, device="cuda", dtype=torch.float64)
        return {"u_f32": torch.cat(u["f32"] or [none]), "u_f16": torch.cat(u["f16"] or [none]),
                "flux": np.array(flux)}
    e = _Exact(case, seed)
    u, p, _ = e.macro(e.f, 0)
    if case["flow"] == "monitor":
        P = e.f.sum()
        sums = np.array(u.abs().sum(1).tolist() + u.sum(1).tolist() + [float(P),
                                                                       float(u.abs().max())])
        up = torch.cat([u.reshape(-1), p])
        e.run(case["steps"])
        return {"up": up, "sums": sums, "residual": _change(e.macro(e.f, e.t)[0], u)}
    e.run(case["steps"])
    out = {"f": e.f.reshape(-1)}
    if case["flow"] == "cavity" and case["steps"] >= 1000:
        out["residual"] = _change(e.macro(e.f, e.t)[0], u)
    return out
