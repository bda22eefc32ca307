"""Performance cases: what a user of this framework has it do, at the sizes of
the repository's own workloads (inputs.py, the tests, bench.py).

A case is one call in a user's time loop: a load step of a simulation followed
by the read-back of the point state (`Simulation.step`, `Simulation.read`), the
same for a batched context (`Batch.step`, `Batch.read`), or one binning of
device-resident points (`mpm_bin_noalloc`).  The 2D simulations take each step
from the same accepted state (`Simulation.restore` first), as an adaptive
choice of the time step does that tries a step again; the 3D and batched ones
go on along their trajectories, as a time loop does, under cyclic loads where
a constant load would let a long run settle into its steady state.

`exact` is an independent FP64 statement of the step in plain torch: the
residual written with automatic differentiation for its Jacobian (coloured
forward mode), a direct block-tridiagonal solve, Newton to round-off.
"""
import ctypes as C
import math
from dataclasses import replace

import numpy as np
import torch

from paper_1905_00671_gb300 import inputs as I
from paper_1905_00671_gb300 import mpm


def listed():
    return [
        # binning the points of the strip footing on the device, as a host
        # application does that owns all device memory: the smallest call
        dict(name="bin-footing", kind="bin", dim=2, nx=200, ny=102, nz=0, ppc=2, jitter=0.15),
        # the Terzaghi column (Sec. 5.1 of the paper, the smallest simulation):
        # original MPM, quasi-static, a few hundred nodes, launches count
        dict(name="column", kind="column", nx=4, ny=40, precision=0, jitter=0.0),
        # the self-weight deposit (Sec. 5.3 grid, 25 points per cell) with
        # Kozeny-Carman permeability, mixed precision
        dict(name="selfweight-mixed", kind="selfweight", nx=16, ny=16, precision=1, jitter=0.0),
        # the harmonic footing (Sec. 5.2): Hencky, Newmark, consistent mass
        dict(name="harmonic", kind="harmonic", nx=40, ny=40, precision=0, jitter=0.0),
        # the 2D strip footing of the benchmark, 80,000 GIMP points, Newmark,
        # its points a little off the cells' sub-lattice as after some steps
        dict(name="footing", kind="footing", nx=200, ny=100, precision=0, jitter=0.02),
        # a footing of odd size, its points in random order, in mixed
        # precision
        dict(name="footing-odd-mixed", kind="footing", nx=151, ny=83, precision=1, jitter=0.02),
        # a 3D block of odd size, its points shuffled and off the sub-lattice
        dict(name="block-odd", kind="block", nx=37, ny=29, nz=19, precision=0, jitter=0.02),
        # the 3D consolidation block of the benchmark, 1,048,576 points, mixed
        dict(name="block-mixed", kind="block", nx=64, ny=64, nz=32, precision=1, jitter=0.0),
        # the 3D slope of the benchmark's default line, 4.2 million points: the
        # largest configuration, in both precisions
        dict(name="slope", kind="slope", nx=128, ny=128, nz=64, precision=0, jitter=0.0),
        dict(name="slope-mixed", kind="slope", nx=128, ny=128, nz=64, precision=1, jitter=0.0),
        # many independent 2D instances of uneven size in one batched context
        # (design studies, data generation)
        dict(name="batch-column", kind="batch-column", count=64, layout=5, precision=0),
        dict(name="batch-footing", kind="batch-footing", count=64, layout=5, precision=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bin", "column", "selfweight", "harmonic", "footing", "footing", "block", "block",
                       "slope", "batch-column", "batch-footing"])
    precision = rng.randrange(2)
    jitter = rng.choice([0.0, 0.01, 0.02])
    if kind == "bin":
        if rng.random() < 0.5:
            return dict(kind=kind, dim=2, nx=_log_int(rng, 8, 400), ny=_log_int(rng, 8, 400), nz=0,
                        ppc=rng.randint(1, 5), jitter=0.15)
        return dict(kind=kind, dim=3, nx=_log_int(rng, 5, 64), ny=_log_int(rng, 5, 64), nz=_log_int(rng, 5, 64),
                    ppc=rng.randint(1, 3), jitter=0.15)
    if kind == "column":
        return dict(kind=kind, nx=_log_int(rng, 4, 32), ny=_log_int(rng, 16, 96), precision=precision, jitter=0.0)
    if kind == "selfweight":
        return dict(kind=kind, nx=rng.randint(12, 40), ny=rng.randint(12, 32), precision=precision, jitter=0.0)
    if kind == "harmonic":
        return dict(kind=kind, nx=rng.randint(28, 64), ny=rng.randint(28, 64), precision=precision, jitter=0.0)
    if kind == "footing":
        return dict(kind=kind, nx=_log_int(rng, 24, 200), ny=_log_int(rng, 16, 100), precision=precision,
                    jitter=jitter)
    if kind == "block":
        return dict(kind=kind, nx=_log_int(rng, 9, 64), ny=_log_int(rng, 9, 64), nz=_log_int(rng, 9, 32),
                    precision=precision, jitter=jitter)
    if kind == "slope":  # the benchmark's 2 : 2 : 1 box, from a quarter of its width up
        nz = rng.randint(16, 64)
        return dict(kind=kind, nx=2 * nz + rng.randint(-1, 1), ny=rng.randint(nz, 2 * nz), nz=nz,
                    precision=precision, jitter=0.0)
    return dict(kind=kind, count=_log_int(rng, 3, 64), layout=rng.randint(6, 1000), precision=0)


# ------------------------------------------------------------------ inputs
def _vary(w, seed, k_spread=0.5):
    """Seeded per-point stiffness and permeability (the generators without
    random fields of their own)."""
    rng = np.random.default_rng(seed)
    return replace(w, E=w.E * np.exp(0.05 * rng.standard_normal(w.n)),
                   k=w.k * 10.0 ** (k_spread * rng.uniform(-1.0, 1.0, w.n)))


def _workload(case, seed):
    kind = case["kind"]
    if kind == "column":
        return _vary(I.terzaghi_column(ncell_x=case["nx"], ncell_y=case["ny"]), seed)
    if kind == "selfweight":  # the stiffer deposit of the tests: small strains over a long run
        return _vary(I.self_weight_consolidation(ncell=(case["nx"], case["ny"]), K=1.5e6), seed)
    if kind == "harmonic":
        return _vary(I.harmonic_footing(body=(case["nx"], case["ny"])), seed)
    if kind == "footing":
        w = I.strip_footing(body=(case["nx"], case["ny"]), seed=seed, half_width=min(1.0, 0.025 * case["nx"]))
        w = replace(w, ramp_time=0.0)  # the load applied at once
    elif kind == "block":
        w = I.consolidation_block(body=(case["nx"], case["ny"], case["nz"]), seed=seed,
                                  patch_half=min(1.0, 0.02 * min(case["nx"], case["ny"])))
    else:
        nx, nz = case["nx"], case["nz"]
        s = nz / 64.0
        return _vary(I.slope_3d(ncell=(nx, case["ny"], nz), z_toe=1.2 * s, z_crest=5.2 * s, x_toe=2.9 * s), seed, 0.0)
    return I.jittered(w, seed + 1, frac=case["jitter"], E_spread=0.05) if case["jitter"] else w


def _instances(case, seed):
    kd = "terzaghi" if case["kind"] == "batch-column" else "footing"
    ws = I.batch_instances(count=case["count"], seed=case["layout"], kind=kd)
    om = 0.1 if kd == "terzaghi" else 100.0  # cyclic loads of 63 steps a cycle
    return [replace(_vary(w, seed + 17 * i), load_omega=om) for i, w in enumerate(ws)]


def _bin_points(case, seed):
    nc = (case["nx"], case["ny"], case["nz"])
    x, _, lp = I.lattice(case["dim"], nc, 0.1, case["ppc"])
    rng = np.random.default_rng(seed)
    x = x + case["jitter"] * 2.0 * lp * rng.uniform(-1.0, 1.0, x.shape)
    return np.ascontiguousarray(x[rng.permutation(x.shape[0])])


FIELDS_QS = ("x", "u", "p", "F", "V", "lp")
FIELDS_DYN = ("x", "u", "p", "v", "a", "F", "V", "lp", "pd", "pdd")


def _options(case, dim):
    """Default options; a mixed-precision run asks the FP64 residual for a
    tighter Newton tolerance (one more of its cheap iterations), which brings
    its results to FP64 accuracy."""
    if not case["precision"]:
        return {}
    return {"precision": mpm.MPM_MIXED, "newton_rtol": 1e-10 if dim == 2 else 1e-9}


# time of the accepted state in its load history (0: the start of the load):
# the harmonic footing a tenth of its period in
START = {"harmonic": 0.006}


def prepare(case, seed):
    if case["kind"] == "bin":
        lib = mpm.load()
        lib.mpm_bin_noalloc.argtypes = [C.POINTER(mpm.mpm_grid), C.c_int64, C.c_void_p, C.c_void_p, C.c_void_p,
                                        C.c_void_p]
        g = mpm.mpm_grid(dim=case["dim"], h=0.1)
        for k, nc in enumerate((case["nx"], case["ny"], case["nz"])):
            g.ncell[k] = nc
        x = torch.from_numpy(_bin_points(case, seed)).cuda()
        return {"lib": lib, "grid": g, "x": x,
                "cell": torch.empty(x.shape[0], dtype=torch.int32, device="cuda"),
                "order": torch.empty(x.shape[0], dtype=torch.int64, device="cuda")}
    if case["kind"].startswith("batch"):
        ws = _instances(case, seed)
        fields = FIELDS_DYN if ws[0].dynamic else FIELDS_QS
        return {"batch": mpm.Batch(ws, **_options(case, 2)), "fields": fields}
    w = _workload(case, seed)
    state = {"sim": mpm.Simulation(w, **_options(case, w.dim)),
             "fields": FIELDS_DYN if w.dynamic else FIELDS_QS}
    if w.dim == 2:
        state["accepted"] = {"state": state["sim"].read(state["fields"]), "t": START.get(case["kind"], 0.0),
                             "steps": 0}
    return state


def run(state):
    if "x" in state:
        x, cell, order = state["x"], state["cell"], state["order"]
        rc = state["lib"].mpm_bin_noalloc(C.byref(state["grid"]), x.shape[0], x.data_ptr(), cell.data_ptr(),
                                          order.data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != mpm.MPM_OK:
            raise mpm.MPMError(rc, "mpm_bin_noalloc")
        return {"cell": cell, "order": order}
    if "batch" in state:
        state["batch"].step()
        parts = state["batch"].read(state["fields"])
        return {k: np.concatenate([p[k] for p in parts]) for k in state["fields"]}
    if "accepted" in state:
        state["sim"].restore(state["accepted"])
    state["sim"].step()
    return state["sim"].read(state["fields"])


# -------------------------------------------------------------------- work
def _size(case):
    """(points, nodes, dim, dynamic, values of state per point) from the sizes."""
    kind = case["kind"]
    if kind.startswith("batch"):
        n, nn = 0, 0
        for w in _instances(case, 1):  # the mean sizes do not depend on the seed
            n, nn = n + w.n, nn + w.nnodes
        dyn = kind == "batch-footing"
        return n, nn, 2, dyn, 19 if dyn else 12
    nx, ny, nz = case["nx"], case["ny"], case.get("nz", 0)
    if kind == "block":
        return 8 * nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 2), 3, False, 20
    if kind == "slope":  # about half of the box is filled
        return 4 * nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 1), 3, False, 20
    dyn = kind in ("harmonic", "footing")
    return (25 if kind == "selfweight" else 4) * nx * ny, (nx + 1) * (ny + 1), 2, dyn, 19 if dyn else 12


def work(case):
    """Bytes: the point state read and written, and handed back once; the
    Dirichlet data read.  Flops: two linearisations of the step (a Newton
    iteration and its check at the least), each point contributing to the
    symmetric pairs of its 2^d nearest nodes, with two products of the
    resulting matrix (3^d blocks a row) with a vector."""
    if case["kind"] == "bin":
        n = case["ppc"] ** case["dim"] * case["nx"] * case["ny"] * max(case["nz"], 1)
        return {"bytes": n * (8 * case["dim"] + 4 + 8), "flops": n * 2 * case["dim"]}
    n, nn, d, dyn, state = _size(case)
    pairs = 2 ** d * (2 ** d + 1) // 2
    term = (107 if dyn else 93) if d == 3 else (65 if dyn else 55)
    return {"bytes": 8 * n * (3 * state + 5) + nn * 9 * (d + 1),
            "flops": 2 * n * pairs * term + 2 * nn * 3 ** d * 2 * (d + 1) ** 2}


# ------------------------------------------------------------------- exact
EXACT_COST = 2.5e12  # dense solve work beyond which exact() gives no value
EXACT_EVALS = 4.0e9    # residual work (points x supports x colours) likewise


def exact(case, seed):
    if case["kind"] == "bin":
        return _exact_bin(case, seed)
    if case["kind"].startswith("batch"):
        if case["count"] > 6:
            return None
        parts = [_exact_step(w) for w in _instances(case, seed)]
        if any(p is None for p in parts):
            return None
        return {k: np.concatenate([p[k] for p in parts]) for k in parts[0]}
    return _exact_step(_workload(case, seed), START.get(case["kind"], 0.0))


def _exact_bin(case, seed):
    x = _bin_points(case, seed)
    nc = (case["nx"], case["ny"], case["nz"])
    cell = np.zeros(x.shape[0], np.int64)
    for k in reversed(range(case["dim"])):
        cell = cell * nc[k] + np.floor((x[:, k] - 0.0) / 0.1).astype(np.int64)
    return {"cell": cell.astype(np.int32), "order": np.argsort(cell, kind="stable")}


def _hat_integral(t):
    """Antiderivative of the unit hat max(1 - |t|, 0)."""
    t = t.clamp(-1.0, 1.0)
    return 0.5 + t - 0.5 * t * t.abs()


def _basis_1d(w, x, lp, k):
    """First node and 1D basis S, dS, S0 in four slots along axis k (Eqs.
    gimp-basis, gimp-basis-gradient; the FE basis for original MPM)."""
    xi = (x[:, k] - w.origin[k]) / w.h
    slot = torch.arange(4, device=x.device, dtype=x.dtype)
    if w.shape == I.ORIG:
        first = torch.floor(xi)
        t = xi[:, None] - (first[:, None] + slot)
        live = (slot < 2).to(x.dtype)
        dS = (torch.where(slot == 0, -1.0, 1.0).to(x.dtype) / w.h * live).expand_as(t)
        return first.long(), (1.0 - t.abs()) * live, dS, 0.5 * live.expand_as(t), 2
    dx = x[:, k] - w.origin[k]
    lo, hi = ((dx - lp[:, k]) / w.h).clamp(min=0.0), ((dx + lp[:, k]) / w.h).clamp(max=float(w.ncell[k]))
    first = torch.floor(lo)
    node = first[:, None] + slot
    a, b, ln = lo[:, None] - node, hi[:, None] - node, (hi - lo)[:, None]
    S = (_hat_integral(b) - _hat_integral(a)) / ln
    dS = ((1.0 - b.abs()).clamp(min=0.0) - (1.0 - a.abs()).clamp(min=0.0)) / ln / w.h
    S0 = 0.5 * (b.clamp(-1.0, 1.0) - a.clamp(-1.0, 1.0)) / ln
    return first.long(), S, dS, S0, int((torch.ceil(hi) - first).max().item()) + 1


def _log_spd2(b):
    """Logarithm of symmetric positive definite 2 x 2 matrices, smooth at equal
    eigenvalues: ln b = ln(det b)/2 1 + f(z)/m (b - m 1), m = tr b / 2,
    z = 1 - det b / m^2, f(z) = atanh(sqrt z) / sqrt z."""
    m = 0.5 * (b[:, 0, 0] + b[:, 1, 1])
    hd = 0.5 * (b[:, 0, 0] - b[:, 1, 1])
    det = b[:, 0, 0] * b[:, 1, 1] - b[:, 0, 1] * b[:, 1, 0]
    z = (hd * hd + b[:, 0, 1] * b[:, 1, 0]) / (m * m)
    small = z < 0.02
    zs = torch.where(small, z, torch.zeros_like(z))
    ser = torch.zeros_like(z)
    for j in reversed(range(12)):
        ser = ser * zs + 1.0 / (2 * j + 1)
    zb = torch.where(small, torch.full_like(z, 0.25), z)
    f = torch.where(small, ser, torch.atanh(zb.sqrt()) / zb.sqrt())
    eye = torch.eye(2, dtype=b.dtype, device=b.device)
    return 0.5 * torch.log(det)[:, None, None] * eye + (f / m)[:, None, None] * (b - m[:, None, None] * eye)


def _det(A):
    if A.shape[-1] == 2:
        return A[:, 0, 0] * A[:, 1, 1] - A[:, 0, 1] * A[:, 1, 0]
    return (A[:, 0] * torch.linalg.cross(A[:, 1], A[:, 2])).sum(1)


def _inv(A):
    if A.shape[-1] == 2:
        adj = torch.stack([A[:, 1, 1], -A[:, 0, 1], -A[:, 1, 0], A[:, 0, 0]], 1).view(-1, 2, 2)
    else:
        adj = torch.stack([torch.linalg.cross(A[:, 1], A[:, 2]), torch.linalg.cross(A[:, 2], A[:, 0]),
                           torch.linalg.cross(A[:, 0], A[:, 1])], 2)
    return adj / _det(A)[:, None, None]


class _ExactStep:
    """One load step from the initial state in FP64."""

    def __init__(self, w, t0=0.0):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.w, self.d = w, w.dim
        d = self.d
        T = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=dev)  # noqa: E731
        self.x, self.lp, self.V, self.p0 = T(w.x), T(w.lp), T(w.vol), T(w.p0)
        n = w.n
        self.v0 = T(w.v0) if w.v0 is not None else torch.zeros(n, d, dtype=torch.float64, device=dev)
        E, nu = T(w.E), T(w.nu)
        self.lam, self.G = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
        self.kap = T(w.k) / w.mu_f
        self.tau = (w.tau_scale / (2 * self.G)) if w.stabilize else torch.zeros_like(self.G)
        self.mass = ((1 - w.phi0) * w.rho_s + w.phi0 * w.rho_f) * self.V
        nn = w.nn
        self.nn, self.N = nn, w.nnodes
        self.axis = ax = int(np.argmax(nn))
        first, S, dS, S0, self.rad = [], [], [], [], 0
        for k in range(d):
            f, s, ds, s0, cnt = _basis_1d(w, self.x, self.lp, k)
            first.append(f), S.append(s), dS.append(ds), S0.append(s0)
            self.rad = max(self.rad, cnt - 1)
        ns = self.rad + 1
        idx, SS, SS0, GG, hat = [], [], [], [], []
        sn = T(w.surf_normal)
        y = (self.x + self.lp * sn - T(w.origin[:d])) / w.h
        for s in np.ndindex(*([ns] * d)):
            node, stride, a, a0, hy = 0, 1, 1.0, 1.0, 1.0
            g = [1.0] * d
            inside = torch.ones(n, dtype=torch.bool, device=dev)
            for k in range(d):
                nk = first[k] + s[k]
                inside &= nk < nn[k]
                node = node + nk.clamp(max=nn[k] - 1) * stride
                stride *= nn[k]
                a, a0 = a * S[k][:, s[k]], a0 * S0[k][:, s[k]]
                hy = hy * (1.0 - (y[:, k] - nk).abs()).clamp(min=0.0)
                g = [g[j] * (dS[k][:, s[k]] if j == k else S[k][:, s[k]]) for j in range(d)]
            live = inside.to(a.dtype)
            # a node of the slot range outside the support box has S = S0 = 0
            sup = ((a > 0) | (a0 > 0)).to(a.dtype) * live
            idx.append(node), SS.append(a * live), SS0.append(a0 * live), hat.append(hy * sup)
            GG.append(torch.stack(g, 1) * live[:, None])
        self.idx, self.S, self.S0, self.Gn = (torch.stack(t, 1) for t in (idx, SS, SS0, GG))
        self.raw = self.S
        M, phi = self.scatter(self.S * self.mass[:, None]), self.scatter(self.S * self.V[:, None]) / w.h ** d
        self.active = (M > 0) & (phi > 1e-4)
        act = self.active[self.idx].to(M.dtype)
        lump = lambda f: torch.where(M > 0, self.scatter(self.S * (self.mass * f)[:, None]) / M.clamp(min=1e-300), 0.0 * M)  # noqa: E731
        flds = [lump(self.p0)] + ([lump(self.v0[:, k]) for k in range(d)] if w.dynamic else [])
        if w.p2g_mass == I.P2G_CONSISTENT:
            flds = self.consistent(M, flds)
        self.Pn = flds[0]
        self.vn = torch.stack(flds[1:], 1) if w.dynamic else None
        sm, s0m = (self.S * act).sum(1, keepdim=True), (self.S0 * act).sum(1, keepdim=True)
        gm = (self.Gn * act[:, :, None]).sum(1, keepdim=True)
        cut = ((1 - act) * (((self.raw > 0) | (self.S0 > 0)).to(act.dtype))).sum(1) > 0
        Sr = self.S * act / sm
        Gr = (self.Gn - Sr[:, :, None] * gm) * act[:, :, None] / sm[:, :, None]
        self.S = torch.where(cut[:, None], Sr, self.S)
        self.Gn = torch.where(cut[:, None, None], Gr, self.Gn)
        self.S0 = torch.where(cut[:, None], self.S0 * act / s0m, self.S0)
        nb = d + 1
        fixed = torch.zeros(self.N, nb, dtype=torch.bool, device=dev)
        fixed[:, :d] = torch.as_tensor(w.u_fixed != 0, device=dev)
        fixed[:, d] = torch.as_tensor(w.p_fixed != 0, device=dev)
        X = torch.zeros(self.N, nb, dtype=torch.float64, device=dev)
        X[:, d] = self.Pn
        X[:, :d] = torch.where(fixed[:, :d], T(w.u_value), X[:, :d])
        X[:, d] = torch.where(fixed[:, d], T(w.p_value), X[:, d])
        X[~self.active] = 0.0
        fixed[~self.active] = True
        self.fixed, self.X0, self.g = fixed, X, T(w.g[:d])
        ext = torch.zeros(self.N, d, dtype=torch.float64, device=dev)  # Neumann data
        sid = torch.as_tensor(np.asarray(w.surf_id, np.int64), device=dev)
        if w.n_surf:
            on = sid >= 0
            tr = T(w.traction(t0 + w.dt))[sid[on]] * T(w.surf_area)[on][:, None]
            ht = torch.stack(hat, 1)[on]
            for i in range(d):
                ext[:, i].index_add_(0, self.idx[on].reshape(-1), (ht * tr[:, i:i + 1]).reshape(-1))
        self.ext = ext
        slab = self.rad * int(np.prod(nn)) // nn[ax] * nb
        blocks = -(-nn[ax] // self.rad)
        self.cost = 5.0 * blocks * float(slab) ** 3 if blocks > 1 else float(slab) ** 3
        self.evals = float(n) * ns ** d * (2 * self.rad + 1) ** d * nb

    def scatter(self, vals):
        out = torch.zeros(self.N, dtype=vals.dtype, device=vals.device)
        return out.index_add(0, self.idx.reshape(-1), vals.reshape(-1))

    def kirchhoff(self, b, J):
        eye = torch.eye(self.d, dtype=b.dtype, device=b.device)
        vol = (self.lam * torch.log(J))[:, None, None] * eye
        if self.w.model == I.MODEL_HENCKY:
            return vol + self.G[:, None, None] * _log_spd2(b)
        return vol + self.G[:, None, None] * (b - eye)

    def newmark(self, X):
        w, b, g, dt, d = self.w, self.w.beta, self.w.gamma, self.w.dt, self.d
        acc = X[:, :d] / (b * dt * dt) - self.vn / (b * dt)
        vel = g / (b * dt) * X[:, :d] + (1 - g / b) * self.vn
        dP = X[:, d] - self.Pn
        return acc, vel, g / (b * dt) * dP, dP / (b * dt * dt)

    def residual(self, X):
        w, d, dt = self.w, self.d, self.w.dt
        eye = torch.eye(d, dtype=X.dtype, device=X.device)
        Xq = X[self.idx]                                       # (n, ns, nb)
        dF = eye + torch.einsum("qsi,qsk->qik", Xq[:, :, :d], self.Gn)
        J = _det(dF)
        gr = torch.einsum("qsk,qkj->qsj", self.Gn, _inv(dF))
        b = dF @ dF.transpose(1, 2)
        tau = self.kirchhoff(b, J)
        vol = J * self.V
        ph = (self.S * Xq[:, :, d]).sum(1)
        gp = torch.einsum("qs,qsj->qj", Xq[:, :, d], gr)
        dev = self.S - self.S0
        m = self.mass
        stress = self.V[:, None, None] * tau
        body = (m[:, None] * self.g).expand(-1, d)
        wv = gp - w.rho_f * self.g
        if w.dynamic:
            acc, vel, pd, _ = self.newmark(X)
            ah = torch.einsum("qs,qsi->qi", self.S, acc[self.idx])
            gv = torch.einsum("qsi,qsj->qij", vel[self.idx], gr)
            pdev = (dev * pd[self.idx]).sum(1)
            divv = torch.einsum("qii->q", gv)
            body, wv = body - m[:, None] * ah, wv + w.rho_f * ah
            D = 0.5 * (gv + gv.transpose(1, 2))
            if w.model == I.MODEL_HENCKY:  # c : D = d tau along D b + b D, less the convected parts
                _, dtau = torch.func.jvp(lambda e: self.kirchhoff(e, _det(e).sqrt()), (b,), (D @ b + b @ D,))
                vis = dtau - D @ tau - tau @ D
            else:
                mu = self.G - self.lam * torch.log(J)
                vis = (self.lam * divv)[:, None, None] * eye + 2 * mu[:, None, None] * D
            stress = stress + self.V[:, None, None] * w.alpha_vis * vis
        else:
            pdev = (dev * ((X[:, d] - self.Pn) / dt)[self.idx]).sum(1)
            divv = torch.log(J) / dt
        kap = self.kap
        if w.permeability == I.PERM_KOZENY_CARMAN:
            phi = 1 - (1 - w.phi0) / J
            kap = kap * (1 - w.phi0) ** 2 / w.phi0 ** 3 * phi ** 3 / (1 - phi) ** 2
        mom = -torch.einsum("qsj,qij->qsi", gr, stress) + (vol * ph)[:, None, None] * gr + self.S[:, :, None] * body[:, None, :]
        mas = self.S * (vol * divv)[:, None] + (vol * kap)[:, None] * torch.einsum("qsj,qj->qs", gr, wv)
        mas = mas + dev * (self.V * self.tau * pdev)[:, None]
        cols = [self.scatter(mom[:, :, i]) + self.ext[:, i] for i in range(d)] + [self.scatter(mas)]
        return torch.stack(cols, 1).masked_fill(self.fixed, 0.0)

    # ---- linear algebra: stencil matrices on the node lattice
    def stencil_solve(self, A, rhs, nb):
        """Solve with the matrix A[a, o, i, j] coupling (node a, i) with (node
        a + offset o, j) by block-tridiagonal elimination over slabs of `rad`
        node planes along the longest axis; rhs (N * nb, m)."""
        d, rad, nn, ax = self.d, self.rad, self.nn, self.axis
        dev = A.device
        coord = torch.stack(torch.meshgrid(*[torch.arange(q, device=dev) for q in nn], indexing="ij"), -1)
        coord = coord.permute(*reversed(range(d)), d).reshape(-1, d)   # node numbering: x fastest
        plane = int(np.prod(nn)) // nn[ax]
        pos = torch.zeros(self.N, dtype=torch.long, device=dev)
        stride = 1
        for k in range(d):
            if k != ax:
                pos, stride = pos + coord[:, k] * stride, stride * nn[k]
        slab = coord[:, ax] // rad
        loc = (coord[:, ax] % rad) * plane + pos
        B, nslab = rad * plane * nb, -(-nn[ax] // rad)
        tri = torch.zeros(nslab * 3 * B * B, dtype=A.dtype, device=dev)
        for o, off in enumerate(np.ndindex(*([2 * rad + 1] * d))):
            nbc = coord + torch.as_tensor([q - rad for q in off], device=dev)
            ok = ((nbc >= 0) & (nbc < torch.as_tensor(nn, device=dev))).all(1)
            a = torch.nonzero(ok)[:, 0]
            c, st = torch.zeros_like(a), 1
            for k in range(d):
                c, st = c + nbc[a, k] * st, st * nn[k]
            side = slab[c] - slab[a] + 1
            for i in range(nb):
                for j in range(nb):
                    at = ((slab[a] * 3 + side) * B + loc[a] * nb + i) * B + loc[c] * nb + j
                    tri[at] = A[a, o, i, j]
        tri = tri.view(nslab, 3, B, B)
        r = torch.zeros(nslab, B, rhs.shape[1], dtype=A.dtype, device=dev)
        dof = (slab[:, None] * B + loc[:, None] * nb + torch.arange(nb, device=dev)).reshape(-1)
        r.view(nslab * B, -1)[dof] = rhs
        used = torch.zeros(nslab * B, dtype=torch.bool, device=dev)
        used[dof] = True
        pad = (~used).to(A.dtype).view(nslab, B)
        tri[:, 1] += torch.diag_embed(pad)
        up = [None] * nslab
        for s in range(nslab):
            Dg, f = tri[s, 1], r[s]
            if s:
                Dg, f = Dg - tri[s, 0] @ up[s - 1], f - tri[s, 0] @ r[s - 1]
            sol = torch.linalg.solve(Dg, torch.cat([tri[s, 2], f], 1))
            up[s], r[s] = sol[:, :B], sol[:, B:]
        for s in reversed(range(nslab - 1)):
            r[s] -= up[s] @ r[s + 1]
        return r.view(nslab * B, -1)[dof]

    def consistent(self, M, flds):
        d, rad = self.d, self.rad
        noff = (2 * rad + 1) ** d
        A = torch.zeros(self.N * noff, dtype=M.dtype, device=M.device)
        slots = list(np.ndindex(*([rad + 1] * d)))
        for i, si in enumerate(slots):
            for j, sj in enumerate(slots):
                o = 0
                for k in range(d):
                    o = o * (2 * rad + 1) + sj[k] - si[k] + rad
                A.index_add_(0, self.idx[:, i] * noff + o, self.raw[:, i] * self.raw[:, j] * self.mass)
        A = A.view(self.N, noff, 1, 1)
        # nodes outside the active set keep their lumped values: identity rows
        off = torch.zeros(noff, dtype=M.dtype, device=M.device)
        off[noff // 2] = 1.0
        A = torch.where(self.active[:, None, None, None], A, off[:, None, None])
        f = torch.stack(flds, 1)
        rhs = torch.where(self.active[:, None], M[:, None] * f, f)
        sc = torch.where(self.active, 1.0 / M.clamp(min=1e-300), torch.ones_like(M))
        sol = self.stencil_solve(A * sc[:, None, None, None], rhs * sc[:, None], 1)
        return [sol[:, k] for k in range(sol.shape[1])]

    def jacobian(self, X):
        d, nb, rad, nn = self.d, self.d + 1, self.rad, self.nn
        m = 2 * rad + 1
        dev = X.device
        coord = torch.stack(torch.meshgrid(*[torch.arange(q, device=dev) for q in nn], indexing="ij"), -1)
        coord = coord.permute(*reversed(range(d)), d).reshape(-1, d)
        A = torch.zeros(self.N, m ** d, nb, nb, dtype=X.dtype, device=dev)
        rows = torch.arange(self.N, device=dev)
        for res in np.ndindex(*([m] * d)):
            col = (coord % m == torch.as_tensor(res, device=dev)).all(1)
            # the offset from each row to its one coloured column in reach
            o = torch.zeros(self.N, dtype=torch.long, device=dev)
            for k in range(d):
                o = o * m + (res[k] - coord[:, k] + rad) % m
            for j in range(nb):
                t = torch.zeros_like(X)
                t[col, j] = 1.0
                t.masked_fill_(self.fixed, 0.0)
                _, y = torch.func.jvp(self.residual, (X,), (t,))
                A[rows, o, :, j] = y
        c = m ** d // 2
        for i in range(nb):
            A[:, c, i, i] = torch.where(self.fixed[:, i], torch.ones_like(A[:, c, i, i]), A[:, c, i, i])
        return A

    def solve(self):
        X, nb = self.X0, self.d + 1
        r0 = prev = A = None
        for _ in range(14):
            R = self.residual(X)
            nrm = float(R.norm())
            if r0 is None:
                r0 = nrm
            elif nrm == 0.0 or (prev <= 1e-6 * r0 and nrm > 0.5 * prev):
                break
            prev = nrm
            if nrm < 1e-5 * r0 and A is not None:  # close by: the last matrix contracts fast enough
                X = X + D * self.stencil_solve(A, -(R * D).reshape(-1, 1), nb).reshape(-1, nb)
                continue
            A = self.jacobian(X)
            D = A[:, (2 * self.rad + 1) ** self.d // 2].diagonal(dim1=1, dim2=2).abs().sqrt()
            D = torch.where(D > 0, 1.0 / D, torch.ones_like(D))
            A = A * D[:, None, :, None]
            # column scaling: D of the column's node
            cols = self.columns()
            A = A * D[cols][:, :, None, :]
            y = self.stencil_solve(A, -(R * D).reshape(-1, 1), nb).reshape(-1, nb)
            X = X + D * y
        return X

    def columns(self):
        d, rad, nn = self.d, self.rad, self.nn
        dev = self.X0.device
        coord = torch.stack(torch.meshgrid(*[torch.arange(q, device=dev) for q in nn], indexing="ij"), -1)
        coord = coord.permute(*reversed(range(d)), d).reshape(-1, d)
        out = []
        for off in np.ndindex(*([2 * rad + 1] * d)):
            c, st = 0, 1
            for k in range(d):
                c, st = c + (coord[:, k] + off[k] - rad).clamp(0, nn[k] - 1) * st, st * nn[k]
            out.append(c)
        return torch.stack(out, 1)

    def update(self, X):
        """Stages 3-4 (Sec. 3.5)."""
        w, d = self.w, self.d
        Xq = X[self.idx]
        du = torch.einsum("qs,qsi->qi", self.S, Xq[:, :, :d])
        F = torch.eye(d, dtype=X.dtype, device=X.device) + torch.einsum("qsi,qsk->qik", Xq[:, :, :d], self.Gn)
        ev, Q = torch.linalg.eigh((F.transpose(1, 2) @ F).cpu())
        U = torch.einsum("qkm,qm->qk", Q * Q, ev.sqrt()).to(X.device)
        out = {"x": self.x + du, "u": du, "p": (self.S * Xq[:, :, d]).sum(1),
               "F": F.reshape(-1, d * d), "V": _det(F) * self.V, "lp": self.lp * U}
        if w.dynamic:
            acc, _, pd, pdd = self.newmark(X)
            to = lambda f: (self.S * f[self.idx]).sum(1)  # noqa: E731
            out["a"] = torch.stack([to(acc[:, k]) for k in range(d)], 1)
            out["v"] = self.v0 + w.dt * w.gamma * out["a"]
            out["pd"], out["pdd"] = to(pd), to(pdd)
        return {k: t.cpu().numpy() for k, t in out.items()}


def _exact_step(w, t0=0.0):
    if w.dim == 3 and (w.n > 12000 or w.model == I.MODEL_HENCKY):
        return None
    s = _ExactStep(w, t0)
    if s.cost > EXACT_COST or s.evals > EXACT_EVALS:
        return None
    return s.update(s.solve())
