"""Performance cases of the SQ library: the calls its users make, over the sizes they make them at.

A case is a dict of plain values. `prepare` makes what a program holds before the call (handles,
host inputs, a server), `run` is one pass through the public entry points, `exact` recomputes the
pass in 64 bits with plain torch (dense 1-D difference matrices, dense projector rows), sharing no
code with the library, and `work` counts what a pass cannot do without.

SQ_MIXED computes its columns and projections in FP32, so a program keeps its density and stress as
FP32 tensors; those passes return FP32. SQ_FP64 passes return FP64.
"""
import math
import time

import numpy as np
import torch

from paper_2006_03697_gb300 import sq

DENSITY = 0.0375          # H atoms per bohr^3 of the batched and served snapshots
KT = 3.17                 # Ha, hydrogen at 10^6 K
CHEB_M = 2048             # Chebyshev-Gauss points of the coefficients
LANCZOS_K = 40            # the library's default Lanczos steps
EXACT_BYTES = 2.5e13      # projector-row traffic above which the 64-bit recomputation takes too long


def _case(name, kind, n, h, n_o, atoms, proj, r_cut, n_pl, precision, bounds="lanczos", **more):
    return dict(name=name, kind=kind, nx=n[0], ny=n[1], nz=n[2], h=h, n_o=n_o, atoms=atoms, proj=proj, r_cut=r_cut,
                n_pl=n_pl, precision=precision, bounds=bounds, **more)


def listed():
    return [
        # a program that evaluates one small cell once: set up, evaluate, destroy; latency and launches
        _case("oneshot_2H_5x4x6_fp64", "oneshot", (5, 4, 6), 0.7, 2, 2, "sp", 1.5, 12, "fp64"),
        # a quantum-MD program on the small FP64 workload: two successive snapshots on one resident handle
        _case("trajectory_8H_12cube_fp64", "trajectory", (12, 12, 12), 0.5, 3, 8, "s", 3.0, 30, "fp64"),
        # the same program in reduced precision
        _case("trajectory_8H_12cube_mixed", "trajectory", (12, 12, 12), 0.5, 3, 8, "s", 3.0, 30, "mixed"),
        # the headline workload: one whole evaluation of 64 H with a 12th-order stencil
        _case("snapshot_64H_40cube_mixed", "evaluate", (40, 40, 40), 0.3, 6, 64, "sp", 4.0, 60, "mixed"),
        # the smallest class of the batched snapshots (32 H), on its own
        _case("snapshot_32H_32cube_mixed", "evaluate", (32, 32, 32), 0.3, 6, 32, "sp", 3.0, 44, "mixed"),
        # FP64 reference run of a ragged cell with the 12th-order stencil, spectral bounds known beforehand
        _case("snapshot_3H_15x13x11_fp64", "evaluate", (15, 13, 11), 0.3, 6, 3, "sp", 3.3, 41, "fp64", "given"),
        # one SCF iteration: atoms fixed (lists kept), a new V_eff
        _case("scf_4H_16cube_mixed", "scf", (16, 16, 16), 0.3, 6, 4, "sp", 3.0, 50, "mixed"),
        # Sec. 4 to the letter: every node's own spectral bounds
        _case("per_node_8H_12cube_mixed", "evaluate", (12, 12, 12), 0.5, 3, 8, "s", 3.0, 30, "mixed", "per_node"),
        # the Gauss SQ density inside an SCF iteration
        _case("gauss_8H_12cube_mixed", "gauss", (12, 12, 12), 0.5, 3, 8, "s", 3.0, 30, "mixed", k=30),
        # one CUDA graph over uneven snapshots
        _case("batch_4_uneven_mixed", "batch", (10, 12, 13), 0.3, 6, 2, "sp", 2.4, 30, "mixed", members=4),
        # the request loop: successive snapshots of a few resident trajectories
        _case("served_3x2_uneven_mixed", "served", (11, 10, 12), 0.35, 4, 2, "sp", 2.5, 32, "mixed", members=3),
        # Green-Kubo viscosity of a served stress stream
        dict(name="viscosity_6x2001", kind="viscosity", traj=6, steps=2001, max_lag=800, dt=20.0, h=0.3, nx=40),
    ]


def draw(rng):
    kind = rng.choice(["oneshot", "trajectory", "trajectory", "evaluate", "evaluate", "evaluate", "scf", "per_node", "gauss",
                       "batch", "served", "viscosity"])
    if kind == "viscosity":
        steps = int(2 ** rng.uniform(7, 12))
        return dict(kind=kind, traj=rng.randint(1, 12), steps=steps, max_lag=rng.randint(1, steps // 2),
                    dt=rng.uniform(5.0, 40.0), h=0.3, nx=rng.randint(16, 80))
    precision = rng.choice(["fp64", "mixed", "mixed"]) if kind in ("oneshot", "trajectory", "evaluate", "gauss") else "mixed"
    dense = kind in ("per_node", "gauss")        # Krylov vectors of every node
    top = 14 if dense else 7 if kind == "oneshot" else 15 if kind in ("batch", "served") else 18 if precision == "fp64" else 34
    low = 4 if kind == "oneshot" else 8
    while True:
        size = low * (top / low) ** rng.random()
        n = [max(3, int(round(size * rng.uniform(0.8, 1.15)))) for _ in range(3)]
        n_o = rng.choice([2, 3, 4, 6, 6])
        h = rng.uniform(0.45, 0.7) if n_o <= 3 else rng.uniform(0.28, 0.4)
        r_cut = h * (rng.uniform(2.0, 4.5) if kind == "oneshot" else rng.uniform(5.0, 13.2))
        n_pl = rng.randint(10, 30) if kind == "oneshot" else rng.randint(24, 80)
        m = math.floor(r_cut / h + 1e-9)
        cost = n[0] * n[1] * n[2] * (2 * m + 1) ** 3 * (200 if dense else n_pl) * (12 if precision == "fp64" else 1)
        if cost <= (4e9 if dense else 6e9 if kind in ("batch", "served") else 2e10):
            break
    atoms = max(1, int(round(DENSITY * n[0] * n[1] * n[2] * h ** 3 * rng.uniform(0.7, 1.2))))
    more = {}
    bounds = "lanczos"
    if kind == "per_node":
        kind, bounds = "evaluate", "per_node"
    elif kind == "evaluate":
        bounds = rng.choice(["lanczos", "lanczos", "given"])
    elif kind == "gauss":
        more["k"] = rng.randint(12, 40)
    elif kind in ("batch", "served"):
        more["members"] = rng.randint(2, 4)
    c = _case("", kind, n, h, n_o, atoms, rng.choice(["s", "sp", "sp"]), r_cut, n_pl, precision, bounds, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------ inputs
def _positions(rng, atoms, L):
    """Uniform positions, at least 0.8 bohr apart while that can be had."""
    out = np.zeros((0, 3))
    tries = 0
    while len(out) < atoms:
        x = rng.uniform(0.0, 1.0, 3) * L
        d = out - x
        d -= L * np.round(d / L)
        tries += 1
        if tries > 200 * atoms or not len(out) or np.min(np.sum(d * d, axis=1)) >= 0.64:
            out = np.vstack([out, x])
    return out


def _v_eff(L, n, pos):
    """Periodic sum of Gaussian wells (depth 2 Ha, width 0.6 bohr) centred on the atoms, x fastest."""
    fac = []
    for a in range(3):
        x = np.arange(n[a]) * (L[a] / n[a])
        reach = int(math.ceil(6.0 / L[a])) + 1
        d = x[None, :, None] - pos[:, a][:, None, None] - L[a] * np.arange(-reach, reach + 1)[None, None, :]
        fac.append(np.exp(-d * d / 0.72).sum(axis=2))
    plane = (fac[2][:, :, None] * fac[1][:, None, :]).reshape(len(pos), -1)
    return -2.0 * (plane.T @ fac[0]).reshape(-1)


def _instance(case, rng, member=0):
    """One problem instance; further members of a batch or stream are larger and shorter or longer."""
    n = np.array([case["nx"], case["ny"], case["nz"]]) + np.array([2, 1, 3]) * member
    L = n * case["h"]
    atoms = case["atoms"] + member
    pos = _positions(rng, atoms, L)
    proj = [dict(l=0, width=0.5, gamma=1.0, rcut=3.5)]
    if case["proj"] == "sp":
        proj.append(dict(l=1, width=0.5, gamma=0.5, rcut=3.5))
    return dict(L=L, n=n, n_o=case["n_o"], pos=pos, v_eff=_v_eff(L, n, pos), species=np.zeros(atoms, dtype=np.int64),
                proj=[proj], kT=KT * (1.0 + 0.2 * member), n_e=float(atoms), r_cut=case["r_cut"] + 0.4 * case["h"] * member,
                n_pl=case["n_pl"] + 5 * member, M=CHEB_M)


def _moved(inst, rng):
    pos = np.mod(inst["pos"] + rng.normal(0.0, 0.05, inst["pos"].shape), inst["L"])
    return dict(inst, pos=pos, v_eff=_v_eff(inst["L"], inst["n"], pos))


def _given_bounds(case):
    """An interval that holds every spectrum of the ranges used here (the caller knows the bounds)."""
    top = {2: 5.34, 3: 6.05, 4: 6.51, 6: 7.08}[case["n_o"]]
    return (-14.0, 1.5 * top / case["h"] ** 2 + 12.0)


def _problems(case, seed):
    """The instances of a pass, in order."""
    rng = np.random.default_rng([int(seed), 20060303])
    kind = case["kind"]
    if kind in ("oneshot", "evaluate", "gauss"):
        return [_instance(case, rng)]
    if kind == "trajectory":
        a = _instance(case, rng)
        return [a, _moved(a, rng)]
    if kind == "scf":
        a = _instance(case, rng)
        return [dict(a, v_eff=a["v_eff"] * (1.0 + 0.05 * rng.random(a["v_eff"].shape)))]
    first = [_instance(case, rng, m) for m in range(case["members"])]
    return first if kind == "batch" else first + [_moved(a, rng) for a in first]


def _stress_series(case, seed):
    rng = np.random.default_rng([int(seed), 3697])
    x = rng.standard_normal((case["traj"], case["steps"], 3, 3))
    for t in range(1, case["steps"]):                     # correlated in time, as a trajectory's stress is
        x[:, t] = 0.97 * x[:, t - 1] + 0.243 * x[:, t]
    return 2e-3 * (x + np.swapaxes(x, 2, 3)) + 0.4 * np.eye(3)


# ------------------------------------------------------------------------------------ a pass
class _Owner:
    """Owns the library objects of a state and gives them back with it."""

    def __init__(self):
        self.handles, self.batch, self.server, self.streams = [], None, None, []

    def __del__(self):
        if self.server is not None:
            self.server.close()
        if self.batch is not None:
            self.batch.close()
        for h in self.handles:
            sq.sq_destroy(h)


def _precision(case):
    return sq.SQ_FP64 if case["precision"] == "fp64" else sq.SQ_MIXED


def _bounds_arg(case):
    return _given_bounds(case) if case["bounds"] == "given" else None if case["bounds"] == "lanczos" else case["bounds"]


def prepare(case, seed):
    s = {"case": case, "own": _Owner()}
    if case["kind"] == "viscosity":
        s["sigma"] = _stress_series(case, seed)
        return s
    probs = s["probs"] = _problems(case, seed)
    own, prec, kind = s["own"], _precision(case), case["kind"]
    if kind == "oneshot":
        pass
    elif kind == "served":
        s["descs"] = [sq.Desc(p, prec) for p in probs]
        own.server = sq.Server(hbm_budget_bytes=32 << 30, max_inflight=4)
    elif kind == "batch":
        for p in probs:
            own.streams.append(torch.cuda.Stream())
            own.handles.append(sq.sq_setup(sq.Desc(p, prec, stream=own.streams[-1].cuda_stream)))
        own.batch = sq.Batch(own.handles)
    else:
        own.handles.append(sq.sq_setup(sq.Desc(probs[0], prec, bounds=_bounds_arg(case))))
        if kind == "scf":
            sq.sq_keep_lists(own.handles[0], True)
    return s


def _out(case, mu, en, sigma, pressure=None, e_pot=None, rho=None):
    t = np.float64 if case["precision"] == "fp64" else np.float32
    energies = [en[k] for k in ("E_band", "E_s", "E_nl", "F", "N_check")] + ([] if e_pot is None else [e_pot])
    stress = list(np.asarray(sigma).reshape(9)) + ([] if pressure is None else [pressure])
    out = {"mu": t(mu), "energies": np.array(energies, dtype=t), "stress": np.array(stress, dtype=t)}
    if rho is not None:
        out["rho"] = np.asarray(rho).astype(t)
    return out


def _evaluate(case, h, nd):
    sq.sq_moments(h)
    mu = sq.sq_fermi_level(h)
    rho, en, sigma = sq.sq_density_energy_stress(h, mu, nd)
    p, e_pot = sq.sq_pressure(h, mu)
    return _out(case, mu, en, sigma, p, e_pot, rho)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "viscosity":
        volume = (case["h"] * case["nx"]) ** 3
        eta, acf = sq.sq_green_kubo(s["sigma"], case["dt"], volume, KT, case["max_lag"])
        return {"eta": eta, "acf": acf}
    probs, own = s["probs"], s["own"]
    nd = int(np.prod(probs[0]["n"]))
    if kind == "oneshot":
        r = sq.run(probs[0], _precision(case), bounds=_bounds_arg(case))
        return _out(case, r["mu"], r, r["sigma"], r["pressure_A"], r["E_pot"], r["rho"])
    if kind == "served":
        for i, d in enumerate(s["descs"]):
            own.server.submit(d, tag=i, traj=i % case["members"])
        got = []
        while len(got) < len(s["descs"]):
            got += own.server.poll(timeout_ms=1000)
        got.sort(key=lambda r: r["tag"])
        for r in got:
            if r["status"] != 0:
                raise RuntimeError(r["error"])
        return [_out(case, r["mu"], r, r["sigma"]) for r in got]
    if kind == "batch":
        mu, en, sigma = own.batch.run()
        return [_out(case, mu[i], en[i], sigma[i]) for i in range(len(probs))]
    h = own.handles[0]
    if kind == "gauss":
        t = np.float64 if case["precision"] == "fp64" else np.float32
        mu, rho, e_band = sq.sq_gauss_density(h, case["k"], nd)
        return {"mu": t(mu), "rho": rho.astype(t), "E_band": t(e_band)}
    if kind == "evaluate":
        return _evaluate(case, h, nd)
    out = []
    for p in probs:                                       # trajectory: both snapshots; scf: the new V_eff
        sq.sq_update_atoms(h, p["pos"], p["v_eff"])
        out.append(_evaluate(case, h, nd))
    return out


# ------------------------------------------------------------------------------------ work
def _rows_per_point(p):
    """Projector channels whose sphere holds a point, on average."""
    ch = sum(2 * q["l"] + 1 for q in p["proj"][0])
    return ch * len(p["pos"]) / float(np.prod(p["L"])) * 4.0 / 3.0 * math.pi * 3.5 ** 3


def work(case):
    """Bytes: host inputs and results once. Flops: per node, region point and step the Laplacian, V, the
    update, both projector contractions and the nonlocal-stress contraction (Gauss: the Laplacian, V,
    the projectors and one orthogonalisation against the Krylov vectors held)."""
    if case["kind"] == "viscosity":
        n, lags = case["traj"] * case["steps"], case["max_lag"] + 1
        return {"bytes": 72.0 * n + 16.0 * lags, "flops": 10.0 * case["traj"] * sum(case["steps"] - k for k in range(lags))}
    total_b = total_f = 0.0
    for p in _problems(case, 0):
        nd = float(np.prod(p["n"]))
        m = np.floor(p["r_cut"] / (p["L"] / p["n"]) + 1e-9)
        pts = nd * float(np.prod(2 * m + 1))
        rows = _rows_per_point(p)
        per_h = 2.0 * 6 * p["n_o"] + 4 + 4 * rows
        if case["kind"] == "gauss":
            total_f += pts * case["k"] * (per_h + 2.0 * case["k"])
        else:
            total_f += pts * p["n_pl"] * (per_h + 3 + 18)
        if case["bounds"] == "per_node":
            total_f += pts * LANCZOS_K * (per_h + 2.0 * LANCZOS_K)
        total_b += 8.0 * (nd + 3 * len(p["pos"])) + 8.0 * (nd + 17)
    return {"bytes": total_b, "flops": total_f}


# ------------------------------------------------------------------------------------ 64 bits
class _Region:
    """H_q of a group of nodes (q: [B, 3] lattice coordinates) in 64 bits: dense 1-D difference
    matrices on the region, V_eff gathered, every projector row that meets the regions stored."""

    def __init__(self, p, q):
        dev = "cuda"
        self.B = len(q)
        n, L = p["n"], p["L"]
        h = L / n
        m = np.floor(p["r_cut"] / h + 1e-9).astype(int)
        self.m, self.dV, n_o = m, float(np.prod(h)), p["n_o"]
        w, g = np.zeros(n_o + 1), np.zeros(n_o + 1)
        for i in range(1, n_o + 1):
            base = math.factorial(n_o) ** 2 / (math.factorial(n_o - i) * math.factorial(n_o + i))
            w[i] = 2.0 * (-1.0) ** (i + 1) * base / i ** 2
            g[i] = (-1.0) ** (i + 1) * base / i
        w[0] = -2.0 * w.sum()
        self.D, self.G = [], []
        for a in range(3):
            W = 2 * m[a] + 1
            D, G = w[0] * np.eye(W), np.zeros((W, W))
            for i in range(1, n_o + 1):
                up, dn = np.eye(W, k=i), np.eye(W, k=-i)
                D += w[i] * (up + dn)
                G += g[i] * (up - dn)
            self.D.append(torch.tensor(-0.5 * D / h[a] ** 2, device=dev))
            self.G.append(torch.tensor(G / h[a], device=dev))
        self.shape = tuple(int(2 * m[2 - a] + 1) for a in range(3))          # z, y, x
        self.nc = int(np.prod(self.shape))
        lat = [torch.tensor(q[:, a][:, None] + np.arange(-m[a], m[a] + 1)[None, :], device=dev) for a in range(3)]
        v = torch.tensor(p["v_eff"], device=dev).reshape(int(n[2]), int(n[1]), int(n[0]))
        ix = [lat[a] % int(n[a]) for a in range(3)]
        self.V = v[ix[2][:, :, None, None], ix[1][:, None, :, None], ix[0][:, None, None, :]]
        # atom images whose support sphere meets the union box of the regions
        lo, hi = (q.min(axis=0) - m) * h, (q.max(axis=0) + m) * h
        rc = 3.5
        R = []
        for pos in p["pos"]:
            sh = [range(int(math.floor((lo[a] - rc - pos[a]) / L[a])), int(math.ceil((hi[a] + rc - pos[a]) / L[a])) + 1)
                  for a in range(3)]
            for sx in sh[0]:
                for sy in sh[1]:
                    for sz in sh[2]:
                        c = pos + L * np.array([sx, sy, sz])
                        d = np.maximum(0.0, np.maximum(lo - c, c - hi))
                        if d @ d <= rc * rc:
                            R.append(c)
        self.X = None
        chans = [(pj["l"], c, pj["width"], pj["gamma"]) for pj in p["proj"][0] for c in range(2 * pj["l"] + 1)]
        self.W = torch.zeros(3, self.B, self.nc, dtype=torch.float64, device=dev)
        self.W0 = torch.zeros(self.B, self.nc, dtype=torch.float64, device=dev)
        if R:
            R = torch.tensor(np.array(R), device=dev)
            d = [lat[a].double()[:, None, :] * h[a] - R[None, :, a, None] for a in range(3)]      # [B, I, W_a]
            dd = [d[0][:, :, None, None, :], d[1][:, :, None, :, None], d[2][:, :, :, None, None]]
            r2 = dd[0] ** 2 + dd[1] ** 2 + dd[2] ** 2
            inside = r2 <= rc * rc
            self.X = torch.empty(self.B, len(R), len(chans), self.nc, dtype=torch.float64, device=dev)
            at_q = torch.empty(self.B, len(R), len(chans), dtype=torch.float64, device=dev)
            for c, (l, ch, width, _) in enumerate(chans):
                val = (math.pi * width * width) ** -0.75 * torch.exp(-r2 / (2 * width * width)) * inside
                if l == 1:
                    val = val * (math.sqrt(2.0) / width) * dd[ch]
                self.X[:, :, c] = val.reshape(self.B, len(R), -1)
                at_q[:, :, c] = val[:, :, m[2], m[1], m[0]]
            self.gam = torch.tensor([c[3] for c in chans], dtype=torch.float64, device=dev) * self.dV
            ag = at_q * self.gam
            for a in range(3):                            # W_a = sum_rows gamma dV chi(x_q) chi (x - R)_a
                da = dd[a].expand(self.B, len(R), *self.shape).reshape(self.B, len(R), -1)
                self.W[a] = (torch.einsum("bic,bicu->biu", ag, self.X) * da).sum(dim=1)
            rows = len(R) * len(chans)
            self.X = self.X.reshape(self.B, rows, self.nc)
            self.gam = self.gam.repeat(len(R))
            self.W0 = torch.bmm(ag.reshape(self.B, 1, rows), self.X)[:, 0]

    def axis(self, M, a, t):
        t = t.reshape(self.B, *self.shape)
        if a == 0:
            r = t @ M.T
        elif a == 1:
            r = torch.matmul(M, t)
        else:
            r = torch.matmul(M, t.reshape(self.B, self.shape[0], -1))
        return r.reshape(self.B, self.nc)

    def H(self, t):
        y = self.V.reshape(self.B, -1) * t
        for a in range(3):
            y = y + self.axis(self.D[a], a, t)
        if self.X is not None:
            P = torch.bmm(self.X, t[:, :, None]) * self.gam[None, :, None]
            y = y + torch.bmm(P.transpose(1, 2), self.X)[:, 0]
        return y

    def unit(self):
        t = torch.zeros(self.B, *self.shape, dtype=torch.float64, device="cuda")
        t[:, self.m[2], self.m[1], self.m[0]] = 1.0
        return t.reshape(self.B, self.nc)

    def moments(self, t):
        """rho, K (xx yy zz yz xz xy), N, S (row-major) of every node of the group: [B, 17]."""
        c = [int(x) for x in self.m]
        u = t.reshape(self.B, *self.shape)
        row = [self.G[a][c[a]] for a in range(3)]
        line = [u[:, c[2], c[1], :], u[:, c[2], :, c[0]], u[:, :, c[1], c[0]]]
        out = [u[:, c[2], c[1], c[0]]]
        out += [line[a] @ (row[a] @ self.G[a]) for a in range(3)]
        out.append(torch.einsum("z,bzy,y->b", row[2], u[:, :, :, c[0]], row[1]))
        out.append(torch.einsum("z,bzx,x->b", row[2], u[:, :, c[1], :], row[0]))
        out.append(torch.einsum("y,byx,x->b", row[1], u[:, c[2], :, :], row[0]))
        out.append((self.W0 * t).sum(dim=1))
        for a in range(3):
            ga = self.axis(self.G[a], a, t)
            out += [(self.W[b] * ga).sum(dim=1) for b in range(3)]
        return torch.stack(out, dim=1)

    def lanczos(self, v, k):
        """alpha, beta [B, k] and the steps taken per column (classical Gram-Schmidt applied twice)."""
        k = min(k, self.nc)
        alpha, beta = np.zeros((self.B, k)), np.zeros((self.B, k))
        keff = np.zeros(self.B, dtype=int)
        basis = [v / v.norm(dim=1, keepdim=True)]
        for i in range(k):
            w = self.H(basis[i])
            Q = torch.stack(basis, dim=1)
            a = 0.0
            for _ in range(2):
                c = torch.bmm(Q, w[:, :, None])
                w = w - torch.bmm(c.transpose(1, 2), Q)[:, 0]
                a = a + c[:, i, 0]
            b = w.norm(dim=1)
            alpha[:, i], beta[:, i] = a.cpu().numpy(), b.cpu().numpy()
            stop = (keff == 0) & ((beta[:, i] <= 1e-12 * np.maximum(1.0, np.abs(alpha[:, i]))) | (i == k - 1))
            keff[stop] = i + 1
            if (keff > 0).all():
                break
            basis.append(w / torch.clamp(b, min=1e-300)[:, None])
        return alpha, beta, keff

    def start(self, q, n):
        """The library's Lanczos start vectors: 1 + (hash(point, node) mod 1009) / 1009."""
        i = np.arange(self.nc, dtype=np.uint64)[None, :] * np.uint64(2654435761)
        node = (q[:, 0] + n[0] * (q[:, 1] + n[1] * q[:, 2])).astype(np.uint64)[:, None] * np.uint64(40503)
        hsh = (i + node) & np.uint64(0xFFFFFFFF)
        return torch.tensor(1.0 + (hsh % np.uint64(1009)).astype(np.float64) / 1009.0, device="cuda")


def _groups(n, side):
    for z in range(0, n[2], side):
        for y in range(0, n[1], side):
            for x in range(0, n[0], side):
                yield np.array([(i, j, k) for k in range(z, min(z + side, n[2])) for j in range(y, min(y + side, n[1]))
                                for i in range(x, min(x + side, n[0]))])


def _tridiagonal(alpha, beta, n):
    return np.linalg.eigh(np.diag(alpha[:n]) + np.diag(beta[:n - 1], 1) + np.diag(beta[:n - 1], -1))


def _interval(alpha, beta, keff):
    """Ritz extremes of each column, widened by their residual norms."""
    lo, hi = np.zeros(len(keff)), np.zeros(len(keff))
    for c, n in enumerate(keff):
        th, Y = _tridiagonal(alpha[c], beta[c], n)
        lo[c] = th[0] - beta[c, n - 1] * abs(Y[-1, 0])
        hi[c] = th[-1] + beta[c, n - 1] * abs(Y[-1, -1])
    return lo, hi


def _shared_interval(p):
    """Lanczos on the nodes of the 2x2x2 blocks that hold argmin V, argmax V and a stride-n/2 grid."""
    n, v = p["n"], p["v_eff"]
    grid = [range(0, int(n[a]), max(1, int(n[a]) // 2)) for a in range(3)]
    seeds = [int(np.argmin(v)), int(np.argmax(v))] + [x + n[0] * (y + n[1] * z) for z in grid[2] for y in grid[1] for x in grid[0]]
    blocks = {(q % n[0] // 2, q // n[0] % n[1] // 2, q // (n[0] * n[1]) // 2) for q in seeds}
    lo, hi = math.inf, -math.inf
    for b in blocks:
        q = np.array([(2 * b[0] + i, 2 * b[1] + j, 2 * b[2] + k) for k in (0, 1) for j in (0, 1) for i in (0, 1)])
        q = q[(q < n).all(axis=1)]
        r = _Region(p, q)
        l, u = _interval(*r.lanczos(r.start(q, n), LANCZOS_K))
        lo, hi = min(lo, l.min()), max(hi, u.max())
    return lo - 0.01 * (hi - lo), hi + 0.01 * (hi - lo)


def _bisect(count, lo, hi, n_e):
    lo, hi = lo - 40.0 * KT, hi + 40.0 * KT
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if count(mid) < n_e else (lo, mid)
        if hi - lo < 1e-13 * max(1.0, abs(mid)):
            break
    return 0.5 * (lo + hi)


def _fermi(x):
    e = torch.exp(-x.abs())
    return torch.where(x > 0, e / (1 + e), 1 / (1 + e))


def _too_long(p, steps):
    m = np.floor(p["r_cut"] / (p["L"] / p["n"]) + 1e-9)
    ch = sum(2 * q["l"] + 1 for q in p["proj"][0])
    rows = ch * len(p["pos"]) / float(np.prod(p["L"])) * float(np.prod((2 * m + 1) * (p["L"] / p["n"]) + 6.0))
    return float(np.prod(p["n"])) * float(np.prod(2 * m + 1)) * (rows + 12) * 16.0 * steps > EXACT_BYTES


def _exact_evaluation(case, p, full):
    """mu, energies, stress (and rho) of one instance in 64 bits; full: with pressure, E_pot and rho."""
    n, n_pl, kT = p["n"], p["n_pl"], p["kT"]
    nd, dV, vol = int(np.prod(n)), float(np.prod(p["L"] / n)), float(np.prod(p["L"]))
    shared = None
    if case["bounds"] == "given":
        shared = _given_bounds(case)
    elif case["bounds"] == "lanczos":
        shared = _shared_interval(p)
    mom = torch.zeros(nd, n_pl + 1, 17, dtype=torch.float64, device="cuda")
    lo, hi = np.zeros(nd), np.zeros(nd)
    for q in _groups([int(x) for x in n], 4):
        r = _Region(p, q)
        idx = q[:, 0] + n[0] * (q[:, 1] + n[1] * q[:, 2])
        if shared is None:
            l, u = _interval(*r.lanczos(r.start(q, n), LANCZOS_K))
            lo[idx], hi[idx] = l - 0.01 * (u - l), u + 0.01 * (u - l)
        else:
            lo[idx], hi[idx] = shared
        chi = torch.tensor(0.5 * (lo[idx] + hi[idx]), device="cuda")[:, None]
        zeta = torch.tensor(0.5 * (hi[idx] - lo[idx]), device="cuda")[:, None]
        where = torch.tensor(idx, device="cuda")
        prev, t = None, r.unit()
        for j in range(n_pl + 1):
            mom[where, j] = r.moments(t)
            if j < n_pl:
                nxt = (r.H(t) - chi * t) / zeta
                if prev is not None:
                    nxt = 2.0 * nxt - prev
                prev, t = t, nxt
    one = shared is not None                              # one interval: one set of coefficients
    chi = torch.tensor((0.5 * (lo + hi))[:1] if one else 0.5 * (lo + hi), device="cuda")[:, None]
    zeta = torch.tensor((0.5 * (hi - lo))[:1] if one else 0.5 * (hi - lo), device="cuda")[:, None]
    theta = math.pi * (torch.arange(CHEB_M, device="cuda", dtype=torch.float64) + 0.5) / CHEB_M
    cosj = torch.cos(torch.arange(n_pl + 1, device="cuda", dtype=torch.float64)[:, None] * theta[None, :])
    lam = chi + zeta * torch.cos(theta)[None, :]
    half = torch.ones(n_pl + 1, device="cuda", dtype=torch.float64)
    half[0] = 0.5
    rho_j = (mom[:, :, 0].sum(dim=0, keepdim=True) if one else mom[:, :, 0]) * half
    F = rho_j @ cosj
    mu = _bisect(lambda x: float(4.0 / CHEB_M * (_fermi((lam - x) / kT) * F).sum()), lo.min(), hi.max(), p["n_e"])
    x = (lam - mu) / kT
    e = torch.exp(-x.abs())
    ent = -(torch.log1p(e) + x.abs() * e / (1 + e))
    coef = [2.0 / CHEB_M * (f @ cosj.T) * half for f in (_fermi(x), torch.cos(theta)[None, :] * _fermi(x), ent)]
    c, d, s = [k.expand(nd, -1) for k in coef]
    tot = torch.einsum("qj,qjk->k", c, mom)
    r_q = (c * mom[:, :, 0]).sum(dim=1)
    E_band = float(2.0 * (((chi * c + zeta * d)) * mom[:, :, 0]).sum())
    E_s, E_nl = float(2.0 * kT * (s * mom[:, :, 0]).sum()), float(2.0 * tot[7])
    K, S = tot[1:7].cpu().numpy(), tot[8:17].cpu().numpy().reshape(3, 3)
    sig = 2.0 * np.array([[K[0], K[5], K[4]], [K[5], K[1], K[3]], [K[4], K[3], K[2]]])
    sig = (sig - 2.0 * (0.5 * E_nl * np.eye(3) + 2.0 * S)) / vol
    rho = (2.0 / dV * r_q).cpu().numpy()
    E_pot = dV * float(np.dot(p["v_eff"], rho))
    pressure = (2.0 * (E_band - E_pot) + E_nl + 4.0 * np.trace(S)) / (3.0 * vol)
    energies = [E_band, E_s, E_nl, E_band + E_s, dV * rho.sum()] + ([E_pot] if full else [])
    out = {"mu": np.float64(mu), "energies": np.array(energies),
           "stress": np.array(list(sig.reshape(9)) + ([pressure] if full else []))}
    if full:
        out["rho"] = rho
    return out


def _exact_gauss(case, p):
    n, nd, dV = p["n"], int(np.prod(p["n"])), float(np.prod(p["L"] / p["n"]))
    th, wt = np.zeros((nd, case["k"])), np.zeros((nd, case["k"]))
    for q in _groups([int(x) for x in n], 4):
        r = _Region(p, q)
        idx = q[:, 0] + n[0] * (q[:, 1] + n[1] * q[:, 2])
        alpha, beta, keff = r.lanczos(r.unit(), case["k"])
        for c, k in enumerate(keff):
            e, Y = _tridiagonal(alpha[c], beta[c], k)
            th[idx[c], :k], wt[idx[c], :k] = e, Y[0] ** 2
    t, w = torch.tensor(th, device="cuda"), torch.tensor(wt, device="cuda")
    mu = _bisect(lambda x: float(2.0 * (w * _fermi((t - x) / KT)).sum()), th[wt > 0].min(), th[wt > 0].max(), p["n_e"])
    f = w * _fermi((t - mu) / KT)
    return {"mu": np.float64(mu), "rho": (2.0 / dV * f.sum(dim=1)).cpu().numpy(), "E_band": np.float64(2.0 * (f * t).sum())}


def exact(case, seed):
    if case["kind"] == "viscosity":
        sig = _stress_series(case, seed)
        s = np.stack([sig[..., 0, 1], sig[..., 1, 2], sig[..., 2, 0], 0.5 * (sig[..., 0, 0] - sig[..., 1, 1]),
                      0.5 * (sig[..., 1, 1] - sig[..., 2, 2])], axis=-1)
        acf = np.array([np.mean(np.sum(s[:, : case["steps"] - k] * s[:, k:], axis=-1)) / 5.0
                        for k in range(case["max_lag"] + 1)])
        volume = (case["h"] * case["nx"]) ** 3
        run_sum = np.concatenate([[0.0], np.cumsum(0.5 * case["dt"] * (acf[1:] + acf[:-1]))])
        return {"eta": volume / KT * run_sum, "acf": acf}
    probs = _problems(case, seed)
    began = time.monotonic()
    if any(_too_long(p, case.get("k", 0) or p["n_pl"] + 1) for p in probs):
        return None
    if case["kind"] == "gauss":
        return _exact_gauss(case, probs[0])
    full = case["kind"] not in ("batch", "served")
    got = []
    for p in probs:
        if time.monotonic() - began > 15.0:
            got.append(None)
            continue
        got.append(_exact_evaluation(case, p, full))
    return got[0] if case["kind"] in ("oneshot", "evaluate") else got
