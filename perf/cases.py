"""Performance cases of the framework: what a user's program runs, through the public API.

A case is a plain dict: `kind` names the workload (one of the paper's test problems, a batch, the
adjoint, the 3D extension, host buffers), the sizes are vertices (or segments) per direction,
`precision` is the path ("fp64", "fp32" bulk) and `steps` the SSP-RK3 steps of one pass.

  residual  one right-hand side R(U) of the isentropic vortex (hfd_residual): what an outer
            time integrator or a test calls
  vortex    import of a state, CFL steps, export (Sec. 3.1; periodic)
  quad      the same for the four-quadrant Riemann problem with transmissive ghost layers
  tgv       the viscous Taylor-Green vortex, fixed step (periodic)
  couette   viscous Couette channel with fixed wall bands, fixed step (Sec. 3.2)
  sod       circular Sod on a Delaunay mesh with an embedded circle (Sec. 3.3)
  batch     several uneven vortex meshes stepped together, one state array each (hfd_batch_step)
  adjoint   a rollout and its backward pass (autograd.rollout: hfd_step, hfd_adjoint)
  tube      the 3D extension, a vortex tube in a periodic tetrahedral box (hfd3_steps)
  host      steps on pinned host buffers, copies included (hfd_steps_host)

A mesh is laid out once (Plan) and serves every state of its case, as a program keeps it; the
states are drawn from the seed.
"""
import functools
import math

import numpy as np
import torch

import synth
from synth import three_d
from paper_2109_01286_gb300 import Batch, Mesh, Prep, hfd3d
from paper_2109_01286_gb300.autograd import rollout

GAMMA = 1.4
TGV = dict(viscous=True, mu=0.01, prandtl=0.72, R_gas=1.0 / (GAMMA * 0.01))       # Re 100, Mach 0.1
COUETTE = dict(viscous=True, mu=0.1, prandtl=100.0, R_gas=0.4 * 10.0 / 1.4)


def listed():
    return [
        # the smallest call: one right-hand side on a 24x24 mesh (launch latency)
        {"name": "residual 24 fp64", "kind": "residual", "nx": 24, "ny": 24, "precision": "fp64", "steps": 0},
        # the paper's coarsest vortex mesh (3957 nodes): a short output interval of CFL steps
        {"name": "vortex 63 fp64", "kind": "vortex", "nx": 63, "ny": 63, "precision": "fp64", "steps": 10},
        # the paper's finest vortex mesh (36408 nodes) on the FP32-bulk path
        {"name": "vortex 191 fp32", "kind": "vortex", "nx": 191, "ny": 191, "precision": "fp32", "steps": 5},
        # the benchmark's problem and default precision at a quarter of its vertices
        {"name": "quad 512 fp64", "kind": "quad", "nx": 512, "ny": 512, "precision": "fp64", "steps": 2},
        # the same on the FP32-bulk path
        {"name": "quad 512 fp32", "kind": "quad", "nx": 512, "ny": 512, "precision": "fp32", "steps": 2},
        # viscous rows on the FP32-bulk path, whose mixed-precision accuracy this problem measures
        {"name": "tgv 256 fp32", "kind": "tgv", "nx": 256, "ny": 256, "precision": "fp32", "steps": 4},
        # viscous rows in FP64 between walls, a ragged mesh of the Couette sizes
        {"name": "couette 105 fp64", "kind": "couette", "nx": 105, "ny": 106, "precision": "fp64", "steps": 4},
        # an unstructured (Delaunay) mesh with strong waves
        {"name": "sod 100 fp64", "kind": "sod", "nx": 100, "ny": 100, "precision": "fp64", "steps": 2},
        # many uneven meshes at once, each with its own CFL step
        {"name": "batch 8 fp64", "kind": "batch", "nx": 8, "ny": 0, "precision": "fp64", "steps": 1},
        # forward and backward through the time stepping
        {"name": "adjoint 160 fp64", "kind": "adjoint", "nx": 160, "ny": 160, "precision": "fp64", "steps": 4},
        # the 3D extension
        {"name": "tube 24 fp64", "kind": "tube", "nx": 24, "ny": 24, "nz": 24, "precision": "fp64", "steps": 2},
        # a caller whose states live on the host
        {"name": "host 200 fp64", "kind": "host", "nx": 200, "ny": 200, "precision": "fp64", "steps": 3},
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["residual", "vortex", "vortex", "quad", "quad", "tgv", "couette", "sod",
                       "batch", "adjoint", "tube", "host"])
    prec = rng.choice(["fp64", "fp64", "fp32"])
    n = side(17, 400)
    aspect = rng.uniform(0.6, 1.4)
    m = max(17, int(n * aspect))
    if kind == "residual":
        return {"kind": kind, "nx": n, "ny": m, "precision": prec, "steps": 0}
    if kind in ("vortex", "quad", "tgv"):
        return {"kind": kind, "nx": n, "ny": m, "precision": prec, "steps": rng.randint(1, 3)}
    if kind == "couette":
        return {"kind": kind, "nx": side(20, 160), "ny": side(20, 160), "precision": prec, "steps": rng.randint(1, 4)}
    if kind == "sod":
        n = side(24, 160)
        return {"kind": kind, "nx": n, "ny": n, "precision": prec, "steps": rng.randint(1, 2)}
    if kind == "batch":
        return {"kind": kind, "nx": rng.randint(2, 8), "ny": 0, "precision": prec, "steps": 1}
    if kind == "adjoint":
        return {"kind": kind, "nx": side(20, 180), "ny": side(20, 140), "precision": "fp64", "steps": rng.randint(1, 4)}
    if kind == "tube":
        return {"kind": kind, "nx": rng.randint(7, 24), "ny": rng.randint(7, 24), "nz": rng.randint(7, 24),
                "precision": "fp64", "steps": rng.randint(1, 2)}
    return {"kind": kind, "nx": side(17, 300), "ny": side(17, 300), "precision": prec, "steps": rng.randint(1, 3)}


# ------------------------------------------------------------------ meshes (laid out once a case)
def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "steps")))


def _members(case):
    """The first meshes of the batched workload (uneven sizes, log-uniform)."""
    every = synth.batched_vortices(n=8, seed=4, vmin=2e3, vmax=6.4e4)
    return [x["mesh"] for x in every[:case["nx"]]]


def _mesh_of(case):
    k, nx, ny = case["kind"], case["nx"], case["ny"]
    if k in ("residual", "vortex", "host", "adjoint"):
        return synth.jittered_grid(nx, ny, 10.0, 10.0 * ny / nx, seed=1), {}
    if k == "quad":
        return synth.jittered_box_with_ghosts(nx, ny, (0.0, 1.0), (0.0, 1.0), 5, seed=2), {}
    if k == "tgv":
        return synth.jittered_grid(nx, ny, 2 * np.pi, 2 * np.pi, seed=3), TGV
    if k == "couette":
        return synth.couette_channel(nx, ny, 6, seed=7), COUETTE
    if k == "sod":
        return synth.embedded_circle_box(nx, seed=8), {}
    raise ValueError(k)


class Plan:
    """What a program lays out once: the mesh (or batch of meshes) on the device."""

    def __init__(self, case):
        if case["kind"] == "tube":
            nx, ny, nz = case["nx"], case["ny"], case["nz"]
            self.mesh = three_d.periodic_tet_box(nx, ny, nz, 10.0, 10.0 * ny / nx, 10.0 * nz / nx, seed=3)
            self.dev = hfd3d.Mesh3(self.mesh)
        elif case["kind"] == "batch":
            self.mesh = _members(case)
            self.dev = Batch([Prep(m) for m in self.mesh], precision=case["precision"])
        else:
            self.mesh, opts = _mesh_of(case)
            self.dev = Mesh(self.mesh, precision=case["precision"], **opts)


@functools.lru_cache(maxsize=32)
def _plan_by_key(key):
    return Plan(dict(key))


def _plan(case):
    return _plan_by_key(_key(case))


# ------------------------------------------------------------------ states from the seed
def _states(case, mesh, seed):
    """The state(s) of a case as numpy arrays in input order, and the fixed step (0: CFL)."""
    rng = np.random.default_rng(seed)
    k = case["kind"]
    if k == "batch":
        return [synth.isentropic_vortex(m, beta=rng.uniform(2.0, 5.0), center=(0.5 * m["Lx"], 0.5 * m["Ly"]))
                for m in mesh], 0.0
    if k == "tube":
        c = (rng.uniform(0.3, 0.7) * mesh["Lx"], rng.uniform(0.3, 0.7) * mesh["Ly"])
        U = three_d.vortex_tube(mesh, beta=rng.uniform(2.0, 5.0), center=c, mean=(1.0, 1.0, rng.uniform(0.2, 0.8)))
        return U, 0.02 * mesh["Lx"] / case["nx"]
    if k in ("residual", "vortex", "host", "adjoint"):
        c = (rng.uniform(0.3, 0.7) * mesh["Lx"], rng.uniform(0.3, 0.7) * mesh["Ly"])
        U = synth.isentropic_vortex(mesh, beta=rng.uniform(2.0, 5.0), center=c,
                                    mean=(rng.uniform(0.5, 1.5), rng.uniform(0.5, 1.5)))
        return U, 0.05 * mesh["Lx"] / case["nx"] if k == "adjoint" else 0.0
    if k == "quad":
        U = synth.four_quadrant(mesh, xm=rng.uniform(0.4, 0.6), ym=rng.uniform(0.4, 0.6))
        U[:4] *= rng.uniform(0.8, 1.25)          # the Euler equations scale with the state
        return U, 0.0
    if k == "tgv":
        moved = dict(mesh, x=mesh["x"] + rng.uniform(0, 2 * np.pi), y=mesh["y"] + rng.uniform(0, 2 * np.pi))
        p0 = 1.0 / (GAMMA * 0.01)
        return synth.taylor_green(moved), 0.2 * (2 * np.pi / max(case["nx"], case["ny"])) / (1.0 + math.sqrt(GAMMA * p0))
    if k == "couette":
        U = synth.couette(mesh, u0=rng.uniform(0.8, 1.2), T_top=rng.uniform(11.0, 13.0))
        return U, 0.1 * (10.0 / max(case["nx"], case["ny"])) / 8.0
    if k == "sod":
        s = rng.uniform(0.8, 1.25)
        return synth.circular_sod(mesh, inside=(1.0, 0.0, 0.0, s)), 0.0
    raise ValueError(k)


def prepare(case, seed):
    plan = _plan(case)
    U, dt = _states(case, plan.mesh, seed)
    st = {"case": case, "plan": plan, "dt": dt}
    if case["kind"] == "batch":
        st["U0"] = [torch.from_numpy(u).cuda() for u in U]
        st["U"] = [torch.empty_like(u) for u in st["U0"]]
    elif case["kind"] == "host":
        st["U0"] = torch.from_numpy(U).pin_memory()
        st["U"] = torch.empty_like(st["U0"]).pin_memory()
    else:
        st["U0"] = torch.from_numpy(U).cuda()
        st["U"] = torch.empty_like(st["U0"])
        st["out"] = torch.empty_like(st["U0"])
    if case["kind"] == "residual":
        plan.dev.import_state(st["U0"], out=st["U"])
    if case["kind"] == "adjoint":
        st["U0"] = plan.dev.import_state(st["U0"]).requires_grad_(True)
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        st["grad"] = torch.randn(st["U0"].shape, dtype=torch.float64, device="cuda", generator=g)
    return st


def run(st):
    case, dev, dt = st["case"], st["plan"].dev, st["dt"]
    kind, steps = case["kind"], case["steps"]
    if kind == "residual":
        return dev.residual(st["U"], R=st["out"])
    if kind == "batch":
        torch._foreach_copy_(st["U"], st["U0"])
        for _ in range(steps):
            dev.step(st["U"])
        return st["U"]
    if kind == "adjoint":
        st["U0"].grad = None
        out = rollout(st["U0"], dev, dt, steps, 2)
        out.backward(st["grad"])
        return out.detach(), st["U0"].grad
    if kind == "tube":
        return dev.steps(st["U"].copy_(st["U0"]), dt, steps)
    if kind == "host":
        return dev.steps_host(st["U0"], st["U"], dt, steps)
    dev.import_state(st["U0"], out=st["U"])
    dev.steps(st["U"], dt, steps)
    return dev.export_state(st["U"], out=st["out"])


# ------------------------------------------------------------------ the least work of a pass
def work(case):
    """Bytes and operations that the method itself needs: at every Runge-Kutta stage the
    geometry's coefficients (each once) and indices, the stage's state in and out.  A divergence
    row reads about 20 vertices and 44.2 edges (65 and 304 in 3D)."""
    kind = case["kind"]
    T = 8 if case["precision"] == "fp64" else 4
    if kind == "tube":
        V = case["nx"] * case["ny"] * case["nz"]
        E = 7 * V
        row = 65 * (4 + 12 * 8) + 304 * (4 + 4 * 8)
        stage_b = V * (row + 2 * 20 * 8) + E * (24 + 9 * 8 + 40 * 8)
        stage_f = V * 2 * (60 * 65 + 20 * 304) + E * 2 * (160 + 250)
        return {"bytes": 3 * case["steps"] * stage_b, "flops": 3 * case["steps"] * stage_f}
    if kind == "batch":
        V = sum(len(m["x"]) for m in _members(case))
    elif kind == "sod":
        V = (case["nx"] + 11) ** 2
    elif kind == "quad":
        V = (case["nx"] + 10) * (case["ny"] + 10)
    elif kind == "couette":
        V = case["nx"] * (case["ny"] + 12)
    else:
        V = case["nx"] * case["ny"]
    visc = kind in ("tgv", "couette")
    E = 3 * V
    row = 20 * (4 + (12 if visc else 6) * T) + 44.2 * (4 + 3 * T)
    stage_b = V * (row + 2 * 12 * 8) + E * (24 + 32 * T)
    stage_f = V * 2 * (24 * 20 * (2 if visc else 1) + 12 * 44.2) + E * 2 * (120 + 150)
    stages = 1 if kind == "residual" else 3 * case["steps"]
    if kind == "adjoint":                       # forward, and as much again twice for the reverse
        stages *= 3
    b, f = stages * stage_b, stages * stage_f
    return {"bytes": int(b), "flops": int(f)}


# ------------------------------------------------------------------ the method in 64 bits
def _sparse(ptr, idx, val, ncol):
    return torch.sparse_csr_tensor(ptr, idx, val, size=(len(ptr) - 1, ncol), dtype=torch.float64,
                                   device="cuda")


class _Gather(torch.autograd.Function):
    """Sparse matrix times dense matrix, with the transpose product as its derivative."""

    @staticmethod
    def forward(ctx, A, At, x):
        ctx.At = At
        return A @ x

    @staticmethod
    def backward(ctx, g):
        return None, None, ctx.At @ g


class _Matrix:
    def __init__(self, ptr, idx, val, ncol):
        self.A = _sparse(ptr, idx, val, ncol)
        self.At = None
        self.parts = (ptr, idx, val, ncol)

    def __matmul__(self, x):
        if x.requires_grad and self.At is None:
            ptr, idx, val, ncol = self.parts
            rows = torch.repeat_interleave(torch.arange(len(ptr) - 1, device="cuda"), ptr[1:] - ptr[:-1])
            order = torch.argsort(idx, stable=True)
            tptr = torch.zeros(ncol + 1, dtype=torch.int64, device="cuda")
            tptr[1:] = torch.cumsum(torch.bincount(idx, minlength=ncol), 0)
            self.At = _sparse(tptr, rows[order], val[order], len(ptr) - 1)
        return _Gather.apply(self.A, self.At, x.contiguous())


def _cuda(a, dtype=None):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).cuda()


def _row_blocks(coef, N, M, per_v, rows):
    """Row k (of `rows`) of every vertex's block [rows x (per_v N + M)], concatenated."""
    L = per_v * N + M
    off = np.concatenate([[0], np.cumsum(rows * L)])[:-1]
    within = np.arange(L.sum()) - np.repeat(np.cumsum(L) - L, L)
    return [coef[np.repeat(off + k * L, L) + within] for k in range(rows)]


class Exact2:
    """The method on a mesh's own geometry coefficients, in plain torch float64."""

    def __init__(self, mesh, opts):
        P = Prep(mesh, **opts)
        self.opts, self.V = opts, len(mesh["x"])
        V = self.V
        self.sten = _cuda(P.get("stencil").reshape(-1, 6), np.int64)
        nrm = _cuda(P.get("normal").reshape(-1, 2))
        self.nx, self.ny = nrm[:, 0].clone(), nrm[:, 1].clone()
        Ef = len(nrm)
        self.w5 = _cuda(P.get("w5").reshape(-1, 2, 15))
        self.w3 = _cuda(P.get("w3").reshape(-1, 2, 3, 3))
        act = P.get("active")
        self.act = _cuda(act, np.int64)
        self.lmin = _cuda(P.get("lmin"))[self.act]
        vp, ep = P.get("div_vptr").astype(np.int64), P.get("div_eptr").astype(np.int64)
        N, M = np.diff(vp), np.diff(ep)
        pos = np.full(len(P.get("edges")) // 2, -1, np.int64)
        pos[P.get("flux_edges")] = np.arange(Ef)
        vidx, eidx = P.get("div_vidx").astype(np.int64), pos[P.get("div_eidx")]
        L = 2 * N + M
        ptr = np.concatenate([[0], np.cumsum(L)])
        idx = np.empty(ptr[-1], np.int64)
        at = np.repeat(ptr[:-1], N) + 2 * (np.arange(len(vidx)) - np.repeat(vp[:-1], N))
        idx[at], idx[at + 1] = 2 * vidx, 2 * vidx + 1
        idx[np.repeat(ptr[:-1] + 2 * N, M) + np.arange(len(eidx)) - np.repeat(ep[:-1], M)] = 2 * V + eidx
        p, i = _cuda(ptr), _cuda(idx)
        self.D = [_Matrix(p, i, _cuda(c), 2 * V + Ef) for c in _row_blocks(P.get("div_coef"), N, M, 2, 3)]
        if opts.get("viscous"):
            vptr = np.concatenate([[0], np.cumsum(2 * N)])
            vi = np.stack([2 * vidx, 2 * vidx + 1], 1).ravel()
            self.Dv = [_Matrix(_cuda(vptr), _cuda(vi), _cuda(c), 2 * V)
                       for c in _row_blocks(P.get("visc_coef"), N, 0 * M, 2, 3)]
        g, d, f = (np.asarray(mesh[k], np.int64) for k in ("ghost_ids", "ghost_donor", "ghost_flags"))
        keep = d >= 0
        g, d, f = g[keep], d[keep], f[keep]
        src = np.arange(V)
        src[g] = d
        self.ghosts = len(g) > 0
        zero = np.zeros((12, V), bool)
        zero[4:8, g] = (f & 1) != 0
        zero[8:12, g] = (f & 2) != 0
        self.src, self.keep = _cuda(src), _cuda((~zero).astype(np.float64))

    def refresh(self, U):
        return U[:, self.src] * self.keep if self.ghosts else U

    @staticmethod
    def pressure(w):
        return (GAMMA - 1.0) * (w[3] - 0.5 * (w[1] * w[1] + w[2] * w[2]) / w[0])

    def fluxes(self, w):
        p = self.pressure(w)
        u, v = w[1] / w[0], w[2] / w[0]
        return (torch.stack([w[1], w[1] * u + p, w[2] * u, (w[3] + p) * u]),
                torch.stack([w[2], w[1] * v, w[2] * v + p, (w[3] + p) * v]))

    def roe(self, wl, wr):
        rl, rr = torch.sqrt(wl[0]), torch.sqrt(wr[0])
        s = rl + rr
        u, v = (wl[1] / rl + wr[1] / rr) / s, (wl[2] / rl + wr[2] / rr) / s
        H = ((wl[3] + self.pressure(wl)) / rl + (wr[3] + self.pressure(wr)) / rr) / s
        return u, v, H, torch.sqrt((GAMMA - 1.0) * (H - 0.5 * (u * u + v * v)))

    def left(self, u, v, c, a):
        """Characteristic values L a of (4, ...) conservative values."""
        nx, ny = self.nx, self.ny
        b1 = (GAMMA - 1.0) / (c * c)
        b2 = 0.5 * b1 * (u * u + v * v)
        qn, qt = u * nx + v * ny, -u * ny + v * nx
        um = u * a[1] + v * a[2]
        nm = (nx * a[1] + ny * a[2]) / c
        return torch.stack([0.5 * ((b2 + qn / c) * a[0] - b1 * um - nm + b1 * a[3]),
                            (1.0 - b2) * a[0] + b1 * um - b1 * a[3],
                            -qt * a[0] - ny * a[1] + nx * a[2],
                            0.5 * ((b2 - qn / c) * a[0] - b1 * um + nm + b1 * a[3])])

    def right(self, u, v, H, c, C):
        nx, ny = self.nx, self.ny
        qn, qt = u * nx + v * ny, -u * ny + v * nx
        s, d = C[0] + C[1] + C[3], C[3] - C[0]
        return torch.stack([s, u * s + c * nx * d - ny * C[2], v * s + c * ny * d + nx * C[2],
                            H * (C[0] + C[3]) + c * qn * d + 0.5 * (u * u + v * v) * C[1] + qt * C[2]])

    def edge_flux(self, U):
        W = U[:, self.sten]                                     # 12, Ef, 6
        wi, wj = W[:4, :, 2], W[:4, :, 3]
        u, v, H, c = self.roe(wi, wj)
        C = [self.left(u, v, c, W[:4, :, k]) for k in range(6)]
        sides = []
        for side, order in enumerate(((0, 1, 2, 3, 4), (5, 4, 3, 2, 1))):
            w5 = self.w5[:, side]
            nodes = W[:, :, side:side + 5]
            five = sum((nodes[4 * d:4 * d + 4] * w5[:, d::3]).sum(-1) for d in range(3))
            c5 = self.left(u, v, c, five)
            q = [C[k] for k in order]
            b = [13.0 / 12.0 * (q[0] - 2 * q[1] + q[2]) ** 2 + 0.25 * (q[0] - 4 * q[1] + 3 * q[2]) ** 2,
                 13.0 / 12.0 * (q[1] - 2 * q[2] + q[3]) ** 2 + 0.25 * (q[1] - q[3]) ** 2,
                 13.0 / 12.0 * (q[2] - 2 * q[3] + q[4]) ** 2 + 0.25 * (3 * q[2] - 4 * q[3] + q[4]) ** 2]
            a = [k / (1e-2 + x) ** 2 for k, x in zip((1 / 16, 10 / 16, 5 / 16), b)]
            s = a[0] + a[1] + a[2]
            w3 = self.w3[:, side]
            c3 = sum(a[j] / s * sum(w3[:, j, t] * q[j + t] for t in range(3)) for j in range(3))
            o1 = (a[0] / s).detach()
            sides.append(self.right(u, v, H, c, torch.where((o1 > 0.01) & (o1 < 0.79), c5, c3)))
        wl, wr = (torch.where(((w[0] > 0) & (self.pressure(w) > 0))[None], w, e)
                  for w, e in zip(sides, (wi, wj)))
        u, v, H, c = self.roe(wl, wr)
        qn = u * self.nx + v * self.ny
        lam = torch.stack([qn - c, qn, qn, qn + c])
        dl = 0.1 * c
        al = torch.where(lam.abs() < dl, (lam * lam + dl * dl) / (2 * dl), lam.abs())
        diss = self.right(u, v, H, c, al * self.left(u, v, c, wr - wl))
        F = [f * self.nx + g * self.ny for f, g in (self.fluxes(wl), self.fluxes(wr))]
        return 0.5 * (F[0] + F[1]) - 0.5 * diss

    def viscous(self, U):
        w, wx, wy, o = U[:4], U[4:8], U[8:12], self.opts
        u, v = w[1] / w[0], w[2] / w[0]
        p, q2 = self.pressure(w), u * u + v * v
        dv = []
        for d in (wx, wy):
            du, dw = (d[1] - u * d[0]) / w[0], (d[2] - v * d[0]) / w[0]
            dp = (GAMMA - 1.0) * (d[3] - 0.5 * d[0] * q2 - w[0] * (u * du + v * dw))
            dv.append((du, dw, (dp / w[0] - p * d[0] / w[0] ** 2) / o["R_gas"]))
        (ux, vx, Tx), (uy, vy, Ty) = dv
        mu = o["mu"]
        kappa = mu * (GAMMA * o["R_gas"] / (GAMMA - 1.0)) / o["prandtl"]
        txx, tyy = mu * (4 * ux - 2 * vy) / 3, mu * (4 * vy - 2 * ux) / 3
        txy, z = mu * (uy + vx), torch.zeros_like(u)
        return (torch.stack([z, txx, txy, u * txx + v * txy + kappa * Tx]),
                torch.stack([z, txy, tyy, u * txy + v * tyy + kappa * Ty]))

    def residual(self, U):
        F, G = self.fluxes(U[:4])
        X = torch.cat([torch.stack([F, G], -1).reshape(4, -1), self.edge_flux(U)], 1).t()
        R = -torch.cat([(D @ X).t() for D in self.D])
        if self.opts.get("viscous"):
            Y = torch.stack(self.viscous(U), -1).reshape(4, -1).t()
            R = R + torch.cat([(D @ Y).t() for D in self.Dv])
        return torch.zeros_like(U).index_copy(1, self.act, R)

    def step(self, U, dt):
        U = self.refresh(U)
        if dt <= 0.0:
            w = U[:4, self.act]
            speed = torch.sqrt(w[1] ** 2 + w[2] ** 2) / w[0] + torch.sqrt(GAMMA * self.pressure(w) / w[0])
            dt = 0.3 * float((self.lmin / speed).min())
        u1 = self.refresh(U + dt * self.residual(U))
        u2 = self.refresh(0.75 * U + 0.25 * (u1 + dt * self.residual(u1)))
        return self.refresh(U / 3 + 2 / 3 * (u2 + dt * self.residual(u2)))


class Exact3:
    """The 3D extension on the mesh's own geometry coefficients, in plain torch float64."""

    def __init__(self, mesh):
        M = hfd3d.Mesh3(mesh, host_only=1)
        V, E = M.nv, M.nedges
        self.sten = _cuda(M.prep_get("sten").reshape(-1, 6), np.int64)
        fr = _cuda(M.prep_get("frame").reshape(-1, 9))
        self.n, self.t1, self.t2 = ([fr[:, 3 * k + d].clone() for d in range(3)] for k in range(3))
        self.w5 = _cuda(M.prep_get("w5").reshape(-1, 2, 20))
        self.w3 = _cuda(M.prep_get("w3").reshape(-1, 2, 3, 3))
        vp, ep = M.prep_get("vptr").astype(np.int64), M.prep_get("eptr").astype(np.int64)
        vi, ei = M.prep_get("vidx").astype(np.int64), M.prep_get("eidx").astype(np.int64)
        self.Dv, self.De = [], []
        ip = np.stack([3 * vi, 3 * vi + 1, 3 * vi + 2], 1).ravel()
        cv, ce = M.prep_get("cv").reshape(-1, 4, 3), M.prep_get("ce").reshape(-1, 4)
        for k in range(4):
            self.Dv.append(_Matrix(_cuda(3 * vp), _cuda(ip), _cuda(cv[:, k].ravel()), 3 * V))
            self.De.append(_Matrix(_cuda(ep), _cuda(ei), _cuda(ce[:, k]), E))

    @staticmethod
    def pressure(w):
        return (GAMMA - 1.0) * (w[4] - 0.5 * (w[1] ** 2 + w[2] ** 2 + w[3] ** 2) / w[0])

    def roe(self, wl, wr):
        rl, rr = torch.sqrt(wl[0]), torch.sqrt(wr[0])
        u = [(wl[k] / rl + wr[k] / rr) / (rl + rr) for k in (1, 2, 3)]
        H = ((wl[4] + self.pressure(wl)) / rl + (wr[4] + self.pressure(wr)) / rr) / (rl + rr)
        K = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        return u, H, K, torch.sqrt((GAMMA - 1.0) * (H - 0.5 * K))

    @staticmethod
    def dot(a, b):
        return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]

    def left(self, u, K, c, a):
        b1 = (GAMMA - 1.0) / (c * c)
        b2, qc = 0.5 * b1 * K, self.dot(u, self.n) / c
        um, nm = self.dot(u, a[1:4]), self.dot(self.n, a[1:4]) / c
        return torch.stack([0.5 * ((b2 + qc) * a[0] - b1 * um - nm + b1 * a[4]),
                            (1.0 - b2) * a[0] + b1 * um - b1 * a[4],
                            self.dot(self.t1, a[1:4]) - self.dot(u, self.t1) * a[0],
                            self.dot(self.t2, a[1:4]) - self.dot(u, self.t2) * a[0],
                            0.5 * ((b2 - qc) * a[0] - b1 * um + nm + b1 * a[4])])

    def right(self, u, H, K, c, C):
        s, d = C[0] + C[1] + C[4], (C[4] - C[0]) * c
        m = [s * u[k] + d * self.n[k] + C[2] * self.t1[k] + C[3] * self.t2[k] for k in range(3)]
        return torch.stack([s, *m, (C[0] + C[4]) * H + d * self.dot(u, self.n) + 0.5 * K * C[1]
                            + C[2] * self.dot(u, self.t1) + C[3] * self.dot(u, self.t2)])

    def flux(self, w, n):
        """Flux along n: three numbers, or a direction per edge."""
        un, p = self.dot(w[1:4], n) / w[0], self.pressure(w)
        return torch.stack([w[0] * un, *[w[1 + k] * un + p * n[k] for k in range(3)], (w[4] + p) * un])

    def edge_flux(self, U):
        W = U[:, self.sten]
        wi, wj = W[:5, :, 2], W[:5, :, 3]
        u, H, K, c = self.roe(wi, wj)
        C = [self.left(u, K, c, W[:5, :, k]) for k in range(6)]
        sides = []
        for side, order in enumerate(((0, 1, 2, 3, 4), (5, 4, 3, 2, 1))):
            w5 = self.w5[:, side]
            nodes = W[:, :, side:side + 5]
            five = sum((nodes[5 * d:5 * d + 5] * w5[:, d::4]).sum(-1) for d in range(4))
            c5 = self.left(u, K, c, five)
            q = [C[k] for k in order]
            b = [13.0 / 12.0 * (q[0] - 2 * q[1] + q[2]) ** 2 + 0.25 * (q[0] - 4 * q[1] + 3 * q[2]) ** 2,
                 13.0 / 12.0 * (q[1] - 2 * q[2] + q[3]) ** 2 + 0.25 * (q[1] - q[3]) ** 2,
                 13.0 / 12.0 * (q[2] - 2 * q[3] + q[4]) ** 2 + 0.25 * (3 * q[2] - 4 * q[3] + q[4]) ** 2]
            a = [k / (1e-2 + x) ** 2 for k, x in zip((1 / 16, 10 / 16, 5 / 16), b)]
            s = a[0] + a[1] + a[2]
            w3 = self.w3[:, side]
            c3 = sum(a[j] / s * sum(w3[:, j, t] * q[j + t] for t in range(3)) for j in range(3))
            o1 = a[0] / s
            sides.append(self.right(u, H, K, c, torch.where((o1 > 0.01) & (o1 < 0.79), c5, c3)))
        wl, wr = (torch.where(((w[0] > 0) & (self.pressure(w) > 0))[None], w, e)
                  for w, e in zip(sides, (wi, wj)))
        u, H, K, c = self.roe(wl, wr)
        qn = self.dot(u, self.n)
        lam = torch.stack([qn - c, qn, qn, qn, qn + c])
        dl = 0.1 * c
        al = torch.where(lam.abs() < dl, (lam * lam + dl * dl) / (2 * dl), lam.abs())
        diss = self.right(u, H, K, c, al * self.left(u, K, c, wr - wl))
        return 0.5 * (self.flux(wl, self.n) + self.flux(wr, self.n)) - 0.5 * diss

    def residual(self, U):
        F = [self.flux(U[:5], [float(k == d) for k in range(3)]) for d in range(3)]
        X, h = torch.stack(F, -1).reshape(5, -1).t().contiguous(), self.edge_flux(U).t().contiguous()
        return -torch.cat([(a @ X + b @ h).t() for a, b in zip(self.Dv, self.De)])

    def step(self, U, dt):
        u1 = U + dt * self.residual(U)
        u2 = 0.75 * U + 0.25 * (u1 + dt * self.residual(u1))
        return U / 3 + 2 / 3 * (u2 + dt * self.residual(u2))


def exact(case, seed):
    kind, steps = case["kind"], case["steps"]
    if kind == "tube":
        mesh = three_d.periodic_tet_box(case["nx"], case["ny"], case["nz"], 10.0, 10.0 * case["ny"] / case["nx"],
                                        10.0 * case["nz"] / case["nx"], seed=3)
        U, dt = _states(case, mesh, seed)
        U, ex = torch.from_numpy(U).cuda(), Exact3(mesh)
        for _ in range(steps):
            U = ex.step(U, dt)
        return U
    if kind == "batch":
        meshes = _members(case)
        states, dt = _states(case, meshes, seed)
        out = []
        for m, u in zip(meshes, states):
            ex, u = Exact2(m, {}), torch.from_numpy(u).cuda()
            for _ in range(steps):
                u = ex.step(u, dt)
            out.append(u)
        return out
    mesh, opts = _mesh_of(case)
    U, dt = _states(case, mesh, seed)
    U, ex = torch.from_numpy(U).cuda(), Exact2(mesh, opts)
    if kind in ("residual", "adjoint"):
        perm = torch.from_numpy(_plan(case).dev.perm.astype(np.int64)).cuda()     # the plan's vertex order
    if kind == "residual":
        return ex.residual(ex.refresh(U))[:, perm]
    if kind == "adjoint":
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        grad = torch.randn(U.shape, dtype=torch.float64, device="cuda", generator=g)
        U.requires_grad_(True)
        out = U
        for _ in range(steps):
            out = ex.step(out, dt)
        out[:, perm].backward(grad)
        return out.detach()[:, perm], U.grad[:, perm]
    for _ in range(steps):
        U = ex.step(U, dt)
    return U
