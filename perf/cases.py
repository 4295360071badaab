"""Timed cases of the solver: what its users call, through the package's public entry points.

Kinds of case (``kind``):

* ``apply``   one operator apply y = alpha M u + beta K u (``Slab.apply``): the building block of a
              user's own Krylov solver or error estimate, in each precision the entry point offers
              in earnest (FP64, double-float, FP32, FP32 with the bf16 metric).
* ``tissue``  new conductivities and fibre angles on a standing mesh, then the operator's diagonal
              (``Slab.set_tissue``, ``Slab.diagonal``): every evaluation of a parameter study or an
              inverse problem begins with it.
* ``vcycle``  one multigrid V-cycle z = V(r) (``capi.sem_vcycle``): the preconditioner alone, for a
              user's own outer iteration.
* ``step``    time steps of the monodomain problem from a checkpoint (``State.restore``,
              ``State.step``, ``State.checkpoint``): plain FP64 Jacobi-CG, the all-FP64 multigrid
              path, or the mixed-precision one (double-float operator, low-precision V-cycle).
* ``host``    the same step on page-locked host arrays (``capi.sem_step_host_out``): a caller that
              keeps its fields in host memory and rotates three arrays per field.
* ``grad``    sensor traces and the gradient of their misfit in the conductivities and fibre angles
              (``traces(...)`` and ``backward()``): forward and adjoint runs of an inverse problem.

Meshes are the perturbed 20 x 7 x 3 mm slabs (and the 40 x 20 x 6 mm one) of ``workloads``, degrees
1..6, both quadratures ("LG" = SEM, "LGL" = SEM-NI), from the 765-node slab to 30 million nodes.

``exact`` recomputes a case in 64-bit torch from the definitions (tensor-product tables, trilinear
geometry, BDF steps, conjugate gradients to a residual of 1e-13) without any code of the package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

DT = 0.05             # ms, the time step of every run of this repository's benchmark
ALPHA = 1.5 / DT      # its operator is (3 / (2 dt)) M + K
RTOL = 1e-10          # and its stopping rule ||r|| <= 1e-10 ||b||
BOX = (20.0, 7.0, 3.0)

IONIC = dict(u_rest=-85.0, u_amp=100.0, tau_in=0.3, tau_out=6.0, tau_open=120.0, tau_close=150.0,
             v_gate=0.13, kappa=0.01)


def listed():
    return [
        # the smallest call: the 765-node slab of the tests, where launches and host work count
        dict(name="apply_fp64_tiny", kind="apply", p=2, quad="LGL", nx=8, ny=4, nz=2, prec="fp64"),
        # the operator sweep's central row: FP64, Q4, 2.06 million nodes
        dict(name="apply_fp64_p4_2m", kind="apply", p=4, quad="LGL", nx=83, ny=29, nz=13, prec="fp64"),
        # full Gauss quadrature (SEM) in double-float, the sweep's highest degree
        dict(name="apply_df64_sem_p6", kind="apply", p=6, quad="LG", nx=56, ny=20, nz=8, prec="df64"),
        # the largest mesh: 29.9 million nodes, the smoother's precision
        dict(name="apply_bf16_p4_30m", kind="apply", p=4, quad="LGL", nx=207, ny=72, nz=31, prec="bf16"),
        # a parameter update on the sweep slab, at an odd degree
        dict(name="tissue_p5_2m", kind="tissue", p=5, quad="LGL", nx=67, ny=23, nz=10),
        # the benchmark's V-cycle (p 4 -> 2, Chebyshev 6 / 5, bf16 metric)
        dict(name="vcycle_bf16_p4_2m", kind="vcycle", p=4, quad="LGL", nx=83, ny=29, nz=13, prec="bf16",
             degree=6, coarse_degree=5, min_coarse=300000),
        # a whole run on a small mesh: many short solves, bound by latency
        dict(name="step_jacobi_tiny", kind="step", p=2, quad="LGL", nx=8, ny=4, nz=2, method="jacobi", steps=20),
        # the paper's own method: SEM quadrature, FP64 Jacobi-CG, a ragged mid-size mesh
        dict(name="step_jacobi_sem_p3", kind="step", p=3, quad="LG", nx=55, ny=19, nz=9, method="jacobi", steps=3),
        # the benchmark's mixed-precision step
        dict(name="step_mixed_p4_2m", kind="step", p=4, quad="LGL", nx=83, ny=29, nz=13, method="mixed",
             prec="bf16", degree=6, coarse_degree=5, min_coarse=300000, steps=10),
        # the 8.57 million node run: p- and h-levels, Chebyshev(3), activation times recorded
        dict(name="step_mixed_p4_8m", kind="step", p=4, quad="LGL", nx=128, ny=64, nz=16, lx=40.0, ly=20.0, lz=6.0,
             method="mixed", prec="bf16", degree=3, coarse_degree=10, min_coarse=2000, steps=6, track=True),
        # the same step called with host arrays, end to end
        dict(name="host_mixed_p4_2m", kind="host", p=4, quad="LGL", nx=83, ny=29, nz=13, prec="bf16", degree=6,
             coarse_degree=5, min_coarse=300000, steps=4),
        # an inverse problem's loss and gradient on a small mesh
        dict(name="grad_p3_70k", kind="grad", p=3, quad="LGL", nx=36, ny=13, nz=5, steps=8, every=4, sensors=64),
    ]


def _mesh(rng, p, nodes):
    """Element counts of a slab of about ``nodes`` nodes, its sides spread around the 20 : 7 : 3 box."""
    h = (420.0 / max(nodes, 1.0)) ** (1.0 / 3.0) * p
    return [max(1, round(length / h * rng.uniform(0.8, 1.25))) for length in BOX]


def _spread(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "tissue", "vcycle", "step", "step", "step", "host", "grad"])
    p = rng.randint(1, 6)
    quad = rng.choice(["LGL", "LGL", "LG"])
    c = dict(kind=kind, p=p, quad=quad)
    if kind == "apply":
        c["prec"] = rng.choice(["fp64", "df64", "fp32", "bf16"])
        nodes = _spread(rng, 700, 6e6)
    elif kind == "tissue":
        nodes = _spread(rng, 700, 2e6)
    elif kind == "vcycle":
        c["p"] = p = max(2, p)
        nodes = _spread(rng, 3000, 2e6)
        # the coarsest level is a p-level of the fine mesh, as in the listed case
        c.update(prec=rng.choice(["bf16", "fp32", "fp64"]), degree=rng.choice([3, 6]), coarse_degree=rng.choice([5, 10]))
    elif kind == "step":
        c["method"] = rng.choice(["jacobi", "mixed", "mixed", "fp64gmg"])
        nodes = _spread(rng, 700, 1e6 if c["method"] == "mixed" else 2e5)
        c["steps"] = rng.choice([2, 3, 5])
        if c["method"] != "jacobi":
            c.update(prec="fp64" if c["method"] == "fp64gmg" else rng.choice(["bf16", "fp32"]),
                     degree=rng.choice([3, 6]), coarse_degree=rng.choice([5, 10]), min_coarse=rng.choice([2000, 300000]))
        c["track"] = rng.random() < 0.3
    elif kind == "host":
        nodes = _spread(rng, 3000, 1e6)
        c.update(prec="bf16", degree=rng.choice([3, 6]), coarse_degree=5, min_coarse=rng.choice([2000, 300000]), steps=3)
    else:
        c["p"] = p = rng.randint(1, 4)
        nodes = _spread(rng, 700, 4e4)
        c.update(steps=rng.choice([3, 4, 6]), every=rng.choice([2, 4, 20]), sensors=rng.choice([1, 16, 64]))
    c["nx"], c["ny"], c["nz"] = _mesh(rng, p, nodes)
    if kind == "vcycle":  # one p-level below the fine one
        pc = max(1, p // 2)
        c["min_coarse"] = (pc * c["nx"] + 1) * (pc * c["ny"] + 1) * (pc * c["nz"] + 1)
    return c


# ------------------------------------------------------------------ inputs

def _nodes(c):
    return (c["p"] * c["nx"] + 1) * (c["p"] * c["ny"] + 1) * (c["p"] * c["nz"] + 1)


def _lengths(c):
    return (c.get("lx", BOX[0]), c.get("ly", BOX[1]), c.get("lz", BOX[2]))


def _vertices(c, seed):
    """Slab vertices, each moved by up to a tenth of the spacing (faces keep their plane), [z, y, x, 3]."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n = (c["nx"], c["ny"], c["nz"])
    v = np.empty((n[2] + 1, n[1] + 1, n[0] + 1, 3))
    for d, length in enumerate(_lengths(c)):
        shape = [1, 1, 1]
        shape[2 - d] = n[d] + 1
        v[..., d] = np.linspace(0.0, length, n[d] + 1).reshape(shape)
        inner = np.ones(n[d] + 1)
        inner[[0, -1]] = 0.0
        v[..., d] += rng.uniform(-0.1, 0.1, size=v.shape[:3]) * (length / n[d]) * inner.reshape(shape)
    return v


def _tissue(c, seed):
    """Conductivities varied by up to 20 % per element, fibres rotating from -60 to +60 degrees through z."""
    rng = np.random.Generator(np.random.PCG64(seed + 1000003))
    ne = c["nx"] * c["ny"] * c["nz"]
    f = rng.uniform(0.8, 1.2, size=(2, ne))
    z = np.repeat((np.arange(c["nz"]) + 0.5) / c["nz"], c["nx"] * c["ny"])
    theta = np.deg2rad(-60.0 + 120.0 * z) + rng.uniform(-0.05, 0.05, size=ne)
    return 0.12 * f[0], 0.03 * f[1], theta


def _fields(c, seed, device):
    """Two consecutive levels of a travelling front (u in mV, gate h) on the node lattice, float64 on ``device``:
    depolarised behind the front, partly inactivated gate, a little node noise as discrete solutions carry it."""
    g = torch.Generator(device="cpu").manual_seed(seed + 77)
    lx, ly, lz = _lengths(c)
    ax = [torch.linspace(0.0, length, c["p"] * n + 1, dtype=torch.float64, device=device)
          for length, n in ((lx, c["nx"]), (ly, c["ny"]), (lz, c["nz"]))]
    r = torch.rand(4, generator=g, dtype=torch.float64).tolist()
    front = lx * (0.25 + 0.3 * r[0])
    s = ax[0][None, None, :] + (0.4 * r[1] - 0.2) * ax[1][None, :, None] + (0.4 * r[2] - 0.2) * ax[2][:, None, None]
    # the wave moves about 0.03 mm per step
    out = []
    for shift in (0.03, 0.0):
        f = torch.sigmoid((front + shift - s) / (0.35 + 0.2 * r[3]))
        wake = torch.sigmoid((front + shift - 1.0 - s) / 0.8)
        u = -85.0 + 100.0 * f * (1.0 - 0.08 * wake)
        h = 1.0 - 0.55 * wake
        out.append((u.reshape(-1).contiguous(), h.reshape(-1).contiguous()))
    return {"u": out[0][0], "u_prev": out[1][0], "h": out[0][1], "h_prev": out[1][1]}


def _vector(n, seed, dtype, device):
    g = torch.Generator(device=device).manual_seed(seed + 5)
    return torch.rand(n, generator=g, dtype=torch.float64, device=device).mul_(2.0).sub_(1.0).to(dtype)


def _stimulus(c):
    lx, ly, lz = _lengths(c)
    return (-1.0, -1.0, -1.0, 0.15 * lx, 0.5 * ly, lz + 1.0), 50.0, 0.0, 1.0


def _sensors(c, seed):
    rng = np.random.Generator(np.random.PCG64(seed + 9))
    n = _nodes(c)
    return np.sort(rng.choice(n, size=min(c["sensors"], n), replace=False)).astype(np.int64)


def prepare(case, seed):
    import paper_2205_05136_gb300 as gb
    c = dict(case)
    slab = gb.Slab(np.ascontiguousarray(_vertices(c, seed)).reshape(-1, 3), c["nx"], c["ny"], c["nz"], c["p"], c["quad"])
    dev = slab.device
    tissue = [torch.as_tensor(a, dtype=torch.float64, device=dev) for a in _tissue(c, seed)]
    capi = gb.capi
    s = dict(case=c, gb=gb, slab=slab, tissue=tissue)
    if c["kind"] != "grad":
        slab.set_tissue(*tissue)
    precs = dict(fp64=capi.SEM_PREC_FP64, df64=capi.SEM_PREC_DF64, fp32=capi.SEM_PREC_FP32, bf16=capi.SEM_PREC_FP32_BF16)
    if c["kind"] == "apply":
        s["prec"] = precs[c["prec"]]
        s["u"] = _vector(slab.ndofs, seed, torch.float64 if c["prec"] in ("fp64", "df64") else torch.float32, dev)
    elif c["kind"] == "tissue":
        # the next parameter set of the study
        s["tissue"] = [torch.as_tensor(a, dtype=torch.float64, device=dev) for a in _tissue(c, seed + 31)]
    elif c["kind"] == "vcycle":
        capi.sem_set_gmg(slab.ctx, c["degree"], c["coarse_degree"], c["min_coarse"], precs[c["prec"]])
        s["r"] = _vector(slab.ndofs, seed, torch.float64, dev)
    elif c["kind"] in ("step", "host"):
        if c.get("method") != "jacobi":
            capi.sem_set_gmg(slab.ctx, c["degree"], c["coarse_degree"], c["min_coarse"], precs[c["prec"]])
            if c.get("method") != "fp64gmg":
                capi.sem_set_operator_precision(slab.ctx, capi.SEM_PREC_DF64)
        slab.set_ionic()
        box, amp, t0, t1 = _stimulus(c)
        slab.set_stimulus("box", box, amp, t0, t1)
        f = _fields(c, seed, dev)
        if c["kind"] == "step":
            s["state"] = slab.new_state(f["u"], f["h"])
            s["from"] = dict(f, n=5)
            s["precond"] = capi.SEM_PC_JACOBI if c["method"] == "jacobi" else capi.SEM_PC_GMG
        else:
            s["host"] = {k: v.cpu().pin_memory() for k, v in f.items()}
            s["ring"] = [[torch.empty(slab.ndofs, dtype=torch.float64, pin_memory=True) for _ in "uh"] for _ in range(3)]
    else:
        f = _fields(c, seed, dev)
        s["u0"], s["h0"] = f["u"], f["h"]
        s["sensors"] = torch.as_tensor(_sensors(c, seed), dtype=torch.int32, device=dev)
        s["target"] = -85.0 + 10.0 * _vector(c["steps"] * s["sensors"].numel(), seed + 3, torch.float64, dev).reshape(c["steps"], -1)
        slab.set_ionic()
        box, amp, t0, t1 = _stimulus(c)
        slab.set_stimulus("box", box, amp, t0, t1)
        capi.sem_set_gmg(slab.ctx, 3, 10, 2000, capi.SEM_PREC_FP32)
    return s


def run(state):
    s, c, slab, capi = state, state["case"], state["slab"], state["gb"].capi
    kind = c["kind"]
    if kind == "apply":
        return slab.apply(s["u"], ALPHA, 1.0, s["prec"])
    if kind == "tissue":
        slab.set_tissue(*s["tissue"])
        return slab.diagonal(ALPHA, 1.0)
    if kind == "vcycle":
        z = torch.empty_like(s["r"])
        capi.sem_vcycle(slab.ctx, ALPHA, s["r"], z)
        return z
    if kind == "step":
        st = s["state"]
        st.restore(s["from"])
        if c.get("track"):
            st.track_activation()
        st.step(DT, c["steps"], RTOL, 0.0, 2000, s["precond"])
        out = st.checkpoint()
        out.pop("n")
        if c.get("track"):
            # the times themselves are left out: where the tissue rests, |du/dt| is solver noise and
            # the step at which it peaks is no property of the solution
            out["dudt_max"] = st.activation()[1]
        return out
    if kind == "host":
        f = s["host"]
        u, up, h, hp = f["u"], f["u_prev"], f["h"], f["h_prev"]
        for k in range(c["steps"]):
            un, hn = s["ring"][k % 3]  # never one of the two levels that this step reads
            capi.sem_step_host_out(slab.ctx, u, up, h, hp, un, hn, 5 + k, DT, RTOL, 0.0, 2000, capi.SEM_PC_GMG)
            up, u, hp, h = u, un, h, hn
        return {"u": u, "h": h, "u_prev": up, "h_prev": hp}
    params = [t.detach().clone().requires_grad_(True) for t in s["tissue"]]
    T = s["gb"].traces(slab, *params, s["u0"], s["h0"], DT, c["steps"], s["sensors"], checkpoint_every=c["every"],
                       rtol=1e-12, precond=capi.SEM_PC_GMG)
    loss = 0.5 * DT * ((T - s["target"]) ** 2).sum()
    loss.backward()
    return {"traces": T.detach(), "grad": [q.grad for q in params]}


def work(case):
    """Bytes of every input and output once (geometry as vertices and tissue, not as the stored metric) and the
    flops of plain sum factorization; a solve is counted as the one operator apply that it cannot do without."""
    n, p = _nodes(case), case["p"]
    ne = case["nx"] * case["ny"] * case["nz"]
    m = p + 1
    sweeps = 6 if case["quad"] == "LGL" else 12
    flops = ne * (sweeps * 2 * m ** 4 + 22 * m ** 3)
    geometry = 24 * (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1) + 24 * ne
    kind = case["kind"]
    if kind == "apply":
        return {"bytes": geometry + n * (16 if case["prec"] in ("fp64", "df64") else 8), "flops": flops}
    if kind == "tissue":
        return {"bytes": geometry + 8 * n, "flops": ne * 100 * m ** 3}
    if kind == "vcycle":
        return {"bytes": geometry + 16 * n, "flops": flops * 2 * case["degree"]}
    if kind in ("step", "host"):
        k = case["steps"]
        return {"bytes": geometry + 64 * n, "flops": k * (flops + 60 * n)}
    k = case["steps"]
    return {"bytes": geometry + 16 * n + 24 * ne, "flops": 3 * k * flops}


def tolerance(case):
    kind = case["kind"]
    # about four times what the path was measured to differ by from the 64-bit values below
    if kind == "apply":
        # FP64 3e-14 and float pairs 1.4e-13 (the metric's own rounding included), FP32 7e-8, the bf16 metric 1e-3
        return {"rel": {"fp64": 1.4e-13, "df64": 6e-13, "fp32": 4e-7, "bf16": 4e-3}[case["prec"]]}
    if kind == "tissue":
        return {"rel": 1.3e-13}  # 3.2e-14
    if kind == "vcycle":
        return {"rel": {"fp64": 1e-12, "fp32": 6e-7, "bf16": 2.4e-3}[case["prec"]]}  # bf16 6e-4, FP32 1.4e-7
    if kind in ("step", "host"):
        # solves stopped at ||r|| <= 1e-10 ||b||: up to 3.5e-9, largest in the recorded |du/dt|
        return {"rel": 1.4e-8, "max": 2e-6}
    return {"rel": 2e-8, "max": 2e-6}


# ------------------------------------------------------------------ 64-bit reference

def _legendre_points(p, quad):
    """GLL nodes of degree p, and the nodes and weights of the (p+1)-point rule."""
    L = np.polynomial.legendre
    c = np.zeros(p + 1)
    c[p] = 1.0
    x = np.concatenate([[-1.0], np.sort(L.legroots(L.legder(c)).real), [1.0]]) if p > 1 else np.array([-1.0, 1.0])
    for _ in range(3 if p > 1 else 0):  # polish the interior roots of P_p'
        d1, d2 = L.legder(c), L.legder(c, 2)
        x[1:-1] -= L.legval(x[1:-1], d1) / L.legval(x[1:-1], d2)
    x = 0.5 * (x - x[::-1])
    if quad == "LGL":
        return x, x, 2.0 / (p * (p + 1) * L.legval(x, c) ** 2)
    xq, wq = L.leggauss(p + 1)
    return x, xq, wq


def _lagrange(nodes, x):
    """l_i(x_q) and l_i'(x_q) as [q, i], by products."""
    n = len(nodes)
    B, D = np.ones((len(x), n)), np.zeros((len(x), n))
    for i in range(n):
        for m in range(n):
            if m == i:
                continue
            B[:, i] *= (x - nodes[m]) / (nodes[i] - nodes[m])
            t = np.full(len(x), 1.0 / (nodes[i] - nodes[m]))
            for k in range(n):
                if k not in (i, m):
                    t = t * (x - nodes[k]) / (nodes[i] - nodes[k])
            D[:, i] += t
    return B, D


class _Operator:
    """(alpha M + beta K) in 64-bit torch on one mesh: dense 1-D tables, chunks of elements."""

    def __init__(self, c, vertices, device, p=None):
        self.p = p = c["p"] if p is None else p
        self.quad, self.device = c["quad"], device
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        self.ne, n = nx * ny * nz, p + 1
        self.shape = (p * nz + 1, p * ny + 1, p * nx + 1)
        self.ndofs = self.shape[0] * self.shape[1] * self.shape[2]
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=device)  # noqa: E731
        self.nodes, xq, wq = _legendre_points(p, self.quad)
        B, D = _lagrange(self.nodes, xq)
        self.B, self.D = t(B), t(D)
        self.w = t(wq)[:, None, None] * t(wq)[None, :, None] * t(wq)[None, None, :]
        N, dN = np.stack([0.5 * (1 - xq), 0.5 * (1 + xq)], 1), np.tile([-0.5, 0.5], (n, 1))
        self.N, self.dN = t(N), t(dN)
        v = t(vertices)
        corner = [v[cz:cz + nz, cy:cy + ny, cx:cx + nx].reshape(-1, 3) for cz in (0, 1) for cy in (0, 1) for cx in (0, 1)]
        self.X = torch.stack(corner, 1).reshape(-1, 2, 2, 2, 3)
        ar = lambda m: torch.arange(m, device=device)  # noqa: E731
        e = (ar(nx)[None, None, :] * p + self.shape[2] * (ar(ny)[None, :, None] * p + self.shape[1] * p * ar(nz)[:, None, None])).reshape(-1)
        self.first = e
        self.local = ar(n)[None, None, :] + self.shape[2] * (ar(n)[None, :, None] + self.shape[1] * ar(n)[:, None, None])
        self.chunk = max(1, 6_000_000 // n ** 3)
        self.J = None

    def chunks(self):
        for a in range(0, self.ne, self.chunk):
            yield a, min(self.ne, a + self.chunk)

    def index(self, a, b):
        return (self.first[a:b, None] + self.local.reshape(1, -1)).reshape(-1)

    def geometry(self, a, b):
        """det J and J^{-1} [e, z, y, x, c, d] (d xi_c / d x_d) at the quadrature points."""
        X = self.X[a:b]
        cols = [torch.einsum("zk,yj,xi,ekjid->ezyxd", *m, X) for m in
                ((self.N, self.N, self.dN), (self.N, self.dN, self.N), (self.dN, self.N, self.N))]
        A0, A1, A2 = cols
        c12, c20, c01 = torch.linalg.cross(A1, A2), torch.linalg.cross(A2, A0), torch.linalg.cross(A0, A1)
        det = (A0 * c12).sum(-1)
        return det, torch.stack([c12, c20, c01], -2) / det[..., None, None]

    def metric(self, a, b, tissue):
        det, inv = self.geometry(a, b)
        sl, st, th = (q[a:b, None, None, None] for q in tissue)
        W = self.w * det
        f = torch.stack([torch.cos(th), torch.sin(th), torch.zeros_like(th)], -1)
        along = (inv * f[..., None, :]).sum(-1)
        G = st[..., None, None] * (inv @ inv.transpose(-1, -2)) + (sl - st)[..., None, None] * along[..., :, None] * along[..., None, :]
        return G * W[..., None, None], W

    def set_tissue(self, tissue):
        self.tissue = tissue
        self.G = [self.metric(a, b, tissue) for a, b in self.chunks()]

    def element(self, U, G, W, alpha, beta):
        """Element results [e, k, j, i] of (alpha M + beta K) on element values U."""
        B, D = self.B, self.D
        to = lambda z, y, x, V: torch.einsum("ck,ekji->ecji", z, torch.einsum("bj,ekji->ekbi", y, torch.einsum("ai,ekji->ekja", x, V)))  # noqa: E731
        out = to(B.T, B.T, B.T, alpha * W * to(B, B, B, U)) if alpha != 0.0 else torch.zeros_like(U)
        if beta == 0.0:
            return out
        g = torch.stack([to(B, B, D, U), to(B, D, B, U), to(D, B, B, U)], -1)
        q = (G @ g[..., None])[..., 0] * beta
        return out + to(B.T, B.T, D.T, q[..., 0]) + to(B.T, D.T, B.T, q[..., 1]) + to(D.T, B.T, B.T, q[..., 2])

    def apply(self, u, alpha, beta):
        y = torch.zeros_like(u)
        n = self.p + 1
        for (a, b), (G, W) in zip(self.chunks(), self.G):
            i = self.index(a, b)
            y.index_add_(0, i, self.element(u[i].reshape(-1, n, n, n), G, W, alpha, beta).reshape(-1))
        return y

    def diagonal(self, alpha, beta):
        d = torch.zeros(self.ndofs, dtype=torch.float64, device=self.device)
        bb, bd, dd = self.B * self.B, self.B * self.D, self.D * self.D
        to = lambda z, y, x, V: torch.einsum("ck,bj,ai,ecba->ekji", z, y, x, V)  # noqa: E731
        for (a, b), (G, W) in zip(self.chunks(), self.G):
            v = alpha * to(bb, bb, bb, W)
            v = v + beta * (to(bb, bb, dd, G[..., 0, 0]) + to(bb, dd, bb, G[..., 1, 1]) + to(dd, bb, bb, G[..., 2, 2])
                            + 2.0 * (to(bb, bd, bd, G[..., 0, 1]) + to(bd, bb, bd, G[..., 0, 2]) + to(bd, bd, bb, G[..., 1, 2])))
            d.index_add_(0, self.index(a, b), v.reshape(-1))
        return d

    def solve(self, alpha, b, x, diag):
        x = x.clone()
        r = b - self.apply(x, alpha, 1.0)
        z = r / diag
        p, rz, stop = z.clone(), torch.dot(r, z), 1e-13 * torch.linalg.norm(b)
        for _ in range(3000):
            if torch.linalg.norm(r) <= stop:
                break
            q = self.apply(p, alpha, 1.0)
            a = rz / torch.dot(p, q)
            x += a * p
            r -= a * q
            z = r / diag
            new = torch.dot(r, z)
            p = z + (new / rz) * p
            rz = new
        return x


def _currents(u_star, h):
    m = IONIC
    v = (u_star - m["u_rest"]) / m["u_amp"]
    return -m["u_amp"] * (h * v * v * (1.0 - v) / m["tau_in"] - v / m["tau_out"])


def _rates(u_star):
    m = IONIC
    v = (u_star - m["u_rest"]) / m["u_amp"]
    s = torch.sigmoid((v - m["v_gate"]) / m["kappa"])
    return (1.0 - s) / m["tau_open"], s / m["tau_close"]


def _step(op, f, n, mask, amp, t0, t1, mass, solve):
    """One BDF step of the partitioned scheme from fields f at step count n."""
    t = (n + 1) * DT
    app = amp * mask if t0 < t <= t1 else 0.0
    if n == 0:
        us, (a, b) = f["u"], _rates(f["u"])
        h = (f["h"] + DT * a) / (1.0 + DT * (a + b))
        hist, alpha = f["u"] / DT, 1.0 / DT
    else:
        us = 2.0 * f["u"] - f["u_prev"]
        a, b = _rates(us)
        h = (4.0 * f["h"] - f["h_prev"] + 2.0 * DT * a) / (3.0 + 2.0 * DT * (a + b))
        hist, alpha = (4.0 * f["u"] - f["u_prev"]) / (2.0 * DT), 1.5 / DT
    u = solve(alpha, mass(hist - _currents(us, h) + app), f["u"])
    return {"u": u, "u_prev": f["u"], "h": h, "h_prev": f["h"]}


def _mask(c, op, device):
    """Nodes inside the closed stimulus box (on the perturbed mesh)."""
    (x0, y0, z0, x1, y1, z1), _, _, _ = _stimulus(c)
    x = torch.as_tensor(op.nodes, dtype=torch.float64, device=device)
    N = torch.stack([0.5 * (1 - x), 0.5 * (1 + x)], 1)
    mask = torch.zeros(op.ndofs, dtype=torch.float64, device=device)
    for a, b in op.chunks():
        P = torch.einsum("zk,yj,xi,ekjid->ezyxd", N, N, N, op.X[a:b])
        inside = ((P >= torch.tensor([x0, y0, z0], device=device)) & (P <= torch.tensor([x1, y1, z1], device=device))).all(-1)
        mask[op.index(a, b)] = inside.reshape(-1).to(torch.float64)
    return mask


def _vcycle(c, vertices, tissue, r, device):
    """The V-cycle with one p-level below the fine one, as its definition reads (Section 4.3)."""
    fine = _Operator(c, vertices, device)
    pc = max(1, c["p"] // 2)
    coarse = _Operator(c, vertices, device, pc)
    inv, lam = [], []
    for op in (fine, coarse):
        op.set_tissue(tissue)
        d = 1.0 / op.diagonal(ALPHA, 1.0)
        # largest eigenvalue of D^{-1} A: Lanczos tridiagonal of ten Jacobi-PCG steps
        i = torch.arange(op.ndofs, dtype=torch.int64, device=device)
        v = ((i * 2654435761) & 0xFFFFFFFF).to(torch.float64) / 4294967296.0 - 0.5
        z = d * v
        q, rz, al, be = z.clone(), float(torch.dot(v, z)), [], []
        for _ in range(10):
            y = op.apply(q, ALPHA, 1.0)
            al.append(rz / float(torch.dot(q, y)))
            v = v - al[-1] * y
            z = d * v
            new = float(torch.dot(v, z))
            be.append(new / rz)
            rz, q = new, z + be[-1] * q
        T = np.diag([1.0 / al[j] + (be[j - 1] / al[j - 1] if j else 0.0) for j in range(10)])
        for j in range(9):
            T[j, j + 1] = T[j + 1, j] = math.sqrt(be[j]) / al[j]
        inv.append(d)
        lam.append(float(np.linalg.eigvalsh(T)[-1]))

    def smooth(k, b, x, degree):
        lo, hi = 0.08 * lam[k], 1.2 * lam[k]
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        sigma = theta / delta
        op, rho, d = (fine, coarse)[k], delta / theta, None
        for j in range(degree):
            res = b if x is None else b - op.apply(x, ALPHA, 1.0)
            if j == 0:
                d = inv[k] * res / theta
            else:
                new = 1.0 / (2.0 * sigma - rho)
                d = new * rho * d + 2.0 * new / delta * (inv[k] * res)
                rho = new
            x = d.clone() if x is None else x + d
        return x

    P = torch.as_tensor(_lagrange(coarse.nodes, fine.nodes)[0], dtype=torch.float64, device=device)
    fi, ci, n, m = fine.index(0, fine.ne), coarse.index(0, coarse.ne), c["p"] + 1, pc + 1
    count = torch.zeros_like(r).index_add_(0, fi, torch.ones(fi.numel(), dtype=torch.float64, device=device))
    x = smooth(0, r, None, c["degree"])
    res = (r - fine.apply(x, ALPHA, 1.0)) / count
    e = torch.einsum("zk,yj,xi,ezyx->ekji", P, P, P, res[fi].reshape(-1, n, n, n))
    b = torch.zeros(coarse.ndofs, dtype=torch.float64, device=device).index_add_(0, ci, e.reshape(-1))
    xc = smooth(1, b, None, c["coarse_degree"])
    up = torch.empty_like(r)
    up[fi] = torch.einsum("zk,yj,xi,ekji->ezyx", P, P, P, xc[ci].reshape(-1, m, m, m)).reshape(-1)
    return smooth(0, r, x + up, c["degree"])


class _Solve(torch.autograd.Function):
    """u = (alpha M + K(tissue))^{-1} b with gradients in b and the tissue."""

    @staticmethod
    def forward(ctx, b, sl, st, th, op, alpha, diag, x0):
        u = op.solve(alpha, b.detach(), x0.detach(), diag)
        ctx.save_for_backward(u, sl, st, th)
        ctx.more = (op, alpha, diag)
        return u

    @staticmethod
    def backward(ctx, g):
        u, sl, st, th = ctx.saved_tensors
        op, alpha, diag = ctx.more
        w = op.solve(alpha, g, torch.zeros_like(g), diag)
        par = [q.detach().requires_grad_(True) for q in (sl, st, th)]
        n = op.p + 1
        with torch.enable_grad():
            i = op.index(0, op.ne)
            G, W = op.metric(0, op.ne, par)
            E = op.element(u[i].reshape(-1, n, n, n), G, W, 0.0, 1.0)
            e = -(w[i].reshape(-1, n, n, n) * E).sum()
        return (w, *torch.autograd.grad(e, par), None, None, None, None)


def exact(case, seed):
    c, device = dict(case), "cuda" if torch.cuda.is_available() else "cpu"
    kind = c["kind"]
    vertices = _vertices(c, seed)
    put = lambda a: [torch.as_tensor(q, dtype=torch.float64, device=device) for q in a]  # noqa: E731
    tissue = put(_tissue(c, seed + 31 if kind == "tissue" else seed))
    if kind == "vcycle":
        return _vcycle(c, vertices, tissue, _vector(_nodes(c), seed, torch.float64, device), device)
    op = _Operator(c, vertices, device)
    op.set_tissue(tissue)
    if kind == "apply":
        u = _vector(op.ndofs, seed, torch.float64, device)
        if c["prec"] in ("fp32", "bf16"):
            u = u.to(torch.float32).to(torch.float64)
        return op.apply(u, ALPHA, 1.0)
    if kind == "tissue":
        return op.diagonal(ALPHA, 1.0)
    f = _fields(c, seed, device)
    mask = _mask(c, op, device)
    _, amp, t0, t1 = _stimulus(c)
    mass = lambda g: op.apply(g, 1.0, 0.0)  # noqa: E731
    if kind in ("step", "host"):
        diag = op.diagonal(ALPHA, 1.0)
        solve = lambda alpha, b, x: op.solve(alpha, b, x, diag)  # noqa: E731
        top = torch.full_like(f["u"], -1.0)
        for k in range(c["steps"]):
            new = _step(op, f, 5 + k, mask, amp, t0, t1, mass, solve)
            top = torch.maximum(top, (3.0 * new["u"] - 4.0 * f["u"] + f["u_prev"]).abs() / (2.0 * DT))
            f = new
        out = {k: f[k] for k in ("u", "u_prev", "h", "h_prev")}
        if c.get("track"):
            out["dudt_max"] = top
        return out
    par = [q.clone().requires_grad_(True) for q in tissue]
    sens = torch.as_tensor(_sensors(c, seed), device=device)
    target = -85.0 + 10.0 * _vector(c["steps"] * sens.numel(), seed + 3, torch.float64, device).reshape(c["steps"], -1)
    diag = {a: op.diagonal(a, 1.0) for a in (1.0 / DT, ALPHA)}
    solve = lambda alpha, b, x: _Solve.apply(b, *par, op, alpha, diag[alpha], x)  # noqa: E731
    f = {"u": f["u"], "u_prev": f["u"], "h": f["h"], "h_prev": f["h"]}
    rows = []
    for k in range(c["steps"]):
        f = _step(op, f, k, mask, amp, t0, t1, mass, solve)
        rows.append(f["u"][sens])
    T = torch.stack(rows)
    (0.5 * DT * ((T - target) ** 2).sum()).backward()
    return {"traces": T.detach(), "grad": [q.grad for q in par]}
