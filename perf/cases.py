"""The calls whose speed matters to a program that uses this framework.

Every case is one call, or one step's few calls, of the public Python API
(``paper_2311_09465_gb300``) on a rounded duct meshed with linear tetrahedra:
inflow at z = 0, no-slip walls, a resistance outlet at z = L, Re 500, Wo 10,
the regime of the repository's junction workload.  Sizes run from the small
pipe of the tests (9.6 k tetrahedra and below) to the bench junction's size
(190 k), mode counts over the compiled ones.

kinds
  residual      ts_residual: the nonlinear residual, once per Newton step
  jvp           ts_jvp: one tangent product, the inner loop of GMRES
  newton        ts_solve over a fixed number of pseudo-time Newton steps, each
                with 30 Krylov products (the bench's step)
  blocks        ts_block_diagonal, inverted: the nodal block preconditioner's
                set-up, once per Newton step
  assembled     ts_assemble and 16 ts_spmv products with it
  tracer        ts_tracer_residual: the scalar convection-diffusion residual
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2311_09465_gb300 as ts

RHO, RE, WO, DIAMETER = 1.0, 500.0, 10.0, 2.0
MU = RHO * DIAMETER / RE
OMEGA = WO * WO * MU / (RHO * DIAMETER * DIAMETER)
C_I, C1 = 3.0, 1.5
DT = 0.5                      # pseudo-time step of the products
KAPPA = 0.01                  # tracer diffusivity
RESISTANCE = 1.0
WALL, INLET, OUTLET = 0, 1, 3
KRYLOV = 30
SPMV_VECTORS = 16


def listed():
    return [
        # the tests' small pipe: launches and latency decide
        dict(name="residual64_n3_small", kind="residual", bits=64, N=3, across=8, along=25),
        # the bench junction's size and mode count: the residual of every Newton step
        dict(name="residual64_n7_large", kind="residual", bits=64, N=7, across=23, along=59),
        # the mode-count study's reference solve (N = 15 on 12 k tetrahedra)
        dict(name="residual64_n15", kind="residual", bits=64, N=15, across=9, along=26),
        # the FP32 residual on a mid-sized mesh
        dict(name="residual32_n5_mid", kind="residual", bits=32, N=5, across=15, along=39),
        # a product on the small pipe: launch latency
        dict(name="jvp32_n3_small", kind="jvp", bits=32, N=3, variant="lin_a", across=8, along=25),
        # the GMRES hot loop of the bench
        dict(name="jvp32_n7_large", kind="jvp", bits=32, N=7, variant="lin_a", across=23, along=59),
        # the mode sweep's largest N
        dict(name="jvp32_n15_mid", kind="jvp", bits=32, N=15, variant="lin_a", across=15, along=39),
        # the plain FP64 solve's inner loop
        dict(name="jvp64_n7_mid", kind="jvp", bits=64, N=7, variant="lin_a", across=15, along=39),
        # whole call: two pseudo-time Newton steps of the mixed-precision solver
        dict(name="newton_n7_large", kind="newton", N=7, steps=2, across=23, along=59),
        # block preconditioner set-up of a junction solve's Newton step
        dict(name="blocks_n7_mid", kind="blocks", N=7, across=15, along=39),
        # assembled paper-variant tangent and its products
        dict(name="assembled_n5_mid", kind="assembled", N=5, across=15, along=39),
        # scalar transport
        dict(name="tracer64_n7_mid", kind="tracer", bits=64, N=7, across=12, along=31),
    ]


#: kind -> (weight, mode counts, smallest and largest number of tetrahedra at N <= 7)
_RANGES = {
    "residual": (4, (2, 3, 4, 5, 7, 10, 15), 1500, 185000),
    "jvp": (4, (2, 3, 4, 5, 7, 10, 15), 1500, 185000),
    "newton": (1, (3, 5, 7), 9000, 120000),
    "blocks": (1, (2, 3, 5, 7), 1500, 52000),
    "assembled": (1, (2, 3, 5, 7), 1500, 52000),
    "tracer": (1, (3, 5, 7, 10), 1500, 52000),
}


def draw(rng):
    kinds = list(_RANGES)
    kind = rng.choices(kinds, [_RANGES[k][0] for k in kinds])[0]
    _, modes, lo, hi = _RANGES[kind]
    N = rng.choice(modes)
    case = dict(kind=kind, N=N)
    if kind in ("residual", "jvp", "tracer"):
        case["bits"] = rng.choice((32, 64))
    if kind == "jvp":
        case["variant"] = rng.choice(("lin_a", "lin_a", "frozen", "paper"))
    if kind == "newton":
        case["steps"] = rng.choice((1, 2))
    if N > 7:                                 # the work per element grows with N^3
        hi = max(2 * lo, hi * (7 / N) ** 3)
    if case.get("bits") == 64 and kind == "jvp":
        hi = min(hi, 60000)
    tets = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    aspect = rng.uniform(1.5, 4.0)            # cells along per cell across
    across = max(3, round((tets / (6 * aspect)) ** (1 / 3)))
    case["across"] = across
    case["along"] = max(3, int(tets / (6 * across * across)))
    return case


# ------------------------------------------------------------------ inputs

_KUHN = np.array([[0, 1, 3, 7], [0, 1, 5, 7], [0, 2, 3, 7], [0, 2, 6, 7], [0, 4, 5, 7], [0, 4, 6, 7]])


def _mesh(across, along, seed):
    """Rounded duct of diameter 2 (a square lattice bent towards the circle),
    six tetrahedra per lattice cell, interior nodes moved at random."""
    n, m = across, along
    h = DIAMETER / n
    i, j, k = np.meshgrid(np.arange(n + 1), np.arange(n + 1), np.arange(m + 1), indexing="ij")
    idx = lambda a, b, c: (c * (n + 1) + b) * (n + 1) + a                           # noqa: E731
    order = np.argsort(idx(i, j, k).ravel(), kind="stable")
    i, j, k = (a.ravel()[order] for a in (i, j, k))
    inner = (i > 0) & (i < n) & (j > 0) & (j < n) & (k > 0) & (k < m)
    rng = np.random.default_rng(seed)
    move = 0.12 * (2 * rng.random((i.size, 3)) - 1) * inner[:, None]
    x, y = 2 * (i + move[:, 0]) / n - 1, 2 * (j + move[:, 1]) / n - 1
    z = (k + move[:, 2]) * h
    bend = 0.8
    xyz = np.stack([x * np.sqrt(1 - 0.5 * bend * y * y), y * np.sqrt(1 - 0.5 * bend * x * x), z], axis=1)
    ci, cj, ck = np.meshgrid(np.arange(n), np.arange(n), np.arange(m), indexing="ij")
    ci, cj, ck = (a.transpose(2, 1, 0).ravel() for a in (ci, cj, ck))
    corner = np.stack([idx(ci + (b & 1), cj + ((b >> 1) & 1), ck + (b >> 2)) for b in range(8)], axis=1)
    tets = corner[:, _KUHN].reshape(-1, 4).astype(np.int32)
    p = xyz[tets]
    vol = np.einsum("ei,ei->e", p[:, 1] - p[:, 0], np.cross(p[:, 2] - p[:, 0], p[:, 3] - p[:, 0]))
    tets[vol < 0] = tets[vol < 0][:, [0, 2, 1, 3]]
    # boundary triangles: faces that one tetrahedron has
    faces = np.concatenate([tets[:, f] for f in ([1, 2, 3], [0, 3, 2], [0, 1, 3], [0, 2, 1])])
    key = np.sort(faces.astype(np.int64), axis=1)
    key = (key[:, 0] * xyz.shape[0] + key[:, 1]) * xyz.shape[0] + key[:, 2]
    _, first, count = np.unique(key, return_index=True, return_counts=True)
    bfaces = np.ascontiguousarray(faces[np.sort(first[count == 1])])
    kk = k[bfaces]
    tag = np.where((kk == 0).all(1), INLET, np.where((kk == m).all(1), OUTLET, WALL)).astype(np.int32)
    mask = np.zeros(xyz.shape[0], dtype=bool)
    mask[bfaces[tag != OUTLET].ravel()] = True
    return SimpleNamespace(xyz=np.ascontiguousarray(xyz), tets=tets, bfaces=bfaces, btag=tag, n_nodes=xyz.shape[0],
                           n_tets=tets.shape[0], dirichlet=mask)


def _field(mesh, N, fields, seed, flow):
    """[V, fields, N, 2] float64 on the GPU: smooth functions of position with
    10 % noise, decaying like 1/(1+n)^2; `flow` adds the duct's mean profile
    to the axial velocity and holds the walls."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.tensor(mesh.xyz, dtype=torch.float64, device="cuda")
    V = x.shape[0]
    xc = (x - x.mean(0)) / float(np.ptp(mesh.xyz, axis=0).max())
    basis = torch.cat([torch.ones(V, 1, dtype=torch.float64, device="cuda"), xc, xc * xc, torch.sin(3 * xc)], 1)
    coef = torch.randn(basis.shape[1], fields * N * 2, generator=g, dtype=torch.float64, device="cuda")
    y = (basis @ coef).reshape(V, fields, N, 2)
    y += 0.1 * torch.randn(V, fields, N, 2, generator=g, dtype=torch.float64, device="cuda")
    y /= ((1.0 + torch.arange(N, dtype=torch.float64, device="cuda")) ** 2)[:, None]
    if flow:
        y *= 0.3
        r2 = (x[:, 0] ** 2 + x[:, 1] ** 2).clamp(max=1.0)
        y[:, 2, 0, 0] += 2 * (1 - r2)
        wall = torch.zeros(V, dtype=torch.bool, device="cuda")
        wall[torch.tensor(mesh.bfaces[mesh.btag == WALL].ravel().astype(np.int64), device="cuda")] = True
        y[wall, :3] = 0
    y[:, :, 0, 1] = 0
    return y.contiguous()


def _problem(mesh, N, variant, dt):
    return ts.GLSProblem(SimpleNamespace(mesh=mesh, N=N, rho=RHO, mu=MU, omega=OMEGA, C_I=C_I, c1=C1,
                                         dirichlet_tags=(WALL, INLET), resistance={OUTLET: RESISTANCE}),
                         variant=variant, dt_pseudo=dt)


def _inputs(case, seed):
    """mesh and fields of a case, the same for prepare() and exact()."""
    mesh = _mesh(case["across"], case["along"], seed)
    N, kind = case["N"], case["kind"]
    dtype = torch.float32 if case.get("bits") == 32 else torch.float64
    if kind == "tracer":
        a = _field(mesh, N, 4, seed, True)[:, :3].contiguous()
        return mesh, a.to(dtype), _field(mesh, N, 1, seed + 1000, False)[:, 0].contiguous().to(dtype)
    y = _field(mesh, N, 4, seed, True)
    if kind == "jvp":
        return mesh, y.to(dtype), _field(mesh, N, 4, seed + 1000, False).to(dtype)
    if kind == "assembled":
        v = torch.stack([_field(mesh, N, 4, seed + 1000 + k, False) for k in range(SPMV_VECTORS)])
        return mesh, y, v.float()
    return mesh, y.to(dtype), None


def prepare(case, seed):
    mesh, y, v = _inputs(case, seed)
    N, kind = case["N"], case["kind"]
    s = SimpleNamespace(case=case, y=y, v=v)
    if kind == "tracer":
        s.mesh = ts.ts_mesh_load(mesh.xyz, mesh.tets, mesh.bfaces, mesh.btag)
        s.tracer = ts.Tracer(s.mesh, mesh.n_nodes, N, KAPPA, OMEGA, C_I, dirichlet_tags=(WALL, INLET))
        s.out = torch.empty_like(v)
        s.owner = _MeshOwner(s.mesh, s.tracer)
        return s
    variant = "paper" if kind == "assembled" else case.get("variant", "lin_a")
    s.problem = _problem(mesh, N, variant, DT)
    if kind == "residual":
        s.out = torch.empty_like(y)
    elif kind == "jvp":
        s.problem.residual(y)
        s.out = torch.empty_like(v)
    elif kind == "blocks":
        s.problem.residual(y)
    elif kind == "assembled":
        s.problem.residual(y)
        s.out = torch.empty_like(v)
    return s


class _MeshOwner:
    """Frees the tracer before the mesh it was made on."""

    def __init__(self, mesh, tracer):
        self.mesh, self.tracer = mesh, tracer

    def __del__(self):
        try:
            self.tracer.close()
            ts.ts_mesh_free(self.mesh)
        except Exception:
            pass


def run(s):
    kind = s.case["kind"]
    if kind == "residual":
        return s.problem.residual(s.y, s.out)
    if kind == "jvp":
        return s.problem.jvp(s.v, s.out)
    if kind == "newton":
        y = s.y.clone()
        rep = s.problem.solve(y, precision=32, tol=1e-300, max_steps=s.case["steps"], krylov=KRYLOV, eps_ls=1e-30,
                              max_matvec=KRYLOV, precond=1, raise_on_noconv=False, reject=0.0)
        return {"y": y, "steps": rep["steps"], "matvecs": rep["matvecs"]}
    if kind == "blocks":
        return s.problem.block_diagonal(invert=True)
    if kind == "assembled":
        s.problem.assemble()
        for k in range(SPMV_VECTORS):
            s.problem.spmv(s.v[k], s.out[k])
        return s.out
    return s.tracer.residual(s.y, s.v, s.out)


# ------------------------------------------------------------------ the work of a pass

def work(case):
    """Inputs and outputs once, and the arithmetic of the method as stated:
    M and its inverse square root at four points an element (45 n^3 flops, n = 2N-1),
    the convective products on 3N-2 time samples, tau times the strong residual."""
    N, kind = case["N"], case["kind"]
    E = 6 * case["across"] ** 2 * case["along"]
    V = (case["across"] + 1) ** 2 * (case["along"] + 1)
    n, C, K = 2 * N - 1, 2 * N, 3 * N - 2
    b = case.get("bits", 64) // 8
    mesh = 16 * E + 3 * b * V
    field = 4 * C * b * V
    tau = 4 * 45 * n ** 3
    cache = 4 * b * n * (n + 1) // 2 * E
    # per element: 33 transforms (12 + 12 at points, 9 of the SUPG sums), tau, products on samples
    element = 2 * (33 * C * K // 2 + 12 * n * n + 100 * K + 40 * C)
    if kind == "residual":
        return {"bytes": mesh + 2 * field + cache, "flops": E * (tau + element)}
    if kind == "jvp":
        extra = 2 if case["variant"] == "lin_a" else 1
        return {"bytes": mesh + 3 * field + cache + (12 * C * b * E if extra == 2 else 0), "flops": E * element * extra}
    if kind == "newton":
        s, m = case["steps"], KRYLOV
        product = 16 * E + 12 * V + 3 * 16 * C * V + 16 * E * n * (n + 1) // 2 + 48 * C * E
        # the basis is read twice by each Gram-Schmidt step
        basis = 2 * 8 * 4 * C * V * m * (m + 1) // 2
        return {"bytes": (s + 1) * (mesh + 2 * field + cache) + s * (m * product + basis),
                "flops": (s + 1) * E * (tau + element) + s * m * (2 * E * element + 4 * 4 * C * V * m)}
    if kind == "blocks":
        # per (element, node): three n x n products at four points; an inversion per node
        return {"bytes": mesh + field + cache + 4 * 64 * N * N * V, "flops": 4 * E * 4 * 3 * 2 * n ** 3 + 2 * (8 * N) ** 3 * V}
    if kind == "assembled":
        links = 14 * V
        record = 4 * 8 * n * n
        return {"bytes": mesh + field + cache + links * record * (1 + SPMV_VECTORS) + SPMV_VECTORS * 2 * 16 * C * V,
                "flops": 4 * E * 4 * 4 * 2 * n ** 3 // 2 + SPMV_VECTORS * links * 2 * 10 * n * n}
    return {"bytes": mesh + 5 * field // 4, "flops": E * (tau + element // 3)}


# ------------------------------------------------------------------ the results in 64 bits

_BARY = np.where(np.eye(4) > 0, 0.5854101966249685, 0.1381966011250105)


class _Exact:
    """The discrete equations in float64 with explicit convolution matrices, in
    the orthonormal real basis (x_0, sqrt2 Re x_n, sqrt2 Im x_n) of a
    conjugate-symmetric mode vector."""

    def __init__(self, mesh, N):
        self.N, self.n = N, 2 * N - 1
        dev = dict(dtype=torch.float64, device="cuda")
        n, full = self.n, range(-(N - 1), N)
        P = np.zeros((n, n), dtype=complex)             # complex modes = P xi
        P[N - 1, 0] = 1
        for k in range(1, N):
            P[N - 1 + k, 2 * k - 1] = P[N - 1 - k, 2 * k - 1] = 1 / math.sqrt(2)
            P[N - 1 + k, 2 * k], P[N - 1 - k, 2 * k] = 1j / math.sqrt(2), -1j / math.sqrt(2)
        B = np.zeros((n, n, n))                          # convolution matrix = sum_c xi_c B[c]
        for c in range(n):
            a = P[:, c]
            A = np.array([[a[N - 1 + p - q] if abs(p - q) < N else 0 for q in full] for p in full])
            B[c] = (P.conj().T @ A @ P).real
        D = P.conj().T @ np.diag([1j * p for p in full]) @ P
        self.B, self.D = torch.tensor(B, **dev), torch.tensor(D.real, **dev)
        self.bary = torch.tensor(_BARY, **dev)
        x = torch.tensor(mesh.xyz, **dev)
        self.tets = torch.tensor(mesh.tets.astype(np.int64), device="cuda")
        p = x[self.tets]
        inv = torch.linalg.inv((p[:, 1:] - p[:, :1]).transpose(1, 2))      # d xi_k / d x_i
        self.dN = torch.cat([-inv.sum(1, keepdim=True), inv], 1)
        self.vol = torch.linalg.det(p[:, 1:] - p[:, :1]).abs() / 6
        self.G = inv.transpose(1, 2) @ inv
        self.mask = torch.tensor(mesh.dirichlet, device="cuda")
        f = torch.tensor(mesh.bfaces[mesh.btag == OUTLET].astype(np.int64), device="cuda")
        c = torch.linalg.cross(x[f[:, 1]] - x[f[:, 0]], x[f[:, 2]] - x[f[:, 0]]) / 6
        self.outlet = torch.zeros_like(x)
        self.outlet.index_add_(0, f.reshape(-1), c.repeat_interleave(3, 0))
        self.step = max(64, int(3e8) // (n * n * 8 * 12 * 3))

    def xi(self, y):
        y = y.double()
        r = torch.empty(*y.shape[:-2], self.n, dtype=torch.float64, device="cuda")
        r[..., 0] = y[..., 0, 0]
        r[..., 1::2], r[..., 2::2] = math.sqrt(2) * y[..., 1:, 0], math.sqrt(2) * y[..., 1:, 1]
        return r

    def stored(self, r):
        y = torch.zeros(*r.shape[:-1], self.N, 2, dtype=torch.float64, device="cuda")
        y[..., 0, 0] = r[..., 0]
        y[..., 1:, 0], y[..., 1:, 1] = r[..., 1::2] / math.sqrt(2), r[..., 2::2] / math.sqrt(2)
        return y

    def conv(self, a):
        return torch.einsum("...c,crs->...rs", a, self.B)

    def tau(self, A, G, nu):
        GA = torch.einsum("eij,eqjrs->eqirs", G, A)
        M = torch.matmul(A, GA).sum(2)
        M = 0.5 * (M + M.transpose(-1, -2))
        M += (C_I * nu * nu * (G * G).sum((1, 2)))[:, None, None, None] * torch.eye(self.n, dtype=M.dtype, device="cuda")
        lam, vec = torch.linalg.eigh(M)
        return torch.matmul(vec / lam.sqrt()[..., None, :], vec.transpose(-1, -2))

    def chunks(self):
        for s in range(0, self.tets.shape[0], self.step):
            e = slice(s, min(s + self.step, self.tets.shape[0]))
            yield self.tets[e], self.dN[e], self.vol[e], self.G[e]

    def apply(self, y0, v, variant, mass):
        """The residual at y0 (v None), or the tangent product at y0 with v."""
        residual = v is None
        Y0 = self.xi(y0)
        Y = Y0 if residual else self.xi(v)
        if not residual:
            Y = Y.clone()
            Y[self.mask, :3] = 0
        out = torch.zeros_like(Y)
        om = OMEGA * self.D
        for t, dN, vol, G in self.chunks():
            u0, u, p = Y0[t, :3], Y[t, :3], Y[t, 3]
            w = vol / 4
            uq, gu, gp = (torch.einsum("qa,eaic->eqic", self.bary, u), torch.einsum("eaj,eaic->eijc", dN, u),
                          torch.einsum("eaj,eac->ejc", dN, p))
            A = self.conv(torch.einsum("qa,eaic->eqic", self.bary, u0))
            tau = self.tau(A, G, MU / RHO)
            c = torch.einsum("eqjrs,eijs->eqir", A, gu)
            if variant == "lin_a" and not residual:
                gu0, gp0 = torch.einsum("eaj,eaic->eijc", dN, u0), torch.einsum("eaj,eac->ejc", dN, Y0[t, 3])
                L0 = RHO * (torch.einsum("rs,qa,eais->eqir", om, self.bary, u0) + torch.einsum("eqjrs,eijs->eqir", A, gu0)) + gp0[:, None]
                T0 = torch.einsum("eqrs,eqis->eqir", tau, L0)
                Av = self.conv(uq)
                c = c + torch.einsum("eqjrs,eijs->eqir", Av, gu0)
            Lu = RHO * (torch.einsum("rs,eqis->eqir", om, uq) + c)
            Lp = gp[:, None].expand_as(Lu)
            T = torch.einsum("eqrs,eqis->eqir", tau, Lu if variant == "paper" and not residual else Lu + Lp)
            Tc = torch.einsum("eqrs,eqis->eqir", tau, Lp) if variant == "paper" and not residual else T
            AT = torch.einsum("eqjrs,eqis->eqjir", A, T)
            if variant == "lin_a" and not residual:
                AT = AT + torch.einsum("eqjrs,eqis->eqjir", Av, T0)
            r = torch.zeros_like(Y[t])
            r[:, :, :3] = torch.einsum("qa,eqir->eair", self.bary, Lu - torch.einsum("rs,eqis->eqir", om, T))
            r[:, :, :3] += torch.einsum("eaj,eqjir->eair", dN, AT)
            r[:, :, :3] -= torch.einsum("eai,er->eair", dN, p.sum(1))
            r[:, :, :3] += 4 * MU * torch.einsum("eaj,eijr->eair", dN, gu)
            if mass and not residual:
                r[:, :, :3] += 0.2 * mass * (u.sum(1, keepdim=True) + u)
            r[:, :, 3] = torch.einsum("eiir->er", gu)[:, None] + torch.einsum("eai,eqir->ear", dN, Tc) / RHO
            out.index_add_(0, t.reshape(-1), (w[:, None, None, None] * r).reshape(-1, 4, self.n))
        flux = torch.einsum("vi,vir->r", self.outlet, Y[:, :3])
        out[:, :3] += RESISTANCE * self.outlet[:, :, None] * flux
        out[self.mask, :3] = 0
        return self.stored(out)

    def tracer(self, a, phi):
        A_, F = self.xi(a), self.xi(phi)
        out = torch.zeros_like(F)
        om = OMEGA * self.D
        for t, dN, vol, G in self.chunks():
            A = self.conv(torch.einsum("qa,eaic->eqic", self.bary, A_[t]))
            tau = self.tau(A, G, KAPPA)
            g, f = torch.einsum("eaj,eac->ejc", dN, F[t]), torch.einsum("qa,eac->eqc", self.bary, F[t])
            res = torch.einsum("rs,eqs->eqr", om, f) + torch.einsum("eqjrs,ejs->eqr", A, g)
            T = torch.einsum("eqrs,eqs->eqr", tau, res)
            r = torch.einsum("qa,eqr->ear", self.bary, res - torch.einsum("rs,eqs->eqr", om, T))
            r += torch.einsum("eaj,eqjrs,eqs->ear", dN, A, T) + 4 * KAPPA * torch.einsum("eaj,ejr->ear", dN, g)
            out.index_add_(0, t.reshape(-1), (vol[:, None, None] / 4 * r).reshape(-1, self.n))
        out[self.mask] = 0
        return self.stored(out)

    def blocks(self, y0, mass):
        """Inverted nodal blocks of the frozen tangent (TS_JVP_FROZEN's nodal
        couplings), in stored coordinates, column-major."""
        n, N = self.n, self.N
        Y0 = self.xi(y0)
        V = Y0.shape[0]
        H = torch.zeros(V, 4, n, 4, n, dtype=torch.float64, device="cuda")
        eye, om = torch.eye(n, dtype=torch.float64, device="cuda"), OMEGA * self.D
        for t, dN, vol, G in self.chunks():
            A = self.conv(torch.einsum("qa,eaic->eqic", self.bary, Y0[t, :3]))
            tau = self.tau(A, G, MU / RHO)
            for a in range(4):
                lam, d = self.bary[:, a], dN[:, a]
                GA = torch.einsum("ej,eqjrs->eqrs", d, A)
                S = RHO * (lam[:, None, None] * om + GA)
                W = GA - lam[:, None, None] * om
                WT, TS = torch.matmul(W, tau), torch.matmul(tau, S)
                K = (lam[:, None, None] * S + torch.matmul(WT, S)).sum(1)
                K += (4 * MU * (d * d).sum(1) + 0.4 * mass)[:, None, None] * eye
                b = torch.zeros(t.shape[0], 4, n, 4, n, dtype=torch.float64, device="cuda")
                for i in range(3):
                    b[:, i, :, i] = K
                b[:, :3, :, 3] = d[:, :, None, None] * (WT.sum(1) - eye)[:, None]
                b[:, 3, :, :3] = (d[:, :, None, None] * (eye + TS.sum(1) / RHO)[:, None]).transpose(1, 2)
                b[:, 3, :, 3] = ((d * d).sum(1) / RHO)[:, None, None] * tau.sum(1)
                H.index_add_(0, t[:, a], b * (vol / 4)[:, None, None, None, None])
        o = self.outlet
        H[:, :3, :, :3] += RESISTANCE * torch.einsum("vi,vj,rs->virjs", o, o, eye)
        H[self.mask, :3] = 0
        H[self.mask, :, :, :3] = 0
        for i in range(3):
            H[self.mask, i, :, i] = eye
        inv = torch.linalg.inv(H.reshape(V, 4 * n, 4 * n)).reshape(V, 4, n, 4, n)
        scale = torch.full((n,), 1 / math.sqrt(2), dtype=torch.float64, device="cuda")
        scale[0] = 1
        inv = inv * scale[:, None, None] / scale
        at = torch.tensor([0] + list(range(2, 2 * N)), device="cuda")
        out = torch.zeros(V, 4, 2 * N, 4, 2 * N, dtype=torch.float64, device="cuda")
        for i in range(4):
            out[:, i, 1, i, 1] = 1
        out[:, :, at[:, None, None], torch.arange(4, device="cuda")[:, None], at] = inv
        return out.reshape(V, 8 * N, 8 * N).transpose(1, 2).contiguous()


def exact(case, seed):
    kind, N = case["kind"], case["N"]
    if kind == "newton":
        return None                          # a whole solver call
    mesh, y, v = _inputs(case, seed)
    X = _Exact(mesh, N)
    mass = C1 * RHO / DT
    if kind == "residual":
        return X.apply(y, None, "frozen", 0.0)
    if kind == "jvp":
        return X.apply(y, v, case["variant"], mass)
    if kind == "blocks":
        return X.blocks(y, mass)
    if kind == "assembled":
        return torch.stack([X.apply(y, v[k], "paper", mass) for k in range(SPMV_VECTORS)])
    return X.tracer(y, v)
