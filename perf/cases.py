"""Performance cases of the PCEXP library: what its users run, through the public binding.

A case names a mesh family and size, a DG order, a precision form and one call: a whole step
(``Context.set_state``, ``step``, ``get_state``), a few iterations of the steady march, one
residual / J v / J^T w, or the reverse of a step.  ``prepare`` makes the context and device
tensors such a program holds, ``run`` is one pass, and ``exact`` gives the same outputs from a
plain 64-bit torch restatement of the scheme kept in this file (its own bases, quadrature, fluxes,
faces and Krylov process).

States are coefficients in the binding's default basis.  The FP32-mixed form computes its
increments, residuals and products in FP32, so its results are returned as FP32 tensors (a
snapshot of such a run carries no more); results of the FP64 form stay FP64.
"""
import functools
import itertools
import math
import types

import numpy as np
import torch

from paper_1801_06300_gb300 import capi

GAMMA = 1.4
F64 = torch.float64

# ------------------------------------------------------------------------------- the cases


def _case(name, call, mesh, nx, p, m=0, **kw):
    c = dict(name=name, call=call, mesh=mesh, nx=nx, ny=nx, p=p, m=m, mixed=False, scheme="pcexp", dt="global",
             cfl=1.0, tol=0.0, steps=1)
    c.update(kw)
    return c


def listed():
    return [
        # a student's or a test's problem: the smallest whole step, a few hundred triangles
        _case("step_tri_small", "step", "square", 16, 1, 10, cfl=5.0),
        # the stiff stretched-mesh vortex at CFL 1000 with the Krylov tolerance (adaptive dimension)
        _case("step_tri_stretched_adaptive", "step", "stretched", 24, 2, 30, cfl=1000.0, tol=1e-5),
        # steady channel flow with local time steps, the FP32-mixed form: thousands of such steps
        _case("step_bump_mixed", "step", "bump", 192, 2, 30, ny=64, mixed=True, dt="local", cfl=20.0),
        # the same channel marched to steady state in FP64 with the CFL ramp, three iterations at a time
        _case("march_bump_fp64", "march", "bump", 96, 2, 30, ny=32, dt="local", cfl=10.0, steps=3),
        # unsteady vortex at high order on triangles, FP32-mixed production run
        _case("step_tri_p3_mixed", "step", "square", 256, 3, 30, mixed=True, cfl=20.0),
        # the largest: unsteady 3D vortex, FP32-mixed production run
        _case("step_tet_mixed", "step", "cube", 48, 2, 30, mixed=True, cfl=10.0),
        # 3D reference run in FP64
        _case("step_tet_fp64", "step", "cube", 20, 2, 30, cfl=10.0),
        # one-stage step at low order, open boundaries and walls, ragged size and Krylov dimension
        _case("exp1_tet_p1_mixed", "step", "boxcube", 21, 1, 17, mixed=True, scheme="exp1", cfl=10.0),
        # one operator evaluation (an outer time integrator of the user's own, output of R)
        _case("residual_tet_fp64", "residual", "cube", 24, 2),
        # one Jacobian-vector product (an outer linear solver)
        _case("jvp_tet_mixed", "jvp", "cube", 33, 2, mixed=True),
        # one transposed product (an outer adjoint solver), high order on triangles
        _case("vjp_tri_p3_fp64", "vjp", "square", 101, 3),
        # reverse of one step in a gradient computation on the channel
        _case("backward_bump_fp64", "backward", "bump", 96, 2, 30, ny=32, cfl=5.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "step", "march", "residual", "jvp", "vjp", "backward"])
    mixed = rng.random() < 0.5 and call not in ("backward", "march")
    mesh = rng.choice(["square", "bump", "cube", "boxcube"])
    solid = mesh in ("cube", "boxcube")
    p = rng.choice([0, 1, 1, 2, 2, 2] if solid else [0, 1, 2, 2, 3, 3])
    m = rng.randint(5, 32)
    kw = dict(mixed=mixed)
    if call == "backward":
        p, m = rng.choice([1, 2]), rng.randint(5, 30)
        nx = _log(rng, 4, 7) if solid else _log(rng, 8, 64)
    elif call == "march":
        mesh, solid, p = "bump", False, rng.choice([1, 2])
        nx = _log(rng, 12, 128)
    elif call == "step":
        nx = _log(rng, 4, 40 if mixed else 18) if solid else _log(rng, 6, 256 if mixed else 128)
    else:
        nx = _log(rng, 4, 40) if solid else _log(rng, 6, 320)
    ny = nx
    if mesh == "bump":
        ny = max(4, nx // 3 + rng.randint(-1, 2))
        # FP32-mixed steps stay at moderate local CFL numbers: at 100 its error from this start passes 1e-5
        kw.update(dt="local", cfl=10.0 if call == "march" else rng.uniform(5.0, 20.0 if mixed else 100.0))
    else:
        kw.update(cfl=rng.uniform(2.0, 20.0))
    if call == "backward":
        kw.update(dt="global", cfl=rng.uniform(2.0, 8.0))
    if call == "march":
        kw.update(steps=rng.randint(1, 3))
    if call == "step":
        kw.update(scheme=rng.choice(["pcexp", "pcexp", "exp1"]))
        if kw.get("dt") != "local" and rng.random() < 0.25:
            kw.update(scheme="etd2", steps=2)
    if call in ("residual", "jvp", "vjp"):
        m = 0
    c = _case("", call, mesh, nx, p, m, ny=ny, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------------------- the meshes


def _quads(nx, ny):
    j, i = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    v00 = (j * (nx + 1) + i).reshape(-1)
    v10, v01, v11 = v00 + 1, v00 + nx + 1, v00 + nx + 2
    return np.stack([v00, v10, v11, v00, v11, v01], 1).reshape(-1, 3).astype(np.int32)


@functools.lru_cache(maxsize=4)
def _mesh(kind, nx, ny):
    """A mesh as the binding takes it: periodic squares and cubes of side 10 or 20, the paper's
    stretched square of side 0.1, a channel with a bump (walls, open ends), a cube with open sides
    between two walls."""
    rng = np.random.default_rng(nx * 1000 + ny)
    if kind in ("square", "stretched"):
        jj, ii = (a.reshape(-1) for a in np.meshgrid(np.arange(nx + 1), np.arange(nx + 1), indexing="ij"))
        master = ((jj % nx) * nx + ii % nx).astype(np.int32)
        if kind == "square":
            side = 20.0 if nx >= 64 else 10.0
            off = 0.15 * side / nx * rng.uniform(-1, 1, (nx * nx, 2))
            x = np.stack([ii, jj], 1) * (side / nx) + off[master]
        else:
            side = 0.1
            s = 0.5 * (1.0 + (2.0 * np.arange(nx + 1) / nx - 1.0) ** 3) * side
            x = np.stack([s[ii], s[jj]], 1)
        elems, bf, bt, dim = _quads(nx, nx), np.zeros((0, 2), np.int32), np.zeros(0, np.int32), 2
    elif kind == "bump":
        jj, ii = np.meshgrid(np.arange(ny + 1), np.arange(nx + 1), indexing="ij")
        jx, jy = 0.15 * rng.uniform(-1, 1, (2, ny + 1, nx + 1))
        inx, iny = (ii > 0) & (ii < nx), (jj > 0) & (jj < ny)
        px = -1.0 + 3.0 / nx * (ii + np.where(inx, jx, 0.0))
        eta = (jj + np.where(iny, jy, 0.0)) / ny
        yb = np.where((px >= 0) & (px <= 1), 0.1 * np.sin(np.pi * px) ** 2, 0.0)
        x = np.stack([px, yb + (1 - yb) * eta], 2).reshape(-1, 2)
        master, side, dim = np.arange(len(x), dtype=np.int32), 0.0, 2
        elems, v = _quads(nx, ny), (jj * (nx + 1) + ii).astype(np.int32)
        lo, hi = np.stack([v[0, :-1], v[0, 1:]], 1), np.stack([v[-1, 1:], v[-1, :-1]], 1)
        le, ri = np.stack([v[1:, 0], v[:-1, 0]], 1), np.stack([v[:-1, -1], v[1:, -1]], 1)
        bf = np.concatenate([lo, hi, le, ri]).astype(np.int32)
        bt = np.repeat([capi.PCEXP_BC_SLIP_WALL, capi.PCEXP_BC_FARFIELD], [2 * nx, 2 * ny]).astype(np.int32)
    else:
        side, dim, n = 10.0, 3, nx
        kk, jj, ii = (a.reshape(-1) for a in np.meshgrid(*[np.arange(n + 1)] * 3, indexing="ij"))
        if kind == "cube":
            master = (((kk % n) * n + jj % n) * n + ii % n).astype(np.int32)
            off = 0.1 * side / n * rng.uniform(-1, 1, (n ** 3, 3))[master]
        else:
            master = np.arange((n + 1) ** 3, dtype=np.int32)
            inner = (ii > 0) & (ii < n) & (jj > 0) & (jj < n) & (kk > 0) & (kk < n)
            off = np.where(inner[:, None], 0.1 * side / n * rng.uniform(-1, 1, (len(master), 3)), 0.0)
        x = np.stack([ii, jj, kk], 1) * (side / n) + off
        ck, cj, ci = (a.reshape(-1) for a in np.meshgrid(*[np.arange(n)] * 3, indexing="ij"))
        base, step = (ck * (n + 1) + cj) * (n + 1) + ci, (1, n + 1, (n + 1) ** 2)
        tets = []
        for a, b, c in itertools.permutations(range(3)):
            t = [base, base + step[a], base + step[a] + step[b], base + sum(step)]
            if (a, b, c) not in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
                t[2], t[3] = t[3], t[2]  # odd paths: positive orientation
            tets.append(np.stack(t, 1))
        elems = np.stack(tets, 1).reshape(-1, 4).astype(np.int32)
        bf, bt = np.zeros((0, 3), np.int32), np.zeros(0, np.int32)
        if kind == "boxcube":
            lat, out = np.stack([ii, jj, kk], 1), []
            for f in range(4):
                fv = elems[:, [(f + k) % 4 for k in (1, 2, 3)]]
                P = lat[fv]
                on = ((P == 0).all(1) | (P == n).all(1)).any(1)
                out.append(fv[on])
            bf = np.concatenate(out).astype(np.int32)
            z = lat[bf][:, :, 2]  # walls below and above (the flow is along them), open sides
            bt = np.where((z == 0).all(1) | (z == n).all(1), capi.PCEXP_BC_SLIP_WALL, capi.PCEXP_BC_FARFIELD).astype(np.int32)
    return types.SimpleNamespace(dim=dim, coords=np.ascontiguousarray(x, np.float64), elems=np.ascontiguousarray(elems),
                                 vert_master=master, bfaces=bf, btags=bt, side=side)


def _freestream(mesh_kind):
    alpha = {"bump": 0.0, "stretched": 0.0, "boxcube": 30.0}.get(mesh_kind, 45.0)
    return types.SimpleNamespace(gamma=GAMMA, mach=0.5, alpha_deg=alpha, rho=1.0, p=1.0)


# ------------------------------------------------------- basis, states (torch, 64 bits)


def _gauss(n, a):
    """Gauss-Jacobi rule on [0, 1] for the weight (1 - t)^a, a = 0, 1, 2 (Golub-Welsch)."""
    k = np.arange(n, dtype=np.float64)
    s = 2 * k + a
    diag = np.where(s > 0, -a * a / np.where(s > 0, s * (s + 2), 1.0), 0.0)
    diag[0] = -a / (a + 2)
    k, s = k[1:], s[1:]
    off = np.sqrt(4 * k * k * (k + a) ** 2 / (s * s * (s + 1) * (s - 1)))
    t, V = np.linalg.eigh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1))
    return 0.5 * (t + 1), V[0] ** 2 / (a + 1)


def _volume_rule(dim, p):
    """Collapsed Gauss rules with p + 1 points per direction; the symmetric 14-point rule of degree
    5 (Walkington, 2000) on tetrahedra at p = 2.  Points in reference coordinates."""
    if dim == 3 and p == 2:
        pts, w = [], []
        for a, b, ww in ((0.31088591926330060980, 1, 0.018781320953002641800),
                         (0.092735250310891226402, 1, 0.012248840519393658257),
                         (0.045503704125649649492, 2, 0.0070910034628469110730)):
            bary = (a, a, a, 1 - 3 * a) if b == 1 else (a, a, 0.5 - a, 0.5 - a)
            for q in sorted(set(itertools.permutations(bary))):
                pts.append(q[1:])
                w.append(ww)
        return np.array(pts), np.array(w)
    g = [_gauss(p + 1, a) for a in range(dim)]
    pts, w = [], []
    for ix in itertools.product(range(p + 1), repeat=dim):
        t = [g[d][0][ix[d]] for d in range(dim)]
        pts.append([t[d] * math.prod(1 - t[e] for e in range(d + 1, dim)) for d in range(dim)])
        w.append(math.prod(g[d][1][ix[d]] for d in range(dim)))
    return np.array(pts), np.array(w)


def _face_rule(dim, p):
    """Barycentric face points and weights that sum to 1; Radon's 7-point rule at p = 2 in 3D."""
    if dim == 2:
        t, w = _gauss(p + 1, 0)
        return np.stack([1 - t, t], 1), w
    if p == 2:
        r = math.sqrt(15.0)
        b, w = [(1 / 3, 1 / 3, 1 / 3)], [9 / 40]
        for a, ww in (((6 - r) / 21, (155 - r) / 1200), ((6 + r) / 21, (155 + r) / 1200)):
            for q in sorted(set(itertools.permutations((a, a, 1 - 2 * a)))):
                b.append(q)
                w.append(ww)
        return np.array(b), np.array(w)
    t, w = _volume_rule(2, p)
    return np.concatenate([1 - t.sum(1, keepdims=True), t], 1), 2 * w


class Space:
    """The orthonormal element basis of the binding (graded monomials about the centroid,
    orthonormalised in order) and the volume points of a mesh, on the GPU."""

    def __init__(self, mesh, p, device="cuda"):
        self.mesh, self.p, self.dim, self.dev = mesh, p, mesh.dim, device
        d = self.dim
        self.verts = torch.tensor(mesh.coords, device=device)[torch.tensor(mesh.elems, device=device).long()]
        self.E = len(self.verts)
        A = self.verts[:, 1:] - self.verts[:, :1]
        self.det = torch.linalg.det(A) if d == 3 else A[:, 0, 0] * A[:, 1, 1] - A[:, 0, 1] * A[:, 1, 0]
        pts, w = _volume_rule(d, p)
        self.rq = torch.einsum("qk,ekd->eqd", torch.tensor(pts, device=device), A)  # offsets from vertex 0
        self.wq = torch.tensor(w, device=device) * self.det[:, None]
        self.exps = [ex for deg in range(p + 1) for ex in sorted(itertools.product(range(deg + 1), repeat=d), reverse=True)
                     if sum(ex) == deg]
        self.N, self.nv = len(self.exps), d + 2
        self.rc = A.sum(1) / (d + 1)
        self.scale = 0.5 * (self.verts.amax(1) - self.verts.amin(1))
        chi = self.monomials(self.rq, slice(None))
        C, psi = [], []
        for i in range(self.N):
            c = torch.zeros(self.E, self.N, device=device, dtype=F64)
            c[:, i] = 1.0
            v = chi[:, :, i].clone()
            for _ in range(2):  # orthogonalised twice: to rounding
                for j in range(i):
                    h = (self.wq * v * psi[j]).sum(1, keepdim=True)
                    v = v - h * psi[j]
                    c = c - h * C[j]
            s = (self.wq * v * v).sum(1, keepdim=True).sqrt()
            psi.append(v / s)
            C.append(c / s)
        self.C = torch.stack(C, 1)
        self.psi = torch.stack(psi, 2)  # [E, nq, N]

    def monomials(self, r, rows):
        X = (r - self.rc[rows][:, None]) / self.scale[rows][:, None]
        return torch.stack([math.prod([X[:, :, d] ** e for d, e in enumerate(ex) if e], start=torch.ones_like(X[:, :, 0]))
                            for ex in self.exps], 2)

    def at(self, rows, r):
        return torch.einsum("eik,eqk->eqi", self.C[rows], self.monomials(r, rows))

    def gradients(self):
        X, out = (self.rq - self.rc[:, None]) / self.scale[:, None], []
        for d in range(self.dim):
            g = []
            for ex in self.exps:
                t = torch.full_like(X[:, :, 0], float(ex[d]))
                for k, e in enumerate(ex):
                    e = e - 1 if k == d else e
                    if ex[d] and e:
                        t = t * X[:, :, k] ** e
                g.append(t / self.scale[:, None, d])
            out.append(torch.einsum("eik,eqk->eqi", self.C, torch.stack(g, 2)))
        return out

    def project(self, state):
        x = self.verts[:, :1] + self.rq
        return torch.einsum("eq,eqi,eqv->evi", self.wq, self.psi, state(x)).reshape(-1)


def _flow_state(case, mesh, seed):
    """Pointwise state: an isentropic vortex in the free stream on the square and cube meshes, the
    free stream with four small Gaussian (rho, p) pulses in the channel; centres and strengths from
    the seed."""
    rng, fs = np.random.default_rng(seed), _freestream(case["mesh"])
    a, cinf = math.radians(fs.alpha_deg), math.sqrt(GAMMA)
    u0, v0 = fs.mach * cinf * math.cos(a), fs.mach * cinf * math.sin(a)
    if case["mesh"] == "bump":
        blobs = rng.uniform([-0.5, 0.2, -1e-2, -1e-2], [1.5, 0.8, 1e-2, 1e-2], (4, 4))
    else:
        rad = 0.5 * mesh.side if case["mesh"] == "stretched" else 1.0
        eps = (2 * math.pi * 0.2 * u0 * math.exp(-0.5) if case["mesh"] == "stretched" else 5.0) * rng.uniform(0.8, 1.0)
        xc, yc = mesh.side * (0.5 + 0.05 * rng.uniform(-1, 1, 2))

    def state(x):
        rho = torch.ones_like(x[..., 0])
        pr, u, v = rho.clone(), u0 * rho, v0 * rho
        if case["mesh"] == "bump":
            for bx, by, ar, ap in blobs:
                g = torch.exp(-((x[..., 0] - bx) ** 2 + (x[..., 1] - by) ** 2) / 0.01)
                rho, pr = rho + ar * g, pr + ap * g
        else:
            dx, dy = ((x[..., k] - c) for k, c in ((0, xc), (1, yc)))
            if case["mesh"] != "boxcube":
                dx, dy = (t - mesh.side * torch.round(t / mesh.side) for t in (dx, dy))
            dx, dy = dx / rad, dy / rad
            r2 = dx * dx + dy * dy
            f = eps / (2 * math.pi) * torch.exp(0.5 * (1 - r2))
            u, v = u - f * dy, v + f * dx
            T = 1 - (GAMMA - 1) * eps ** 2 / (8 * GAMMA * math.pi ** 2) * torch.exp(1 - r2)
            rho = T ** (1 / (GAMMA - 1))
            pr = rho * T
        mom = [rho * u, rho * v] + [torch.zeros_like(rho)] * (x.shape[-1] - 2)
        return torch.stack([rho] + mom + [pr / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)], -1)
    return state


def _inputs(case, seed, space):
    """(U, v, w): a flow state, a direction (the difference of two flow states and as much noise: a
    basis vector of an outer solver has smooth and rough parts) and a cotangent of unit size."""
    mesh = space.mesh
    U = space.project(_flow_state(case, mesh, seed))
    if case["call"] in ("step", "march", "residual"):
        return U, None, None
    g = torch.Generator(device=space.dev).manual_seed(seed + 7)
    noise = lambda: torch.randn(U.shape, generator=g, device=space.dev, dtype=F64)  # noqa: E731
    v = space.project(_flow_state(case, mesh, seed + 1000)) - U
    v = v + v.norm() / math.sqrt(v.numel()) * noise()
    w = noise()
    return U, v, w / w.norm()


# ------------------------------------------------------------------------------ the calls

SCHEMES = {"pcexp": capi.PCEXP_SCHEME_PCEXP, "exp1": capi.PCEXP_SCHEME_EXP1, "etd2": capi.PCEXP_SCHEME_ETD2}


def prepare(case, seed):
    mesh = _mesh(case["mesh"], case["nx"], case["ny"])
    free = _freestream(case["mesh"])
    space = Space(mesh, case["p"])
    U, v, w = _inputs(case, seed, space)
    dt = float(local_dt(space, U, case["cfl"], free).min()) if case["call"] == "backward" else 0.0
    del space
    capi.load()
    ctx = capi.Context(mesh, case["p"], free, capi.PCEXP_FP32_MIXED if case["mixed"] else capi.PCEXP_FP64,
                       m_max=max(case["m"], 1), krylov_tol=case["tol"])
    return dict(case=case, ctx=ctx, U=U, v=v, w=w, dt=dt)


def run(state):
    c, ctx, U = state["case"], state["ctx"], state["U"]
    if c["call"] == "step":
        mode = capi.PCEXP_DT_LOCAL_CFL if c["dt"] == "local" else capi.PCEXP_DT_GLOBAL_CFL
        ctx.set_state(U)
        for _ in range(c["steps"]):
            ctx.step(SCHEMES[c["scheme"]], mode, c["cfl"], c["m"], info=False)
        out = ctx.get_state(torch.empty_like(U))
        return out.float() if c["mixed"] else out
    if c["call"] == "march":
        ctx.set_state(U)
        info = ctx.march_steady(capi.PCEXP_SCHEME_PCEXP, c["cfl"], 10.0, c["steps"], c["m"])
        return dict(info, state=ctx.get_state(torch.empty_like(U)))
    if c["call"] == "backward":
        ubar, theta = ctx.step_backward(U, state["dt"], c["m"], state["w"], with_theta=True)
        return dict(ubar=ubar, theta=theta)
    if c["call"] == "residual":
        out = ctx.residual(U)
    elif c["call"] == "jvp":
        out = ctx.jvp(U, state["v"])
    else:
        out = ctx.vjp(U, state["w"])
    return out.float() if c["mixed"] else out


def work(case):
    """Bytes: the state-shaped inputs and outputs (64 bits each) and the mesh's geometry once.
    Flops: the contractions of the DG operator (traces, tests, lifts), the flux Jacobian products,
    and two flops per entry and column of each Gram-Schmidt projection and update."""
    d, p, m = (3 if "cube" in case["mesh"] else 2), case["p"], case["m"]
    E = 6 * case["nx"] ** 3 if d == 3 else 2 * case["nx"] * case["ny"]
    nv, nb = d + 2, math.comb(p + d, d)
    nq, nfq = len(_volume_rule(d, p)[1]), len(_face_rule(d, p)[1])
    K, F, word = E * nv * nb, E * (d + 1) // 2, 4 if case["mixed"] else 8
    geo = E * (d * d + 2 * (d + 1)) * word
    op = 2 * E * (nq * (nv * nb + d * nv * nv) + nv * nb * (d * nq + (d + 1) * nfq)) + 2 * F * nfq * (2 * nv * nb + 2 * nv * nv)
    cols = m * (m + 1) // 2
    call, n = case["call"], case["steps"]
    if call in ("step", "march"):
        stages = n * (1 if case["scheme"] == "exp1" else 2) - (1 if case["scheme"] == "etd2" else 0)
        return dict(bytes=16 * K + geo, flops=stages * ((m + 1) * op + 4 * K * cols))
    if call == "backward":  # the step, its reverse Gram-Schmidt (twice the products) and J^T w, d(J v)/du per column
        return dict(bytes=24 * K + geo, flops=2 * ((3 * m + 3) * op + 16 * K * cols))
    return dict(bytes=(16 if call == "residual" else 24) * K + geo, flops=op)


# ------------------------------------------------- the scheme in plain 64-bit torch (exact)


class Operator(Space):
    """R(u), J(u) v and the time-step rule of the DG scheme on the GPU in 64 bits."""

    def __init__(self, mesh, p, free):
        super().__init__(mesh, p)
        d, NF, E, dev = self.dim, self.dim + 1, self.E, self.dev
        self.free = free
        self.gpsi = [g * self.wq[:, :, None] for g in self.gradients()]
        elems, master = torch.tensor(mesh.elems, device=dev).long(), torch.tensor(mesh.vert_master, device=dev).long()
        loc = torch.tensor([[(f + k) % NF for k in range(1, NF)] for f in range(NF)], device=dev)  # face opposite f
        fv = elems[:, loc]  # [E, NF, d]
        key = master[fv].sort(-1).values.reshape(E * NF, d)
        _, ids = torch.unique(key, dim=0, return_inverse=True)
        order = torch.argsort(ids, stable=True)
        ids = ids[order]
        first = torch.ones_like(ids, dtype=torch.bool)
        first[1:] = ids[1:] != ids[:-1]
        start = torch.nonzero(first).reshape(-1)
        count = torch.diff(torch.cat([start, torch.tensor([len(ids)], device=dev)]))
        eL, fL = order[start] // NF, order[start] % NF
        two = count == 2
        sR = order[(start + 1).clamp(max=len(order) - 1)]
        eR, fR = torch.where(two, sR // NF, eL), torch.where(two, sR % NF, fL)
        self.eL, self.eR, self.two, F = eL, eR, two, len(eL)
        iF = torch.arange(F, device=dev)[:, None]
        corner = loc[fL]  # the L element's local vertices, in its order
        cL = self.verts[eL[:, None], corner]
        mL, locR = master[elems[eL[:, None], corner]], loc[fR]
        match = (master[elems[eR[:, None], locR]][:, None, :] == mL[:, :, None]).int().argmax(-1)
        cR = self.verts[eR[:, None], locR[iF, match]]
        e1 = cL[:, 1] - cL[:, 0]
        if d == 2:
            nrm = torch.stack([e1[:, 1], -e1[:, 0]], 1)
            meas = nrm.norm(dim=1)
        else:
            nrm = torch.linalg.cross(e1, cL[:, 2] - cL[:, 0])
            nrm = nrm * torch.sign(((cL[:, 0] - self.verts[eL, fL]) * nrm).sum(1, keepdim=True))
            meas = 0.5 * nrm.norm(dim=1)
        self.n = (nrm / nrm.norm(dim=1, keepdim=True))[:, None].unbind(-1)
        bary, w = _face_rule(d, p)
        bary = torch.tensor(bary, device=dev)
        self.wf = (meas[:, None] * torch.tensor(w, device=dev))[:, :, None]
        pts = lambda e, c: (c[:, :1] - self.verts[e, :1]) + torch.einsum("qk,fkd->fqd", bary[:, 1:], c[:, 1:] - c[:, :1])  # noqa: E731
        self.bL, self.bR = self.at(eL, pts(eL, cL)), self.at(eR, pts(eR, cR))
        area = torch.zeros(E, NF, device=dev, dtype=F64)
        area[eL, fL] = meas
        area[eR, fR] = torch.where(two, meas, area[eR, fR])
        self.slot = torch.zeros(E, NF, device=dev, dtype=torch.long)  # face of every element side
        self.slot[eL, fL] = torch.arange(F, device=dev)
        self.slot[eR, fR] = torch.arange(F, device=dev)
        self.lift = torch.zeros(E, NF, len(w), self.N, device=dev, dtype=F64)
        self.lift[eL, fL] = -self.bL
        self.lift[eR[two], fR[two]] = self.bR[two]
        tag = torch.zeros(F, dtype=torch.long, device=dev)
        if len(mesh.btags):
            bkey = torch.tensor(mesh.bfaces, device=dev).long().sort(-1).values
            nvert = len(mesh.coords)
            code = lambda k: sum(k[:, i] * nvert ** i for i in range(d))  # noqa: E731
            bcode, perm = code(bkey).sort()
            at = torch.searchsorted(bcode, code(fv[eL, fL].sort(-1).values)).clamp(max=len(bcode) - 1)
            tag = torch.where(two, tag, torch.tensor(mesh.btags, device=dev).long()[perm][at])
        self.wall, self.open = (tag == capi.PCEXP_BC_SLIP_WALL)[:, None, None], (tag == capi.PCEXP_BC_FARFIELD)[:, None, None]
        self.any_wall, self.any_open = bool(self.wall.any()), bool(self.open.any())
        self.volume = self.wq.sum()
        self.theta = torch.tensor([free.mach, free.alpha_deg], device=dev, dtype=F64)

    def normal_flux(self, U, n):
        rho, v, pr, H = _primitives(U)
        q = sum(a * b for a, b in zip(v, n))
        return [rho * q] + [rho * a * q + pr * b for a, b in zip(v, n)] + [rho * H * q]

    def residual(self, u, theta=None):
        d, u = self.dim, u.reshape(self.E, self.nv, self.N)
        U = torch.einsum("eqi,evi->eqv", self.psi, u).unbind(-1)
        R = 0
        rho, v, pr, H = _primitives(U)
        for k in range(d):
            F = [rho * v[k]] + [rho * v[j] * v[k] + (pr if j == k else 0) for j in range(d)] + [rho * H * v[k]]
            R = R + torch.einsum("eqi,eqv->evi", self.gpsi[k], torch.stack(F, -1))
        UL = torch.einsum("fqi,fvi->fqv", self.bL, u[self.eL])
        UR = torch.einsum("fqi,fvi->fqv", self.bR, u[self.eR])
        if self.any_wall:
            m = sum(UL[..., 1 + k] * self.n[k] for k in range(d))
            G = torch.stack([UL[..., 0]] + [UL[..., 1 + k] - 2 * m * self.n[k] for k in range(d)] + [UL[..., -1]], -1)
            UR = torch.where(self.wall, G, UR)
        if self.any_open:
            UR = torch.where(self.open, self.far(UL, self.theta if theta is None else theta), UR)
        G = torch.stack(self.roe(UL.unbind(-1), UR.unbind(-1)), -1) * self.wf
        return (R + torch.einsum("ekqi,ekqv->evi", self.lift, G[self.slot])).reshape(-1)

    def far(self, UL, theta):
        g, g1, n, d = GAMMA, GAMMA - 1, self.n, self.dim
        rho, v, pr, _ = _primitives(UL.unbind(-1))
        a, ci = theta[1] * (math.pi / 180), math.sqrt(GAMMA)
        vi = [theta[0] * ci * torch.cos(a), theta[0] * ci * torch.sin(a)] + [torch.zeros_like(a)] * (d - 2)
        c, q = torch.sqrt(g * pr / rho), sum(x * y for x, y in zip(v, n))
        qi = sum(x * y for x, y in zip(vi, n))
        rp = torch.where(q > -c, q + 2 * c / g1, qi + 2 * ci / g1)
        rm = torch.where(q < c, qi - 2 * ci / g1, q - 2 * c / g1)
        qb, cb = 0.5 * (rp + rm), 0.25 * g1 * (rp - rm)
        out = qb >= 0
        s = torch.where(out, pr / rho ** g, torch.ones_like(pr))
        vb = [torch.where(out, v[k] - q * n[k], vi[k] - qi * n[k] + 0 * q) + qb * n[k] for k in range(d)]
        rb = (cb * cb / (g * s)) ** (1 / g1)
        return torch.stack([rb] + [rb * x for x in vb] + [rb * cb * cb / (g * g1) + 0.5 * rb * sum(x * x for x in vb)], -1)

    def roe(self, L, R):
        n, d = self.n, self.dim
        rL, vL, pL, HL = _primitives(L)
        rR, vR, pR, HR = _primitives(R)
        sL, sR = rL.sqrt(), rR.sqrt()
        mean = lambda a, b: (sL * a + sR * b) / (sL + sR)  # noqa: E731
        v, H, rh = [mean(a, b) for a, b in zip(vL, vR)], mean(HL, HR), sL * sR
        q2 = sum(x * x for x in v)
        cc = (GAMMA - 1) * (H - 0.5 * q2)
        c, q = cc.sqrt(), sum(x * y for x, y in zip(v, n))
        dv = [b - a for a, b in zip(vL, vR)]
        dq, dp = sum(x * y for x, y in zip(dv, n)), pR - pL
        a1, a4 = (q - c).abs() * (dp - rh * c * dq) / (2 * cc), (q + c).abs() * (dp + rh * c * dq) / (2 * cc)
        a2, sh = q.abs() * ((rR - rL) - dp / cc), q.abs() * rh
        D = [a1 + a2 + a4]
        D += [a1 * (v[k] - c * n[k]) + a2 * v[k] + sh * (dv[k] - dq * n[k]) + a4 * (v[k] + c * n[k]) for k in range(d)]
        D += [a1 * (H - c * q) + a2 * 0.5 * q2 + sh * (sum(x * y for x, y in zip(v, dv)) - q * dq) + a4 * (H + c * q)]
        return [0.5 * (a + b - x) for a, b, x in zip(self.normal_flux(L, n), self.normal_flux(R, n), D)]

    def jvp(self, u, v, theta=None):
        return torch.func.jvp(lambda x: self.residual(x, theta), (u,), (v,))[1]


def _primitives(U):
    rho, E = U[0], U[-1]
    v = [m / rho for m in U[1:-1]]
    pr = (GAMMA - 1) * (E - 0.5 * rho * sum(x * x for x in v))
    return rho, v, pr, (E + pr) / rho


def local_dt(space, U, cfl, free):
    """CFL h / ((2p + 1)(|v| + c)) per element, h = 2 d |E| / |dE|, the state at the centroid."""
    d = space.dim
    rows = torch.arange(space.E, device=space.dev)
    u = torch.einsum("eqi,evi->eqv", space.at(rows, space.rc[:, None]), U.reshape(space.E, space.nv, space.N))[:, 0]
    rho, v, pr, _ = _primitives(u.unbind(-1))
    around = 0
    for f in range(d + 1):
        c = space.verts[:, [k for k in range(d + 1) if k != f]]
        e = c[:, 1:] - c[:, :1]
        around = around + (e[:, 0].norm(dim=1) if d == 2 else 0.5 * torch.linalg.cross(e[:, 0], e[:, 1]).norm(dim=1))
    h = 2 * d * space.det / (2.0 if d == 2 else 6.0) / around
    return cfl * h / ((2 * space.p + 1) * (sum(x * x for x in v).sqrt() + (GAMMA * pr / rho).sqrt()))


def _phi(H, k, dt):
    A = torch.nn.functional.pad(dt * H[:k, :k], (0, 2, 0, 2))
    B = torch.zeros_like(A)
    B[0, k] = B[k, k + 1] = 1.0
    X = torch.linalg.matrix_exp(A + B)
    return X[:k, k], X[:k, k + 1]


def _arnoldi(matvec, b, m, dt=None, tol=0.0):
    beta = b.norm()
    V, cols = [b / beta], []
    for j in range(m):
        w, Q = matvec(V[-1]), torch.stack(V)
        h = Q @ w
        w = w - h @ Q
        h2 = Q @ w
        w = w - h2 @ Q
        s = w.norm()
        cols.append(torch.nn.functional.pad(torch.cat([h + h2, s[None]]), (0, m - 1 - j)))
        V.append(w / s)
        if tol > 0 and (j + 1) % 5 == 0 and j + 1 < m:
            H, k = torch.stack(cols, 1), j + 1
            y1, y2 = _phi(H, k, dt)
            if float(dt * s * y2[k - 1].abs() / y1.norm()) <= tol:
                break
    return V, torch.stack(cols, 1), beta


def _phi_product(matvec, b, dt, case, which=0):
    V, H, beta = _arnoldi(matvec, b, case["m"], dt, case["tol"])
    k = H.shape[1]
    return dt * beta * (_phi(H, k, dt)[which] @ torch.stack(V[:k]))


def _step(op, u, dt, case, scale=1.0, theta=None):
    """One PCEXP or EXP1 step of du/dt = scale R(u) with the given dt."""
    J = lambda v: scale * op.jvp(u, v, theta)  # noqa: E731
    R = scale * op.residual(u, theta)
    delta = _phi_product(J, R, dt, case)
    if case["scheme"] == "exp1":
        return u + delta
    d = scale * op.residual(u + delta, theta) - R - J(delta)
    return u + delta + 0.5 * _phi_product(J, d, dt, case)


def _etd2(op, u, case, free):
    """Two ETD2 steps, the first without history."""
    dt = float(local_dt(op, u, case["cfl"], free).min())
    R0 = op.residual(u)
    u1 = u + _phi_product(lambda v: op.jvp(u, v), R0, dt, case)
    dt1 = float(local_dt(op, u1, case["cfl"], free).min())
    R1, J = op.residual(u1), lambda v: op.jvp(u1, v)
    return u1 + _phi_product(J, R1, dt1, case) + dt1 / dt * _phi_product(J, R1 - R0 - J(u1 - u), dt1, case, 1)


def exact(case, seed):
    c = case
    mesh, free = _mesh(c["mesh"], c["nx"], c["ny"]), _freestream(c["mesh"])
    op = Operator(mesh, c["p"], free)
    U, v, w = _inputs(c, seed, op)
    if c["call"] == "residual":
        return op.residual(U)
    if c["call"] == "jvp":
        return op.jvp(U, v)
    if c["call"] == "vjp":
        return torch.func.vjp(op.residual, U)[1](w)[0]
    if c["call"] == "backward":
        dt = float(local_dt(op, U, c["cfl"], free).min())
        ubar, theta = torch.func.vjp(lambda u, t: _step(op, u, dt, c, 1.0, t), U, op.theta)[1](w)
        return dict(ubar=ubar, theta=theta.cpu().numpy())
    if c["call"] == "march":
        u, hist = U, []
        for n in range(1, c["steps"] + 2):
            hist.append(float(op.residual(u).reshape(op.E, op.nv, -1)[:, 0].norm() / op.volume))
            if n <= c["steps"]:
                cfl = min(c["cfl"], max(hist[-1] ** -3, 1 + (n - 1) / (2 * c["p"] + 1)))
                dte = local_dt(op, u, cfl, free)
                u = _step(op, u, 1.0, c, dte.repeat_interleave(op.nv * op.N))
        return dict(iterations=None, res_first=hist[0], res_last=hist[-1], converged=None, state=u)
    if c["scheme"] == "etd2":
        return _etd2(op, U, c, free)
    u = U
    for _ in range(c["steps"]):
        dte = local_dt(op, u, c["cfl"], free)
        local = c["dt"] == "local"
        u = _step(op, u, 1.0 if local else float(dte.min()), c, dte.repeat_interleave(op.nv * op.N) if local else 1.0)
    return u
