"""The work that users of libmtf have it do, as cases that can be prepared, run and checked.

A user holds a skeleton mesh, assembles the operator, solves for plane waves and evaluates fields; codes that bring
their own Krylov solver call the operator and preconditioner applies.  Every case names one such call (``op``), a mesh
family with its size, the precision of the system and the number of right-hand sides (``nrhs``); materials, wavenumber,
waves and vectors come from the seed.  ``listed()`` holds the sizes of this repository's own configurations and
``draw()`` spreads over their ranges, odd block sizes (latitude-longitude spheres) and uneven subdomains (cut spheres)
among them.  Mixed-precision systems state 1e-5 on currents and fields and store their blocks in FP32: a program that
keeps their results keeps them in complex64, and so do these cases.  ``exact()`` restates the Galerkin integrals, the
exchange, block-OSRC and the fields in plain FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import mtf_inputs as mi
from paper_2502_10907_gb300.api import Mesh, System, solve_batch

OBS = np.stack([np.cos(np.linspace(0.0, 2.0 * np.pi, 181)), np.sin(np.linspace(0.0, 2.0 * np.pi, 181)), np.zeros(181)], 1)

# the options a mixed-precision program sets (README): block-OSRC with Pade order 16 and a restart length that holds
# the whole cycle
MIXED = dict(precision=1, precond=1, osrc_np=16, restart=600, max_iter=4000)
PLAIN = dict(restart=1500, max_iter=3000)


def listed():
    return [
        # the first thing a user runs: one dielectric sphere, plain MTF in FP64 (GMRES without preconditioner or
        # restart at the default tolerance), from host arrays to the far field; the smallest whole call
        dict(name="oneshot_sphere_fp64", op="oneshot", mesh="sphere", size=2, precision=0, nrhs=1),
        # one more wavenumber of a sweep in FP64, blocks read back
        dict(name="assemble_split_fp64", op="assemble", mesh="split", size=7, precision=0, nrhs=1),
        # the same on the mixed path with block-OSRC, for three large blocks
        dict(name="assemble_split_mixed", op="assemble", mesh="split", size=11, precision=1, nrhs=1),
        # and for one large and eight smaller blocks (the 2 x 2 x 2 cube)
        dict(name="assemble_cube2_mixed", op="assemble", mesh="cube2", size=9, precision=1, nrhs=1),
        # FP64 operator apply of a caller's own solver or residual check, two polarisations
        dict(name="matvec_split_fp64", op="matvec", mesh="split", size=11, precision=0, nrhs=2),
        # FP32 operator apply of few right-hand sides: the small, latency-sensitive call
        dict(name="matvec_split_f32", op="matvec_f32", mesh="split", size=11, precision=1, nrhs=2),
        # FP32 operator apply of many right-hand sides on the 4 x 4 x 4 cube
        dict(name="matvec_cube4_f32", op="matvec_f32", mesh="cube4", size=5, precision=1, nrhs=16),
        # block-OSRC apply on the same operator
        dict(name="precond_cube4_f32", op="precond_f32", mesh="cube4", size=5, precision=1, nrhs=16),
        # mixed solve of two polarisations on an assembled system: one Krylov space per right-hand side
        dict(name="solve_split_mixed", op="solve", mesh="split", size=11, precision=1, nrhs=2),
        # one step of a parameter sweep, the largest whole call: reassembly, 16 waves in one block Krylov space, far field
        dict(name="sweep_cube4_mixed", op="sweep", mesh="cube4", size=5, precision=1, nrhs=16),
        # uneven small scatterers solved together (size = their number)
        dict(name="batch_cut_spheres", op="batch", mesh="cut", size=6, precision=1, nrhs=8),
        # post-processing of 16 solutions: far-field cut and a near-field map
        dict(name="fields_cube2", op="fields", mesh="cube2", size=9, precision=1, nrhs=16),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    op = rng.choice(["oneshot", "assemble", "assemble", "matvec", "matvec_f32", "matvec_f32", "precond_f32", "solve",
                     "sweep", "batch", "fields", "fields"])
    if op == "batch":
        return dict(op=op, mesh="cut", size=rng.randint(2, 6), precision=1, nrhs=rng.choice([4, 6, 8]))
    if op == "oneshot":
        return dict(op=op, mesh="uv", size=log_int(5, 10), precision=0, nrhs=rng.randint(1, 2))
    # (a program reads back the blocks of few subdomains; few waves converge one by one where few subdomains couple,
    # many waves share a block space elsewhere)
    mesh = rng.choice({"assemble": ["uv", "split", "cube2"], "solve": ["uv", "split"]}.get(op, ["uv", "split", "cube2", "cube4"]))
    precision = 0 if op == "matvec" else rng.randint(0, 1) if op in ("assemble", "fields") else 1
    large = {"uv": 31, "split": 11, "cube2": 9, "cube4": 5}[mesh]
    small = {"uv": 6, "split": 3, "cube2": 2, "cube4": 1}[mesh]
    if precision == 0:  # FP64 blocks take twice the memory and the narrow pipe
        large = {"uv": 24, "split": 11, "cube2": 6, "cube4": 3}[mesh]
    if op in ("solve", "sweep") and mesh == "uv":  # its pole triangles get thin with the size
        large = 15
    if op == "solve":
        nrhs = rng.randint(1, 3)
    elif op == "sweep":
        nrhs = rng.randint(12 if mesh == "cube4" else 4, 16)
    elif op == "assemble":
        nrhs = 1
    else:
        nrhs = log_int(1, 32)
    return dict(op=op, mesh=mesh, size=log_int(small, large), precision=precision, nrhs=nrhs)


# ---------------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------------
def _meshes(case):
    size = case["size"]
    kind = case["mesh"]
    if kind == "sphere":
        return [mi.icosphere(size)]
    if kind == "uv":  # 2 + (size - 1)(2 size + 1) vertices: odd and even block sizes
        return [mi.uv_sphere(size, 2 * size + 1)]
    if kind == "split":
        return [mi.split_sphere(size)]
    if kind == "cube2":
        return [mi.cube_partition((2, 2, 2), size)]
    if kind == "cube4":
        return [mi.cube_partition((4, 4, 4), size)]
    # cut spheres: 2..7 slabs, 500..1300 triangles, as uneven as a batch's scatterers are
    out = []
    for q in range(size):
        ncut = 1 + (5 * q + 2) % 6
        cuts = np.linspace(-0.7, 0.7, ncut) if ncut > 1 else np.array([0.1])
        area = 4 * np.pi + np.pi * np.sum(1 - cuts ** 2)
        out.append(mi.cut_sphere(cuts, float(np.sqrt(2.3 * area / (500 + 160 * (q % 6))))))
    return out


def _problem(case, mesh, rng):
    """k0, eps_r, mu_r, directions and polarisations of one scatterer: the repository's configurations, varied from
    seed to seed (little for the split sphere, whose interior resonances are sharp at its size; the cut spheres stay below theirs)."""
    kind = case["mesh"]
    k0 = {"sphere": 1.0, "uv": 1.0, "split": 2.0, "cube2": 3.0, "cube4": 4.0, "cut": 1.2}[kind]
    if kind == "split":
        k0 *= rng.uniform(0.99, 1.01)
        eps = np.array([1.0, 2.0, 4.0]) * np.array([1.0, *rng.uniform(0.98, 1.02, 2)])
    else:
        k0 *= rng.uniform(0.9, 1.1)
        eps = np.concatenate([[1.0], rng.uniform(1.5, {"cube2": 4.0, "cube4": 4.0, "cut": 2.0}.get(kind, 2.5), mesh.n_domains - 1)])
    d = rng.normal(size=(case["nrhs"], 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    p = np.cross(rng.normal(size=d.shape), d)
    p /= np.linalg.norm(p, axis=1, keepdims=True)
    return dict(k0=float(k0), eps_r=eps, mu_r=np.ones(mesh.n_domains), dirs=d, pols=p.astype(np.complex128))


def _problems(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    meshes = _meshes(case)
    return meshes, [_problem(case, m, rng) for m in meshes], rng


def _vectors(seed, nrhs, n, dtype):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((nrhs, n), generator=g, dtype=torch.complex128, device="cuda").to(dtype)


def _points(case, mesh, rng):
    """Near-field map: a plane above the scatterer (exterior) and, in the partitioned cubes, points around the centres
    of the sub-boxes (their own subdomains)."""
    hi = mesh.vertices.max(axis=0)
    g = np.linspace(-1.0, 1.0, 24)
    X, Y = np.meshgrid(g, g)
    pts = np.stack([X.ravel(), Y.ravel(), np.full(X.size, hi[2] + 0.4)], 1) + rng.uniform(-0.02, 0.02, 3)
    dom = np.zeros(len(pts), dtype=np.int32)
    P = {"cube2": 2, "cube4": 4}.get(case["mesh"])
    if P:
        c = np.array([(ix, iy, iz) for iz in range(P) for iy in range(P) for ix in range(P)])
        inner = (c + 0.5) / P + rng.uniform(-0.1, 0.1, c.shape) / P
        pts = np.concatenate([pts, inner])
        dom = np.concatenate([dom, 1 + np.arange(P ** 3, dtype=np.int32)])
    return pts, dom


def _system(case, mesh, p):
    op = case["op"]
    if case["precision"] == 0:
        opts = {}
    elif op in ("matvec_f32", "fields"):
        opts = dict(precision=1)
    elif op == "sweep":
        opts = dict(MIXED, tol=1e-7)
    elif op == "batch":
        opts = dict(MIXED, tol=1e-7, residual_fp64=1)
    else:
        opts = dict(MIXED, tol=1e-8)
    return System(Mesh.from_inputs(mesh), p["k0"], p["eps_r"], p["mu_r"], **opts)


def prepare(case, seed):
    meshes, probs, rng = _problems(case, seed)
    st = dict(case=case, op=case["op"], meshes=meshes, probs=probs)
    if case["op"] == "oneshot":
        return st
    st["systems"] = [_system(case, m, p) for m, p in zip(meshes, probs)]
    if case["op"] in ("assemble", "sweep"):  # the step's own wavenumber and materials
        st["next"] = _problem(case, meshes[0], rng)
    n = st["systems"][0].mesh.n_total
    if case["op"] in ("matvec", "fields"):
        st["x"] = _vectors(seed, case["nrhs"], n, torch.complex128)
    if case["op"] in ("matvec_f32", "precond_f32"):
        st["x"] = _vectors(seed, case["nrhs"], n, torch.complex64)
    if case["op"] == "fields":
        st["points"], st["domains"] = _points(case, meshes[0], rng)
    return st


# ---------------------------------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------------------------------
def run(st):
    op = st["op"]
    if op == "oneshot":
        m, p = st["meshes"][0], st["probs"][0]
        s = System(Mesh.from_inputs(m), p["k0"], p["eps_r"], p["mu_r"], **PLAIN)
        x, _ = s.solve(p["dirs"], p["pols"])
        return x, s.farfield(x, OBS)
    if op == "batch":
        xs, _ = solve_batch(st["systems"], [p["dirs"] for p in st["probs"]], [p["pols"] for p in st["probs"]])
        return [x.to(torch.complex64) for x in xs]
    s = st["systems"][0]
    if op == "assemble":
        q = st["next"]
        s.reassemble(q["k0"], q["eps_r"], q["mu_r"])
        out = []
        for i in range(s.mesh.n_domains):
            T, K = s.block(i)
            out += [T, K] if st["case"]["precision"] == 0 else [T.to(torch.complex64), K.to(torch.complex64)]
        return out
    if op == "matvec":
        return s.matvec(st["x"])
    if op == "matvec_f32":
        return s.matvec_f32(st["x"])
    if op == "precond_f32":
        return s.precond_f32(st["x"])
    if op == "solve":
        p = st["probs"][0]
        return s.solve(p["dirs"], p["pols"])[0].to(torch.complex64)
    if op == "sweep":
        q = st["next"]
        s.reassemble(q["k0"], q["eps_r"], q["mu_r"])
        x, _ = s.solve(q["dirs"], q["pols"])
        return x.to(torch.complex64), s.farfield(x, OBS).to(torch.complex64)
    return s.farfield(st["x"], OBS), s.nearfield(st["x"], st["points"], st["domains"])


# ---------------------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    """Stored operator entries {T, K} read or written once (32 B in FP64, 16 B in FP32), vectors and results once; the
    two Calderon products of an entry are 16 flops per right-hand side, a kernel evaluation of the quadrature 57."""
    nbytes = flops = 0.0
    ent_b = 32.0 if case["precision"] == 0 else 16.0
    vec_b = 16.0 if case["op"] not in ("matvec_f32", "precond_f32") else 8.0
    for m in _meshes(case):
        mesh = Mesh.from_inputs(m)
        N = mesh.n_dofs.astype(np.float64)
        ent, n, nrhs = float(np.sum(N ** 2)), float(mesh.n_total), case["nrhs"]
        pc = mesh.pair_counts().astype(np.float64)
        quad = 57.0 * float(0.5 * 36 * pc[3] + 1536 * pc[0] + 640 * pc[1] + 256 * pc[2])
        op = case["op"]
        if op in ("assemble", "oneshot", "sweep"):
            nbytes += ent * ent_b
            flops += quad
        if op in ("oneshot", "sweep", "solve", "batch"):  # at least one apply and the solutions
            nbytes += ent * ent_b + n * nrhs * vec_b
            flops += 16 * ent * nrhs
        if op in ("matvec", "matvec_f32"):
            nbytes += ent * ent_b + 2 * n * nrhs * vec_b
            flops += 16 * ent * nrhs
        if op == "precond_f32":
            nbytes += ent * 4 + 2 * n * nrhs * vec_b
            flops += 16 * ent * nrhs
        if op == "fields":
            pts = len(OBS) + 576 + {"cube2": 8, "cube4": 64}.get(case["mesh"], 0)
            nbytes += n * nrhs * vec_b + pts * nrhs * 48
            flops += (len(OBS) + 576) * 2 * N[0] * (40 + 16 * nrhs)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------------------------------------
# the same results in plain FP64 torch
# ---------------------------------------------------------------------------------------------------------------------
def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (x + 1) / 2, w / 2


def _triangle_rule():
    """Degree-4 symmetric 6-point rule: orbits (a, a, 1 - 2a) from its moment equations (closed form)."""
    r = math.sqrt(38 - 44 * math.sqrt(0.4))
    a = [(8 - math.sqrt(10) + r) / 18, (8 - math.sqrt(10) - r) / 18]
    q = math.sqrt(213125 - 53320 * math.sqrt(10))
    w = [(620 + q) / 3720, (620 - q) / 3720]
    st = [(s, t, 0.5 * wc) for c, wc in zip(a, w) for s, t in ((c, c), (1 - 2 * c, c), (c, 1 - 2 * c))]
    return np.array(st).T


def _sauter_schwab(kind, n=4):
    """Points in K x K (K = {0 <= x2 <= x1 <= 1}) and weights: Sauter & Schwab 2011, Sec. 5.2."""
    g, gw = _gauss(n)
    xi, e1, e2, e3 = (v.ravel() for v in np.meshgrid(g, g, g, g, indexing="ij"))
    W = np.einsum("a,b,c,d->abcd", gw, gw, gw, gw).ravel()
    if kind == 0:
        A = (xi, xi * (1 - e1 + e1 * e2)), (xi * (1 - e1 * e2 * e3), xi * (1 - e1))
        B = (xi, xi * e1 * (1 - e2 + e2 * e3)), (xi * (1 - e1 * e2), xi * e1 * (1 - e2))
        C = (xi * (1 - e1 * e2 * e3), xi * e1 * (1 - e2 * e3)), (xi, xi * e1 * (1 - e2))
        regs, jac = [A, A[::-1], B, B[::-1], C, C[::-1]], [xi ** 3 * e1 ** 2 * e2] * 6
    elif kind == 1:
        regs = [((xi, xi * e1 * e3), (xi * (1 - e1 * e2), xi * e1 * (1 - e2))),
                ((xi, xi * e1), (xi * (1 - e1 * e2 * e3), xi * e1 * e2 * (1 - e3))),
                ((xi * (1 - e1 * e2), xi * e1 * (1 - e2)), (xi, xi * e1 * e2 * e3)),
                ((xi * (1 - e1 * e2 * e3), xi * e1 * e2 * (1 - e3)), (xi, xi * e1)),
                ((xi * (1 - e1 * e2 * e3), xi * e1 * (1 - e2 * e3)), (xi, xi * e1 * e2))]
        jac = [xi ** 3 * e1 ** 2] + [xi ** 3 * e1 ** 2 * e2] * 4
    else:
        V = (xi, xi * e1), (xi * e2, xi * e2 * e3)
        regs, jac = [V, V[::-1]], [xi ** 3 * e2] * 2
    X = np.concatenate([np.stack(r[0], 1) for r in regs])
    Y = np.concatenate([np.stack(r[1], 1) for r in regs])
    return _cuda(X), _cuda(Y), _cuda(np.concatenate([W * j for j in jac]))


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


class _Exact:
    """Spaces of a skeleton mesh (one RWG function per edge of each closed Gamma_i) and the operators on them."""

    def __init__(self, mesh):
        V, F, L = mesh.vertices, np.array(mesh.triangles, dtype=np.int64), np.array(mesh.labels, dtype=np.int64)
        flip = L[:, 0] > L[:, 1]
        F[flip], L[flip] = F[flip][:, [0, 2, 1]], L[flip][:, ::-1]
        self.V, self.nd = V, mesh.n_domains
        self.F, self.v, self.dof, self.c, self.area, self.n, self.N, self.edges, self.tri = [], [], [], [], [], [], [], [], []
        for i in range(self.nd):
            t = np.concatenate([np.where((L == (min(i, j), max(i, j))).all(1))[0] for j in range(self.nd) if j != i])
            sw = np.where(L[t, 0] == i, 1.0, -1.0)
            f = F[t]
            ends = np.stack([f[:, [1, 2]], f[:, [2, 0]], f[:, [0, 1]]], 1)
            lo, hi = ends.min(2), ends.max(2)
            key, inv = np.unique((lo * len(V) + hi).ravel(), return_inverse=True)
            cr = np.cross(V[f[:, 1]] - V[f[:, 0]], V[f[:, 2]] - V[f[:, 0]])
            A = 0.5 * np.linalg.norm(cr, axis=1)
            ln = np.linalg.norm(V[hi] - V[lo], axis=2)
            c = np.where(ends[..., 0] < ends[..., 1], 1.0, -1.0) * sw[:, None] * ln / (2 * A[:, None])
            self.F.append(_cuda(f)), self.v.append(_cuda(V[f])), self.dof.append(_cuda(inv.reshape(-1, 3)))
            self.c.append(_cuda(c)), self.area.append(_cuda(A)), self.n.append(_cuda(sw[:, None] * cr / (2 * A[:, None])))
            self.N.append(len(key)), self.edges.append(np.stack([key // len(V), key % len(V)], 1)), self.tri.append(t)
        self.off = np.concatenate([[0], np.cumsum(2 * np.array(self.N))])
        s, t, w = _triangle_rule()
        lam = _cuda(np.stack([1 - s - t, s, t], 1))
        self.X = [torch.einsum("qa,tac->tqc", lam, v) for v in self.v]  # points, weights, RWG values of the 6-point rule
        self.W = [2 * a[:, None] * _cuda(w)[None] for a in self.area]
        self.f = [c[:, :, None, None] * (X[:, None] - v[:, :, None]) for c, X, v in zip(self.c, self.X, self.v)]

    def _add(self, M, rows, cols, loc):
        M.view(-1).index_add_(0, (rows[:, :, None] * M.shape[1] + cols[:, None, :]).reshape(-1), loc.reshape(-1))

    def blocks(self, i, k):
        """T_i, K_i (test rows, trial columns), in batches of triangle pairs."""
        N, T, F, v, c, dof = self.N[i], len(self.c[i]), self.F[i], self.v[i], self.c[i], self.dof[i]
        Tm, Km = (torch.zeros((N, N), dtype=torch.complex128, device="cuda") for _ in range(2))

        def kernel(R):
            r = torch.linalg.vector_norm(R, dim=-1)
            G = torch.exp(1j * k * r) / (4 * math.pi * r)
            return G, G * (1j * k - 1 / r) / r

        ids = torch.arange(T, device="cuda")
        f, fx = self.f[i], torch.cross(self.f[i], self.X[i][:, None].expand_as(self.f[i]), dim=-1)
        shared = sum((F[:, a, None] == F[None, :, b]).to(torch.uint8) for a in range(3) for b in range(3))
        a_all, b_all = torch.nonzero((shared == 0) & (ids[:, None] < ids[None, :]), as_tuple=True)
        for s in range(0, len(a_all), 1 << 18):
            a, b = a_all[s:s + (1 << 18)], b_all[s:s + (1 << 18)]
            G, g = kernel(self.X[i][a][:, :, None] - self.X[i][b][:, None])
            w = self.W[i][a][:, :, None] * self.W[i][b][:, None]

            def form(K, u, h, a=a, b=b):
                Ku = torch.einsum("npq,nbqc->nbpc", K, h.to(K.dtype)).reshape(len(a), 3, 18)
                return torch.matmul(u.to(K.dtype).reshape(len(a), 3, 18), Ku.transpose(1, 2))

            G, g = w * G, w * g
            Tl = -1j * k * form(G, f[a], f[b]) + (1j / k) * 4 * c[a][:, :, None] * c[b][:, None, :] * G.sum((1, 2))[:, None, None]
            Kl = -(form(g, fx[a], f[b]) + form(g, f[a], fx[b]))  # grad G . (g x f) = g_scalar ((f x x) . g + f . (g x y))
            self._add(Tm, dof[a], dof[b], Tl), self._add(Tm, dof[b], dof[a], Tl.transpose(1, 2))
            self._add(Km, dof[a], dof[b], Kl), self._add(Km, dof[b], dof[a], Kl.transpose(1, 2))
        for kind in range(3):  # coincident, common edge (test edge A -> B), common vertex
            xh, yh, w = _sauter_schwab(kind)
            a_all, b_all = torch.nonzero((shared == 3 - kind) & (ids[:, None] <= ids[None, :]), as_tuple=True)
            for s in range(0, len(a_all), 4096):
                a, b = a_all[s:s + 4096], b_all[s:s + 4096]
                hit = (F[a][:, :, None] == F[b][:, None, :])
                ina, inb = hit.any(2), hit.any(1)
                roll = torch.arange(3, device="cuda")[None]
                if kind == 0:
                    oa = ob = roll.expand(len(a), 3)
                elif kind == 1:
                    first = (ina & ina.roll(-1, 1)).to(torch.uint8).argmax(1)
                    oa = (first[:, None] + roll) % 3
                    at = hit.to(torch.uint8).argmax(2).gather(1, oa[:, :2])
                    ob = torch.cat([at, (~inb).to(torch.uint8).argmax(1)[:, None]], 1)
                else:
                    oa = (ina.to(torch.uint8).argmax(1)[:, None] + roll) % 3
                    ob = (inb.to(torch.uint8).argmax(1)[:, None] + roll) % 3
                Pa = v[a].gather(1, oa[:, :, None].expand(-1, 3, 3))
                Pb = v[b].gather(1, ob[:, :, None].expand(-1, 3, 3))
                o = Pa[:, :1]

                def points(P, z, o=o):
                    return (P[:, :1] - o) + z[None, :, :1] * (P[:, 1:2] - P[:, :1]) + z[None, :, 1:] * (P[:, 2:] - P[:, 1:2])

                X, Y = points(Pa, xh), points(Pb, yh)
                R = points(Pa, xh - yh) if kind == 0 else X - Y
                G, g = kernel(R)
                ww = 4 * (self.area[i][a] * self.area[i][b])[:, None] * w[None]
                u = c[a][:, :, None, None] * (X[:, None] - (v[a] - o)[:, :, None])
                h = c[b][:, :, None, None] * (Y[:, None] - (v[b] - o)[:, :, None])

                def form(K, p, q, a=a):
                    Q = p.shape[2] * 3
                    Kp = (p * K[:, None, :, None]).reshape(len(a), 3, Q)
                    return torch.matmul(Kp, q.to(K.dtype).reshape(len(a), 3, Q).transpose(1, 2))

                G, g = ww * G, ww * g
                cross = torch.cross(R[:, None].expand_as(h), h, dim=-1)  # (x - y) x g_b
                Tl = -1j * k * form(G, u, h) + (1j / k) * 4 * c[a][:, :, None] * c[b][:, None, :] * G.sum(1)[:, None, None]
                Kl = -form(g, u, cross)
                self._add(Tm, dof[a], dof[b], Tl), self._add(Km, dof[a], dof[b], Kl)
                if kind:
                    self._add(Tm, dof[b], dof[a], Tl.transpose(1, 2)), self._add(Km, dof[b], dof[a], Kl.transpose(1, 2))
        return Tm, Km

    def exchange(self):
        """(rows, columns, values) of the transmission Grams between D slots; N slots are shifted by N_i and N_j."""
        where = [dict(zip(t.tolist(), range(len(t)))) for t in self.tri]
        R, C, Z, SR, SC = [], [], [], [], []
        for i in range(self.nd):
            for j in range(self.nd):
                both = [t for t in self.tri[i].tolist() if i != j and t in where[j]]
                if not both:
                    continue
                li, lj = (torch.tensor([where[q][t] for t in both], device="cuda") for q in (i, j))
                nxf = torch.cross(self.n[i][li][:, None, None].expand_as(self.f[i][li]), self.f[i][li], dim=-1)
                loc = torch.einsum("tq,tbqc,taqc->tab", self.W[i][li], self.f[j][lj], nxf)
                rows = (self.off[i] + self.dof[i][li])[:, :, None].expand_as(loc)
                cols = (self.off[j] + self.dof[j][lj])[:, None, :].expand_as(loc)
                R.append(rows.reshape(-1)), C.append(cols.reshape(-1)), Z.append(loc.reshape(-1))
                SR.append(torch.full_like(R[-1], self.N[i])), SC.append(torch.full_like(C[-1], self.N[j]))
        if not R:
            e = torch.zeros(0, dtype=torch.int64, device="cuda")
            return e, e, e.double()
        R, C, Z, SR, SC = (torch.cat(q) for q in (R, C, Z, SR, SC))
        return torch.cat([R, R + SR]), torch.cat([C, C + SC]), torch.cat([Z, Z])

    def apply(self, p, x):
        """M x for x (nrhs, n)."""
        y = torch.zeros_like(x)
        for i in range(self.nd):
            T, K = self.blocks(i, p["k0"] * math.sqrt(p["eps_r"][i] * p["mu_r"][i]))
            rho, o, N = math.sqrt(p["eps_r"][i] / p["mu_r"][i]), self.off[i], self.N[i]
            D, H = x[:, o:o + N], x[:, o + N:o + 2 * N]
            y[:, o:o + N] = 2 * (D @ K.T + H @ T.T / rho)
            y[:, o + N:o + 2 * N] = 2 * (H @ K.T - rho * (D @ T.T))
        R, C, Z = self.exchange()
        return y.index_add_(1, R, x[:, C] * Z)

    def solve(self, p):
        """Solutions (nrhs, n) of the plane waves by LU."""
        n = int(self.off[-1])
        M = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
        for i in range(self.nd):
            T, K = self.blocks(i, p["k0"] * math.sqrt(p["eps_r"][i] * p["mu_r"][i]))
            rho, o, N = math.sqrt(p["eps_r"][i] / p["mu_r"][i]), self.off[i], self.N[i]
            M[o:o + N, o:o + N] = M[o + N:o + 2 * N, o + N:o + 2 * N] = 2 * K
            M[o:o + N, o + N:o + 2 * N] = 2 * T / rho
            M[o + N:o + 2 * N, o:o + N] = -2 * rho * T
        R, C, Z = self.exchange()
        M.view(-1).index_add_(0, R * n + C, Z.to(torch.complex128))
        b = torch.zeros((n, len(p["dirs"])), dtype=torch.complex128, device="cuda")
        for q, (d, e) in enumerate(zip(p["dirs"], p["pols"])):
            ph = torch.exp(1j * p["k0"] * (self.X[0] @ _cuda(d))) * self.W[0]
            for slot, vec in ((0, e), (1, np.cross(d, e))):
                loc = torch.einsum("tq,tqa->ta", ph, torch.einsum("taqc,c->tqa", self.f[0].to(ph.dtype), _cuda(vec.astype(complex))))
                b[:, q].index_add_(0, (slot * self.N[0] + self.dof[0]).reshape(-1), 2 * loc.reshape(-1))
        return torch.linalg.solve(M, b).T.contiguous()

    def farfield(self, p, x):
        obs, k = _cuda(OBS), p["k0"]
        f = self.f[0].to(torch.complex128)
        ph = torch.exp(-1j * k * torch.einsum("tqc,oc->otq", self.X[0], obs)) * self.W[0][None]
        E = []
        for xr in x:
            w = [torch.einsum("otq,tqc->oc", ph, torch.einsum("ta,taqc->tqc", xr[s * self.N[0] + self.dof[0]], f)) for s in (0, 1)]
            ob = obs.to(w[0].dtype)
            E.append(1j * k / (4 * math.pi) * (torch.cross(ob, w[0], dim=1) + torch.cross(torch.cross(ob, w[1], dim=1), ob, dim=1)))
        return torch.stack(E)

    def nearfield(self, p, x, pts, dom):
        """Stratton-Chu representation of block dom[q] at each point."""
        out = torch.zeros((len(x), len(pts), 3), dtype=torch.complex128, device="cuda")
        for i in np.unique(dom):
            sel = torch.from_numpy(np.where(dom == i)[0]).cuda()
            k, rho = p["k0"] * math.sqrt(p["eps_r"][i] * p["mu_r"][i]), math.sqrt(p["eps_r"][i] / p["mu_r"][i])
            f = self.f[i].to(torch.complex128)
            for s in range(0, len(sel), 64):
                q = sel[s:s + 64]
                d = _cuda(pts)[q][:, None, None] - self.X[i][None]
                r = torch.linalg.vector_norm(d, dim=-1)
                G = torch.exp(1j * k * r) / (4 * math.pi * r) * self.W[i][None]
                gd = (G * (1j * k - 1 / r) / r)[..., None] * d
                for n, xr in enumerate(x):
                    uD, uN = xr[self.off[i] + self.dof[i]], xr[self.off[i] + self.N[i] + self.dof[i]] / rho
                    a, b = torch.einsum("ta,taqc->tqc", uD, f), torch.einsum("ta,taqc->tqc", uN, f)
                    div = (2 * uN * self.c[i]).sum(1)
                    out[n, q] = (torch.cross(gd, a[None].expand_as(gd), dim=-1).sum((1, 2)) + 1j * k * torch.einsum("ptq,tqc->pc", G, b)
                                 + (1j / k) * torch.einsum("t,ptqc->pc", div, gd))
        return out

    def osrc(self, p, r):
        """Block-OSRC apply (sphere-like boundaries): T~ = W diag(f) W^T over irrotational and loop modes, Pade order 16."""
        z = torch.zeros_like(r)
        for i in range(self.nd):
            N, F, area, f, dof = self.N[i], self.F[i], self.area[i], self.f[i], self.dof[i]
            G, D = (torch.zeros((N, N), dtype=torch.float64, device="cuda") for _ in range(2))
            self._add(G, dof, dof, torch.einsum("tq,taqc,tbqc->tab", self.W[i], f, f))
            self._add(D, dof, dof, 4 * area[:, None, None] * self.c[i][:, :, None] * self.c[i][:, None])
            vert, pos = torch.unique(F, return_inverse=True)
            S, M = (torch.zeros((len(vert), len(vert)), dtype=torch.float64, device="cuda") for _ in range(2))
            opp = torch.roll(self.v[i], -2, 1) - torch.roll(self.v[i], -1, 1)  # edge opposite each vertex
            self._add(S, pos, pos, torch.einsum("tac,tbc->tab", opp, opp) / (4 * area[:, None, None]))
            self._add(M, pos, pos, area[:, None, None] * ((torch.ones(3, 3) + torch.eye(3)) / 12).double().cuda())

            def pencil(A, B):
                Ci = torch.linalg.inv(torch.linalg.cholesky(B))
                lam, Q = torch.linalg.eigh(Ci @ A @ Ci.T)
                return lam, Ci.T @ Q

            lam, Vi = pencil(D, G)
            mu, Phi = pencil(S, M)
            nirr = len(F) - 1
            e = self.edges[i]
            ln = _cuda(np.linalg.norm(self.V[e[:, 1]] - self.V[e[:, 0]], axis=1))
            lo, hi = (torch.searchsorted(vert, _cuda(e[:, q])) for q in (0, 1))
            U = (Phi[lo, 1:] - Phi[hi, 1:]) / ln[:, None] / torch.sqrt(mu[1:])[None]
            k, rho = p["k0"] * math.sqrt(p["eps_r"][i] * p["mu_r"][i]), math.sqrt(p["eps_r"][i] / p["mu_r"][i])
            keps = k + 1j * 0.39 * k ** (1 / 3) * float(area.sum() / (4 * math.pi)) ** (-1 / 3)
            Np, th = 16, math.pi / 2
            j = np.arange(1, Np + 1)
            a, b, ph = 2 / (2 * Np + 1) * np.sin(j * np.pi / (2 * Np + 1)) ** 2, np.cos(j * np.pi / (2 * Np + 1)) ** 2, np.exp(-1j * th)
            C0 = np.exp(1j * th / 2) * (1 + np.sum(a * (ph - 1) / (1 + b * (ph - 1))))
            A, B = _cuda(np.exp(-1j * th / 2) * a / (1 + b * (ph - 1)) ** 2), _cuda(ph * b / (1 + b * (ph - 1)))

            def root(q):
                q = (-q / keps ** 2)[:, None]
                return complex(C0) + (A * q / (1 + B * q)).sum(1)

            W = torch.cat([Vi[:, -nirr:], U], 1).to(torch.complex128)
            sym = torch.cat([2 * k / (keps * root(lam[-nirr:])), 2 * keps / k * root(mu[1:])])
            o = self.off[i]
            t = [((r[:, o + s * N:o + (s + 1) * N] @ W) * sym) @ W.T for s in (0, 1)]
            z[:, o:o + N], z[:, o + N:o + 2 * N] = t[1] / rho, -rho * t[0]
        return z


def exact(case, seed):
    """What run() returns for prepare(case, seed), in FP64; None where it would take long (LU of more than 20,000
    unknowns, eigenpairs of more than 3,000, blocks of more than 6,000)."""
    meshes, probs, rng = _problems(case, seed)
    op, p = case["op"], probs[0]
    ex = [_Exact(m) for m in meshes]
    n = [int(e.off[-1]) for e in ex]
    if op in ("oneshot", "solve", "sweep", "batch") and sum(float(q) ** 3 for q in n) > 3e12:
        return None
    if op == "precond_f32" and max(ex[0].N) > 3000:
        return None
    if op in ("assemble", "sweep"):
        p = _problem(case, meshes[0], rng)
    if op == "oneshot":
        x = ex[0].solve(p)
        return x, ex[0].farfield(p, x)
    if op == "batch":
        return [e.solve(q) for e, q in zip(ex, probs)]
    if op == "assemble":
        out = []
        for i in range(meshes[0].n_domains):
            out += list(ex[0].blocks(i, p["k0"] * math.sqrt(p["eps_r"][i] * p["mu_r"][i])))
        return out
    if op == "matvec":
        return ex[0].apply(p, _vectors(seed, case["nrhs"], n[0], torch.complex128))
    if op == "matvec_f32":
        return ex[0].apply(p, _vectors(seed, case["nrhs"], n[0], torch.complex64).to(torch.complex128))
    if op == "precond_f32":
        return ex[0].osrc(p, _vectors(seed, case["nrhs"], n[0], torch.complex64).to(torch.complex128))
    if op == "solve":
        return ex[0].solve(p)
    if op == "sweep":
        x = ex[0].solve(p)
        return x, ex[0].farfield(p, x)
    pts, dom = _points(case, meshes[0], rng)
    x = _vectors(seed, case["nrhs"], n[0], torch.complex128)
    return ex[0].farfield(p, x), ex[0].nearfield(p, x, pts, dom)
