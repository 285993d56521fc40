"""Performance cases: the calls a user of the capacity library makes, at the sizes they make them.

Geometry comes from the repository's own generators (cubes, polycubes, tetrahedra).  The
topology of a case is fixed by the case; its seed draws an affine map (rotations, a moderate
anisotropic scaling, a shift), so that another seed is another polyhedron with other panels,
other distances and no accidental symmetry (on a symmetric surface the marking decides ties
that only rounding tells apart).

One library context serves the process, as it does in a user's program: it keeps the tuned
far-field tiles and the memory of earlier calls.
"""
import functools
import math

import numpy as np
import torch

from paper_1901_08393_gb300 import bem, inputs

TOL = 1e-12  # relative residual of the solves: the default of bem.adaptive_run
THETA = 0.5
PRECISION = {"f64": bem.PREC_F64, "df64": bem.PREC_DF64, "f32": bem.PREC_F32}
PRECOND = {"jacobi": bem.PRECOND_JACOBI, "block": bem.PRECOND_BLOCK, "calderon": bem.PRECOND_CALDERON}
BYTES = {"f64": 8, "df64": 8, "f32": 4}


def listed():
    return [
        # the first contact with the library and its smallest call: the unit cube with 192
        # triangles in the default precision, from host arrays to the indicators
        {"name": "evaluate_cube192_f64", "kind": "evaluate", "precision": "f64", "precond": "jacobi",
         "shape": "cube", "n": 4},
        # one level of a user's own adaptive loop on a small mesh: latency
        {"name": "evaluate_polycube604_df64", "kind": "evaluate", "precision": "df64", "precond": "block",
         "shape": "polycube", "g": 6, "s": 1, "shape_seed": 1},
        # a native FP64 operator, assembled, read and applied: the reference precision of a study
        {"name": "assemble_f64_2416", "kind": "assemble", "precision": "f64", "shape": "polycube", "g": 6,
         "s": 2, "shape_seed": 1},
        # the FP64-accurate operator at an ordinary size, an odd one
        {"name": "assemble_df64_9664", "kind": "assemble", "precision": "df64", "shape": "polycube", "g": 6,
         "s": 4, "shape_seed": 1},
        # solves of a kept operator, small (latency) and large (bandwidth), the paper's diagonal
        # preconditioner and the block one
        {"name": "solve_df64_jacobi_2352", "kind": "solve", "precision": "df64", "precond": "jacobi",
         "shape": "cube", "n": 14},
        {"name": "solve_df64_block_15100", "kind": "solve", "precision": "df64", "precond": "block",
         "shape": "polycube", "g": 6, "s": 5, "shape_seed": 1},
        # the precision form: a cube graded toward its edges, FP32 operator, FP64-accurate residuals
        {"name": "evaluate_graded_f32_49152", "kind": "evaluate", "precision": "f32", "precond": "block",
         "shape": "graded", "n": 64},
        # the adaptive step between two solves on a large mesh: indicators, marking, bisection
        {"name": "refine_38656", "kind": "refine", "shape": "polycube", "g": 6, "s": 8, "shape_seed": 1},
        # whole adaptive computations: the primal basis to 20,000 triangles, the dual basis
        # with operator preconditioning
        {"name": "adaptive_polycube_20k", "kind": "adaptive", "basis": "p0", "g": 6, "shape_seed": 1,
         "max_N": 20000},
        {"name": "adaptive_dual_3k", "kind": "adaptive", "basis": "dual", "g": 3, "shape_seed": 2, "max_N": 3000},
        # many uneven meshes assembled and solved together
        {"name": "batch_f32_24", "kind": "batch", "count": 24, "lo": 500, "hi": 12000, "shape_seed": 4},
        # adaptive requests on uneven shapes, served together
        {"name": "serve_f32_6", "kind": "serve", "count": 6, "lo": 5000, "hi": 16000, "shape_seed": 5},
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def polycube(lo, hi):
        """Shape of a polycube whose faces are split into about lo..hi triangles in all."""
        g, seed = rng.randint(2, 7), rng.randrange(1, 1000)
        s = int(round(math.sqrt(log(lo, hi) / _base("polycube", g, 1, seed)[1].shape[0])))
        while s > 1 and _base("polycube", g, 1, seed)[1].shape[0] * s * s > hi:
            s -= 1
        return {"shape": "polycube", "g": g, "s": max(1, s), "shape_seed": seed}

    kind = rng.choice(["evaluate", "assemble", "assemble", "solve", "solve", "precision", "refine", "adaptive",
                       "dual", "batch", "serve"])
    if kind == "evaluate":
        if rng.random() < 0.5:
            return {"kind": "evaluate", "precision": "f64", "precond": "jacobi", "shape": "cube",
                    "n": int(log(3, 14))}
        return dict({"kind": "evaluate", "precision": "df64", "precond": rng.choice(["jacobi", "block"])},
                    **polycube(150, 8000))
    if kind == "assemble":
        p = rng.choice(["f64", "df64", "df64"])
        return dict({"kind": "assemble", "precision": p}, **polycube(300, 4000 if p == "f64" else 15000))
    if kind == "solve":
        return dict({"kind": "solve", "precision": "df64", "precond": rng.choice(["jacobi", "block"])},
                    **polycube(500, 15500))
    if kind == "precision":
        return {"kind": "evaluate", "precision": "f32", "precond": "block", "shape": "graded", "n": int(log(12, 63))}
    if kind == "refine":
        return dict({"kind": "refine"}, **polycube(500, 38000))
    if kind == "adaptive":
        return {"kind": "adaptive", "basis": "p0", "g": rng.randint(4, 6), "shape_seed": rng.randrange(1, 1000),
                "max_N": int(log(3000, 18000))}
    if kind == "dual":
        return {"kind": "adaptive", "basis": "dual", "g": rng.randint(2, 3), "shape_seed": rng.randrange(1, 1000),
                "max_N": int(log(400, 2800))}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(5, 24), "lo": 500, "hi": int(log(1500, 11000)),
                "shape_seed": rng.randrange(1, 1000)}
    return {"kind": "serve", "count": rng.randint(2, 6), "lo": 3000, "hi": int(log(6000, 15000)),
            "shape_seed": rng.randrange(1, 1000)}


# ---------------------------------------------------------------- geometry
@functools.lru_cache(maxsize=256)
def _base(shape, n, s, seed):
    """(vertices, triangles) of a case's surface before its seed's motion."""
    if shape == "cube":
        m = inputs.cube_mesh(n)
    elif shape == "graded":  # between the uniform grid and one graded quadratically to the edges
        m = inputs.cube_mesh(n)
        u = m.verts
        g = np.where(u <= 0.5, 2.0 * u * u, 1.0 - 2.0 * (1.0 - u) * (1.0 - u))
        return 0.4 * u + 0.6 * g, m.tris
    elif shape == "tetra":
        m = inputs.tetra_mesh(n)
    else:
        m = inputs.polycube_mesh(n, 0.5, seed, sub=s)
    return m.verts, m.tris


def _moved(mesh, rng):
    v, t = mesh
    q, _ = np.linalg.qr(rng.standard_normal((2, 3, 3)))
    a = q[0] @ np.diag(rng.uniform(0.85, 1.2, 3)) @ q[1] * rng.uniform(0.5, 2.0)
    if np.linalg.det(a) < 0:
        a = -a
    return np.ascontiguousarray(v @ a.T + rng.uniform(-1.0, 1.0, 3)), t


def _surface(case, rng):
    return _moved(_base(case["shape"], case.get("n", case.get("g")), case.get("s", 1), case.get("shape_seed", 0)), rng)


def _mixed(case):
    """Base meshes of a batch or of a request stream: uneven shapes, sizes log-uniform in lo..hi."""
    rng = np.random.default_rng(case["shape_seed"])
    out = []
    for k in range(case["count"]):
        target = math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))
        g, seed = int(rng.integers(3, 7)), int(rng.integers(1, 1000))
        if case["kind"] == "serve":
            target /= 1.13 ** 3  # three levels of growth before the final size
        if case["kind"] == "serve" and k % 3 == 1:
            out.append(("cube", max(2, int(round(math.sqrt(target / 12.0)))), 1, 0))
        elif case["kind"] == "serve" and k % 3 == 2:
            out.append(("tetra", max(2, int(round(math.sqrt(target / 4.0)))), 1, 0))
        else:
            faces = _base("polycube", g, 1, seed)[1].shape[0]
            out.append(("polycube", g, max(1, int(round(math.sqrt(target / faces)))), seed))
    return out


def _triangles(case):
    if case["kind"] in ("batch", "serve"):
        return [_base(*k)[1].shape[0] for k in _mixed(case)]
    if case["kind"] == "adaptive":
        return _base("polycube", case["g"], 1, case["shape_seed"])[1].shape[0]
    return _base(case["shape"], case.get("n", case.get("g")), case.get("s", 1), case.get("shape_seed", 0))[1].shape[0]


# ---------------------------------------------------------------- the calls
@functools.lru_cache(maxsize=1)
def _context():
    return bem.Context()


@functools.lru_cache(maxsize=1)
def _server():
    return bem.Server(slots=4, hbm_budget_bytes=64 << 30, theta=THETA, precision=bem.PREC_F32, tol=TOL,
                      precond=bem.PRECOND_BLOCK)


def prepare(case, seed):
    rng = np.random.default_rng([seed, 1901])
    kind = case["kind"]
    state = dict(case)
    if kind == "batch":
        ctx = _context()
        meshes = [bem.Mesh.upload(ctx, *_moved(_base(*k), rng)) for k in _mixed(case)]
        state["batch"] = bem.Batch(ctx, meshes, precision=bem.PREC_F32, tol=TOL, precond=bem.PRECOND_BLOCK)
        return state
    if kind == "serve":
        _server()
        state["meshes"] = [_moved(_base(*k), rng) for k in _mixed(case)]
        return state
    if kind == "adaptive":
        state["arrays"] = _moved(_base("polycube", case["g"], 1, case["shape_seed"]), rng)
        state["fine"] = _buffers(2 * case["max_N"])
        return state
    state["arrays"] = _surface(case, rng)
    n = state["arrays"][1].shape[0]
    if kind in ("assemble", "solve", "refine"):
        state["mesh"] = bem.Mesh.upload(_context(), *state["arrays"])
    if kind == "assemble":
        state["x"] = torch.from_numpy(rng.uniform(0.5, 1.5, n)).cuda()
        state["V"] = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    if kind == "solve":
        state["op"] = bem.Operator.assemble(state["mesh"], precision=PRECISION[case["precision"]])
    if kind == "refine":
        state["phi"] = _density(*state["arrays"], rng)
        state["fine"] = _buffers(2 * n)
    return state


def _buffers(n):
    """A caller's arrays for a mesh of up to n triangles: their size does not depend on the marking."""
    return {"verts": np.zeros((n, 3)), "tris": np.zeros((n, 3), np.int32), "parent": np.zeros(n, np.int32),
            "kept": np.zeros(n, np.uint8)}


def _download(mesh, into):
    M, N, _ = mesh.info()
    if max(M, N) > len(into["tris"]):
        raise RuntimeError("the refined mesh does not fit its buffers")
    mesh.ctx.check(bem.lib().bem_mesh_download(mesh.h, *(into[k].ctypes.data
                                                         for k in ("verts", "tris", "parent", "kept"))))
    return into


def _density(verts, tris, rng):
    """A charge density with the concentration toward the surface's outer corners that the solutions have."""
    c = verts[tris].mean(axis=1)
    d = np.linalg.norm(c - c.mean(axis=0), axis=1)
    return (1.0 + (d / d.max()) ** 4) * (1.0 + 0.02 * rng.uniform(-1.0, 1.0, len(d)))


def run(state):
    kind = state["kind"]
    if kind == "evaluate":
        mesh = bem.Mesh.upload(_context(), *state["arrays"])
        op = bem.Operator.assemble(mesh, precision=PRECISION[state["precision"]])
        cap, phi, _ = bem.solve_capacity(op, tol=TOL, precond=PRECOND[state["precond"]])
        eta2, total, _ = bem.zz_estimate(mesh, phi)
        return {"cap": cap, "phi": phi, "eta2": eta2, "total": total}
    if kind == "assemble":
        op = bem.Operator.assemble(state["mesh"], precision=PRECISION[state["precision"]])
        n = op.info()[0]  # the whole matrix into the caller's device array, and a product with it
        op.ctx.check(bem.lib().bem_operator_read(op.h, 0, n, 0, n, state["V"].data_ptr()))
        return {"V": state["V"], "y": op.matvec(state["x"])}
    if kind == "solve":
        phi = torch.empty(state["mesh"].N, dtype=torch.float64, device="cuda")
        cap, _, _ = bem.solve_capacity(state["op"], tol=TOL, precond=PRECOND[state["precond"]], phi_out=phi)
        return {"cap": cap, "phi": phi}
    if kind == "refine":
        eta2, total, _ = bem.zz_estimate(state["mesh"], state["phi"])
        marked, n, fine = bem.mark_refine(state["mesh"], eta2, THETA)
        return dict(_download(fine, state["fine"]), eta2=eta2, total=total, marked=marked, n=n)
    if kind == "adaptive":
        mesh = bem.Mesh.upload(_context(), *state["arrays"])
        dual = state["basis"] == "dual"
        levels, last = bem.adaptive_run(mesh, theta=THETA, max_N=state["max_N"], tol=TOL, precision=bem.PREC_DF64,
                                        precond=PRECOND["calderon" if dual else "block"],
                                        basis=bem.BASIS_DUAL if dual else bem.BASIS_P0, want_final=True)
        out = {f: np.zeros(64, t) for f, t in (("N", np.int64), ("M", np.int64), ("n_marked", np.int64),
                                               ("cap", np.float64), ("eta2_total", np.float64))}
        for k, r in enumerate(levels):
            for f in out:
                out[f][k] = r[f]
        return dict(_download(last, state["fine"]), **out)
    if kind == "batch":
        return {"cap": np.array([r["cap"] for r in state["batch"].run()])}
    server = _server()
    ids = [server.submit(v, t, max_levels=4, max_N=int(1.13 ** 3 * len(t))) for v, t in state["meshes"]]
    done = [server.wait(i) for i in ids]
    caps, sizes = np.zeros((len(done), 4)), np.zeros((len(done), 4), np.int64)
    for k, r in enumerate(done):
        caps[k, :r["levels"]], sizes[k, :r["levels"]] = r["caps"], r["Ns"]
    return {"caps": caps, "sizes": sizes}


# ---------------------------------------------------------------- what a pass cannot do without
_PAIR = 49 * 10.0   # operations of a far pair: 49 distances, reciprocal roots and sums
_PRODUCTS = 50.0    # products of a solve to TOL; each reads half of a symmetric matrix in FP32


def _assembly(n, size):
    return {"bytes": 1.0 * size * n * n, "flops": 0.5 * n * n * _PAIR}


def _solve(n):
    return {"bytes": _PRODUCTS * 2.0 * n * n, "flops": _PRODUCTS * 2.0 * n * n}


def _sum(parts):
    parts = list(parts)
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def work(case):
    kind, n = case["kind"], _triangles(case)
    if kind == "evaluate":
        return _sum([_assembly(n, BYTES[case["precision"]]), _solve(n)])
    if kind == "assemble":
        return _sum([_assembly(n, BYTES[case["precision"]]),  # read back in FP64, and one product
                     {"bytes": (1.5 * BYTES[case["precision"]] + 8.0) * n * n, "flops": 2.0 * n * n}])
    if kind == "solve":
        return _solve(n)
    if kind == "refine":  # indicators and marks out, the mesh in, the refined one out
        return {"bytes": n * (8.0 + 12.0 + 12.0 + 16.0 + 8.0 + 1.0) + 1.2 * n * (12.0 + 12.0 + 5.0), "flops": 40.0 * n}
    if kind == "adaptive":  # levels grow by about 1.28; a level keeps half of its entries
        sizes = [n]
        while sizes[-1] < case["max_N"]:
            sizes.append(1.28 * sizes[-1])
        if case["basis"] == "p0":
            return _sum(_sum([{k: 0.5 * w for k, w in _assembly(m, 8).items()}, _solve(m)]) for m in sizes)
        return _sum({k: 0.5 * w for k, w in _assembly(6.0 * m, 8).items()} for m in sizes)
    if kind == "batch":
        return _sum(_sum([_assembly(m, 4), _solve(m)]) for m in n)
    return _sum(_sum([_assembly(1.13 ** k * m, 4), _solve(1.13 ** k * m)]) for m in n for k in range(4))


# ---------------------------------------------------------------- the same in 64 bits
def _rotated(verts, tris):
    """Each triangle with its longest edge first (ties: the first such edge)."""
    p = verts[tris]
    e = np.stack([((p[:, (k + 1) % 3] - p[:, k]) ** 2).sum(axis=1) for k in range(3)], axis=1)
    return tris[np.arange(len(tris))[:, None], (e.argmax(axis=1)[:, None] + np.arange(3)) % 3]


def _touching(tris):
    """Pairs i < j with a common vertex, and how many vertices each pair shares."""
    n, m = len(tris), tris.max() + 1
    order = np.argsort(tris.ravel(), kind="stable")
    start = np.searchsorted(tris.ravel()[order], np.arange(m + 1))
    count = np.diff(start)
    pairs = []
    for v in np.unique(count[count > 1]):
        at = start[:-1][count == v][:, None] + np.arange(v)
        t = order[at] // 3
        a, b = np.triu_indices(v, 1)
        pairs.append(np.stack([t[:, a].ravel(), t[:, b].ravel()], axis=1))
    pairs = np.sort(np.concatenate(pairs), axis=1).astype(np.int64)
    key, shared = np.unique(pairs[:, 0] * n + pairs[:, 1], return_counts=True)
    return key // n, key % n, shared


def _operator64(verts, tris):
    """The Galerkin matrix by the definition: Radon's rule on pairs without a common vertex, the
    regularised Gauss rule of order 4 on the others; FP64 on the GPU."""
    tris = _rotated(verts, tris)
    n = len(tris)
    p = torch.from_numpy(verts[tris]).cuda()
    area = 0.5 * torch.linalg.norm(torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), dim=1)
    r15 = math.sqrt(15.0)
    pts, wts = [p.mean(dim=1)], [9.0 / 40.0]
    for a, w in (((6.0 - r15) / 21.0, (155.0 - r15) / 1200.0), ((6.0 + r15) / 21.0, (155.0 + r15) / 1200.0)):
        for k in range(3):
            b = [a, a, a]
            b[k] = 1.0 - 2.0 * a
            pts.append(b[0] * p[:, 0] + b[1] * p[:, 1] + b[2] * p[:, 2])
            wts.append(w)
    V = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    rows = max(1, (1 << 24) // n)
    for r in range(0, n, rows):
        for a in range(7):
            for b in range(7):
                x, y = pts[a][r:r + rows], pts[b]
                d = (x[:, None, 0] - y[None, :, 0]) ** 2
                d += (x[:, None, 1] - y[None, :, 1]) ** 2
                d += (x[:, None, 2] - y[None, :, 2]) ** 2
                V[r:r + rows] += wts[a] * wts[b] * d.rsqrt_()
        V[r:r + rows] *= area[r:r + rows, None] * area[None, :]
    gx, gw = np.polynomial.legendre.leggauss(4)
    gx, gw = 0.5 * (gx + 1.0), 0.5 * gw

    def inv(v):
        return 1.0 / torch.linalg.norm(v, dim=-1)

    # identical panels: the six sectors of the difference hexagon
    j1, j2 = p[:, 1] - p[:, 0], p[:, 2] - p[:, 1]
    hexagon = [(1, 0), (1, 1), (0, 1), (-1, 0), (-1, -1), (0, -1), (1, 0)]
    same = torch.zeros(n, dtype=torch.float64, device="cuda")
    for (ax, ay), (bx, by) in zip(hexagon[:-1], hexagon[1:]):
        for x, w in zip(gx, gw):
            same += w * inv((ax + x * (bx - ax)) * j1 + (ay + x * (by - ay)) * j2)
    k = torch.arange(n, device="cuda")
    V[k, k] = 4.0 * area * area * same / 6.0
    i, j, shared = _touching(tris)
    ti, tj = tris[i], tris[j]
    match = ti[:, :, None] == tj[:, None, :]
    X = torch.from_numpy(verts).cuda()
    for c in (1, 2):
        on = shared == c
        if not on.any():
            continue
        a, b, mt = ti[on], tj[on], match[on]
        rows = np.arange(len(a))
        if c == 1:  # both triangles turned to start at the common vertex
            ka, kb = mt.any(axis=2).argmax(axis=1), mt.any(axis=1).argmax(axis=1)
            a = a[rows[:, None], (ka[:, None] + np.arange(3)) % 3]
            b = b[rows[:, None], (kb[:, None] + np.arange(3)) % 3]
        else:  # (u, v, own vertex), u and v in the order of the first triangle
            free = (~mt.any(axis=2)).argmax(axis=1)
            u = np.where(free == 0, 1, 0)
            v = np.where(free == 2, 1, 2)
            cj = b[rows, (~mt.any(axis=1)).argmax(axis=1)]
            a = np.stack([a[rows, u], a[rows, v], a[rows, free]], axis=1)
            b = np.stack([a[:, 0], a[:, 1], cj], axis=1)
        P, Q = X[torch.from_numpy(a.astype(np.int64)).cuda()], X[torch.from_numpy(b.astype(np.int64)).cuda()]
        e, fp, fq = P[:, 1] - P[:, 0], P[:, 2] - P[:, 1], Q[:, 2] - Q[:, 1]
        eq = Q[:, 1] - Q[:, 0]
        s = torch.zeros(len(a), dtype=torch.float64, device="cuda")
        for u, wu in zip(gx, gw):
            for v, wv in zip(gx, gw):
                if c == 2:
                    for own, t, other, w in ((1.0, u * (1.0 - v), u * v, u), (u, 1.0 - v, v, 1.0)):
                        s += wu * wv * w * (inv(t * e + own * fp - other * fq) + inv(-t * e + other * fp - own * fq))
                else:
                    x, y = e + u * fp, eq + v * fq
                    for z, wz in zip(gx, gw):
                        s += wu * wv * wz * z * (inv(x - z * y) + inv(z * x - y))
        I, J = torch.from_numpy(i[on]).cuda(), torch.from_numpy(j[on]).cuda()
        s *= 4.0 * area[I] * area[J] / (3.0 if c == 1 else 6.0)
        V[I, J] = s
        V[J, I] = s
    return V.mul_(0.25 / math.pi), area


def _indicators64(verts, tris, phi):
    """Indicators eta(T)^2 and their sum, and the scale of the solution, in numpy."""
    tris = _rotated(verts, tris)
    p = verts[tris]
    area = 0.5 * np.linalg.norm(np.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]), axis=1)
    h = np.sqrt(np.stack([((p[:, (k + 1) % 3] - p[:, k]) ** 2).sum(axis=1) for k in range(3)])).max(axis=0)
    num, den = np.zeros(len(verts)), np.zeros(len(verts))
    for k in range(3):
        np.add.at(num, tris[:, k], area * phi)
        np.add.at(den, tris[:, k], area)
    d = (num / den)[tris] - phi[:, None]
    eta2 = h * area / 12.0 * ((d ** 2).sum(axis=1) + d.sum(axis=1) ** 2)
    return eta2, float(eta2.sum())


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("evaluate", "assemble", "solve", "refine") or (kind != "refine" and _triangles(case) > 16000):
        return None
    rng = np.random.default_rng([seed, 1901])
    verts, tris = _surface(case, rng)
    if kind == "refine":
        eta2, total = _indicators64(verts, tris, _density(verts, tris, rng))
        return {"eta2": eta2, "total": total, "marked": None, "n": None, "verts": None, "tris": None,
                "parent": None, "kept": None}
    V, area = _operator64(verts, tris)
    if kind == "assemble":
        return {"V": V, "y": (V @ torch.from_numpy(rng.uniform(0.5, 1.5, len(tris))).cuda()).cpu().numpy()}
    phi = torch.linalg.solve(V, area)
    cap = float(area @ phi) * 0.25 / math.pi
    if kind == "solve":
        return {"cap": cap, "phi": phi}
    phi = phi.cpu().numpy()
    eta2, total = _indicators64(verts, tris, phi)
    return {"cap": cap, "phi": phi, "eta2": eta2, "total": total}
