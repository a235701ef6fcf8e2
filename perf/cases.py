"""The calls a user of the eigensolver makes, for timing: the steps of the method (set-up,
orthonormalisation, projection in each precision, inverse power, residuals) and the whole
solve, through the package's Python entry points.

Meshes are closed triangle surfaces (icosphere, unit cube, ellipsoid); bases and test
vectors are complex Gaussian, drawn on the GPU from the seed. A mesh, a contour and a basis
are what a program holds before a step; it keeps one Context per problem.

``exact`` evaluates the same quantities densely with torch in 64 bits, from the formulas of
the discretisation: 7-point rule off the diagonal, polar self term, 8 x 8 conical rule on
near pairs, T = c_G G + c_H (I/2 + K).
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_1906_03938_gb300 as bem

DEV = "cuda:0"
PRECISION = {"fp64": bem.PREC_FP64, "mixed": bem.PREC_MIXED, "hmatrix": bem.PREC_HMATRIX}
# c_G, c_H of the boundary operator: Dirichlet (the default), Neumann, Robin
OPERATOR = {"single": (1.0, 0.0), "neumann": (0.0, 1.0), "robin": (0.5 + 0.2j, 1.0 - 0.3j)}


def _step(name, shape, size, contour, N, nu, precision="mixed", near=0, op="single", av=False):
    centre, a, b = contour
    case = {"kind": "step", "shape": shape, "size": size, "centre": centre, "a": a, "b": b,
            "N": N, "nu": nu, "precision": precision, "near": near, "op": op, "av": av}
    return case if name is None else {"name": name, **case}


def listed():
    return [
        # one projection step (mesh, contour, CholeskyQR2, B_j = w_j V^H A(z_j) V) on the
        # coarse sphere: what a parameter study repeats thousands of times; launches count
        _step("step_sphere320", "ico", 2, (4.0, 1.0, 1.0), 16, 16),
        # the unit cube of the method's first example: the ordinary step
        _step("step_cube3072", "cube", 16, (6.5, 1.5, 0.4), 32, 64),
        # a fine sphere with the near-field rule, as accuracy at that size asks for
        _step("step_sphere20480_near", "ico", 5, (7.0, 1.0, 1.0), 32, 128, near=1),
        # the widest basis: the largest projection
        _step("step_ellipsoid24576", "tet", 5, (9.0, 1.5, 1.5), 16, 256),
        # impedance walls (Robin), ragged sizes, the products A(z_j) V kept for the stopping
        # test
        _step("step_robin1452", "ell", 11, (2.75, 0.9, 0.9), 24, 30, near=1, op="robin", av=True),
        # the default precision of project(): the cube at half resolution in plain FP64
        _step("step_fp64_cube768", "cube", 8, (6.5, 1.5, 0.4), 32, 64, precision="fp64"),
        # the compressed operator (low-rank far field) on the cube
        _step("step_hmatrix_cube3072", "cube", 16, (6.5, 1.5, 0.4), 32, 64, precision="hmatrix"),
        # a sweep over bodies: several ellipsoids projected by one recorded batch, replayed
        {"name": "batch_8_ellipsoids", "kind": "batch", "count": 8, "mix": 1, "tri_lo": 500,
         "tri_hi": 6000, "nu": 32},
        # orthonormalising the widest basis on the finest mesh
        {"name": "orth_98304x256", "kind": "orth", "n": 98304, "nu": 256},
        # improving the basis on the cube: dense factorisation and inverse power steps
        {"name": "improve_cube3072", "kind": "improve", "shape": "cube", "size": 16,
         "centre": 6.5, "a": 1.5, "b": 1.5, "N": 32, "nu": 64, "q": 2},
        # certifying eigenpairs on a middle-sized sphere: FP64 residuals of eight vectors
        {"name": "residual_sphere5120", "kind": "residual", "shape": "ico", "size": 4,
         "centre": 7.0, "near": 1, "m": 8, "arith": 0},
        # the whole method, mesh to refined eigenpairs, on a coarse ellipsoid
        {"name": "solve_ellipsoid768", "kind": "solve", "shape": "ell", "size": 8, "centre": 6.4,
         "a": 0.6, "b": 0.38, "N": 24, "nu": 24, "q": 3},
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def contour():
        a = round(rng.uniform(0.6, 1.6), 3)
        return round(rng.uniform(2.5, 9.0), 3), a, rng.choice([a, a, round(0.3 * a, 3)])

    def mesh(lo, hi):
        shape = rng.choice(["cube", "ell", "ell"])
        return shape, max(2, round(math.sqrt(log(lo, hi) / 12.0)))

    kind = rng.choice(["step"] * 8 + ["batch", "orth", "improve", "residual", "residual", "solve"])
    if kind == "step":
        precision = rng.choice(["mixed", "mixed", "mixed", "fp64", "fp64", "hmatrix"])
        near, op = rng.choice([0, 0, 1]), rng.choice(["single", "single", "neumann", "robin"])
        N = rng.choice([8, 12, 16, 23, 24, 32, 33])
        if precision == "mixed":
            shape, m = mesh(300, 16000)
            n = 12 * m * m
            nu = min(n // 2, round(log(12, 256)))
            while n * n * N * max(nu, 64) > 2.2e12:   # no more than the widest listed step
                N = N // 2
        elif precision == "fp64":
            shape, m = mesh(300, 1100)
            n = 12 * m * m
            nu = min(n // 2, round(log(10, 100)))
            while n * n * N > 2e7:
                N = N // 2
            op = rng.choice(["single", "single", "robin"])
        else:
            shape, m = mesh(700, 4000)
            nu = round(log(16, 128))
            op = "single"
        return _step(None, shape, m, contour(), N, nu, precision, near, op, rng.choice([False, True]))
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 12), "mix": rng.randint(2, 1000),
                "tri_lo": 500, "tri_hi": rng.choice([2000, 4000, 6000]),
                "nu": rng.choice([16, 24, 32])}
    if kind == "orth":
        nu = round(log(8, 256))
        return {"kind": "orth", "n": max(4 * nu, round(log(500, 98000))), "nu": nu}
    shape, m = mesh(600, 3000)
    centre, a, _ = contour()
    if kind == "improve":
        return {"kind": kind, "shape": shape, "size": m, "centre": centre, "a": a, "b": a,
                "N": rng.choice([16, 24, 32]), "nu": round(log(16, 64)), "q": rng.randint(1, 2)}
    if kind == "residual":
        return {"kind": kind, "shape": shape, "size": m, "centre": centre,
                "near": rng.choice([0, 1]), "m": rng.randint(1, 12), "arith": rng.choice([0, 1])}
    return {"kind": "solve", "shape": "ell", "size": rng.choice([6, 7, 8]),
            "centre": round(rng.uniform(6.36, 6.44), 3), "a": 0.6, "b": 0.38,
            "N": rng.choice([24, 32]), "nu": rng.randint(20, 32), "q": 3}


# ---- meshes -------------------------------------------------------------------------------

# (lower corner, u, v) of the faces of the unit cube, u x v outward
_FACES = (((0, 0, 0), (0, 0, 1), (0, 1, 0)), ((1, 0, 0), (0, 1, 0), (0, 0, 1)),
          ((0, 0, 0), (1, 0, 0), (0, 0, 1)), ((0, 1, 0), (0, 0, 1), (1, 0, 0)),
          ((0, 0, 0), (0, 1, 0), (1, 0, 0)), ((0, 0, 1), (1, 0, 0), (0, 1, 0)))
AXES = (1.0, 0.7, 0.5)


def _weld(corners):
    """(points, triangles) of an array (triangles, 3, 3) of corner coordinates."""
    flat = corners.reshape(-1, 3)
    _, first, inverse = np.unique(np.round(flat * 2.0 ** 30).astype(np.int64), axis=0,
                                  return_index=True, return_inverse=True)
    return flat[first], inverse.reshape(-1, 3).astype(np.int32)


def _cube_grid(m):
    i, j = np.meshgrid(np.arange(m), np.arange(m), indexing="ij")
    i, j = i.reshape(-1, 1), j.reshape(-1, 1)
    out = []
    for o, u, v in _FACES:
        o, u, v = (np.array(t, dtype=np.float64) for t in (o, u, v))
        p = lambda x, y: o + (x * u + y * v) / m
        q = [p(i, j), p(i + 1, j), p(i + 1, j + 1), p(i, j + 1)]
        out += [np.stack([q[0], q[1], q[2]], 1), np.stack([q[0], q[2], q[3]], 1)]
    return _weld(np.concatenate(out))


def _split(p, t, project):
    """Each triangle into four at its edge midpoints."""
    a, b, c = (p[t[:, k]] for k in range(3))
    ab, bc, ca = project(0.5 * (a + b)), project(0.5 * (b + c)), project(0.5 * (c + a))
    return _weld(np.concatenate([np.stack(s, 1) for s in
                                 ((a, ab, ca), (ab, b, bc), (ca, bc, c), (ab, bc, ca))]))


def _unit(p):
    return p / np.linalg.norm(p, axis=-1, keepdims=True)


@functools.lru_cache(maxsize=64)
def _mesh(shape, size, axes=AXES):
    if shape == "cube":
        return _cube_grid(size)
    if shape == "ell":
        p, t = _cube_grid(size)
        return np.ascontiguousarray(_unit(2.0 * p - 1.0) * axes), t
    if shape == "ico":
        g = (1.0 + math.sqrt(5.0)) / 2.0
        p = np.array([[s * 1.0, u * g, 0.0] for s in (-1, 1) for u in (-1, 1)])
        p = np.concatenate([p, np.roll(p, 1, axis=1), np.roll(p, 2, axis=1)])
        t = [f for f in itertools.combinations(range(12), 3)
             if all(abs(np.linalg.norm(p[x] - p[y]) - 2.0) < 1e-9
                    for x, y in itertools.combinations(f, 2))]
        t = [f if np.linalg.det(p[list(f)]) > 0 else (f[0], f[2], f[1]) for f in t]
        p, t = _unit(p), np.array(t, dtype=np.int32)
        for _ in range(size):
            p, t = _split(p, t, _unit)
        return np.ascontiguousarray(p), t
    # "tet": cube faces in four about their centres, split ``size`` times, then projected
    tris = []
    for o, u, v in _FACES:
        o, u, v = (2.0 * np.array(x, dtype=np.float64) for x in (o, u, v))
        q = [o - 1.0, o + u - 1.0, o + u + v - 1.0, o + v - 1.0]
        tris += [np.stack([q[k], q[(k + 1) % 4], sum(q) / 4.0]) for k in range(4)]
    p, t = _weld(np.stack(tris))
    for _ in range(size):
        p, t = _split(p, t, lambda x: x)
    return np.ascontiguousarray(_unit(p) * axes), t


def _panels(shape, size):
    return {"cube": 12 * size * size, "ell": 12 * size * size, "ico": 20 * 4 ** size,
            "tet": 24 * 4 ** size}[shape]


def _problems(case):
    """(mesh size, axes, N, centre) of the bodies of a batch."""
    r = np.random.RandomState(case["mix"])
    out = []
    for _ in range(case["count"]):
        axes = tuple(float(x) for x in 0.5 + 1.5 * r.rand(3))
        tri = math.exp(r.uniform(math.log(case["tri_lo"]), math.log(case["tri_hi"])))
        out.append((max(2, int(round(math.sqrt(tri / 12.0)))), axes, int(r.choice([16, 24, 32])),
                    2.0 + 6.0 * float(r.rand())))
    return out


def _gauss(seed, *shape):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return torch.randn(*shape, dtype=torch.complex128, device=DEV, generator=g)


def _columns(seed, n, nu):
    """n x nu Gaussian basis, column-major."""
    return _gauss(seed, nu, n).t()


def _ellipse(case):
    return "circle" if case["a"] == case["b"] else "ellipse"


# ---- the calls ----------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "orth":
        V0 = _columns(seed, case["n"], case["nu"])
        return {"case": case, "ctx": bem.Context(0), "V0": V0, "V": torch.empty_like(V0)}
    if kind == "batch":
        ctxs, Vs = [], []
        for k, (m, axes, N, centre) in enumerate(_problems(case)):
            xyz, tri = _mesh("ell", m, axes)
            ctx = bem.Context(0)
            ctx.set_mesh(xyz, tri)
            ctx.set_contour("circle", centre, 0.8, 0.8, N)
            ctxs.append(ctx)
            Vs.append(_columns(1000 * seed + k, len(tri), case["nu"]))
        return {"case": case, "batch": bem.Batch(ctxs, Vs)}
    xyz, tri = _mesh(case["shape"], case["size"])
    n = len(tri)
    ctx = bem.Context(0)
    ctx.set_mesh(xyz, tri)
    state = {"case": case, "ctx": ctx}
    if kind == "residual":
        ctx.set_near_field(case["near"])
        lam, X = _pairs(case, seed, n)
        return {**state, "lam": lam, "X": X}
    V0 = _columns(seed, n, case["nu"])
    if kind == "step":
        ctx.set_async(True)
        ctx.set_operator(*OPERATOR[case["op"]])
        ctx.set_near_field(case["near"])
        if case["precision"] == "hmatrix":
            ctx.set_hmatrix()
        return {**state, "xyz": xyz, "tri": tri, "V0": V0, "V": torch.empty_like(V0)}
    ctx.set_contour(_ellipse(case), case["centre"], case["a"], case["b"], case["N"])
    if kind == "improve":
        return {**state, "V0": V0, "V": torch.empty_like(V0)}
    return {**state, "V0": V0, "w": _probe(n)}


def _pairs(case, seed, n):
    """Trial eigenpairs: values near the real axis about the centre, unit vectors."""
    r = np.random.RandomState(seed % 2 ** 31)
    lam = case["centre"] + 0.8 * r.uniform(-1, 1, case["m"]) + 1j * r.uniform(-1e-2, 1e-2, case["m"])
    X = _columns(seed, n, case["m"])
    return lam, X / torch.linalg.vector_norm(X, dim=0)


def _probe(n):
    """The fixed vector that eigenvectors are scaled by, w^H x = 1."""
    return _gauss(20190609, n)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        return state["batch"].run()
    ctx = state["ctx"]
    if kind == "step":
        ctx.set_mesh(state["xyz"], state["tri"])
        ctx.set_contour(_ellipse(case), case["centre"], case["a"], case["b"], case["N"])
        V = state["V"]
        V.copy_(state["V0"])
        ctx.cholqr2(V, want_R=False)
        out = ctx.project(V, PRECISION[case["precision"]], AV=case["av"])
        return {"V": V, "B": out[0], "Y": out[1]} if case["av"] else {"V": V, "B": out}
    if kind == "orth":
        V = state["V"]
        V.copy_(state["V0"])
        ctx.cholqr2(V, want_R=False)
        return V
    if kind == "improve":
        V = state["V"]
        V.copy_(state["V0"])
        ctx.inverse_power(V, case["q"], _shift(case))
        return V
    if kind == "residual":
        return ctx.residual_arith(state["lam"], state["X"], arith=case["arith"])[:2]
    lam, X, _ = ctx.solve(state["V0"], q=case["q"], precision=bem.PREC_MIXED)
    order = np.argsort(lam.real)
    X = X[:, torch.from_numpy(order).to(X.device)]
    # eigenvectors in a scaling of the caller's own; the residuals at convergence are
    # rounding noise and are not kept
    return {"lam": lam[order], "X": X / (state["w"].conj() @ X)}


def _shift(case):
    return complex(case["centre"], 0.3 * case["a"])


# ---- what a pass cannot do without --------------------------------------------------------

POINT = 24.0   # flops of one quadrature point of the kernel: distance, root, exponential, sum


def _projection_work(n, N, nu, av=False):
    return {"bytes": 16.0 * (n * nu + N * nu * nu + (N * n * nu if av else 0)) + 40.0 * n,
            "flops": float(n) * n * N * (7 * POINT + 8.0 * nu) + 8.0 * N * n * nu * nu}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_projection_work(12 * m * m, N, case["nu"]) for m, _, N, _ in _problems(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "orth":
        n, nu = case["n"], case["nu"]
        # two Gram matrices (Hermitian halves) and two triangular products
        return {"bytes": 32.0 * n * nu, "flops": 16.0 * n * nu * nu}
    n = _panels(case["shape"], case["size"])
    if kind == "step":
        w = _projection_work(n, case["N"], case["nu"], case["av"])
        w["bytes"] += 16.0 * n * case["nu"]
        w["flops"] += 16.0 * n * case["nu"] ** 2
        return w
    if kind == "residual":
        return {"bytes": 32.0 * n * case["m"] + 40.0 * n,
                "flops": float(n) * n * case["m"] * (7 * POINT + 8)}
    N, nu, q = case["N"], case["nu"], case["q"]
    # the summed matrix, its factorisation, q node-summed products and solves
    improve = (float(n) * n * N * 7 * POINT + 8.0 / 3.0 * float(n) ** 3
               + q * (float(n) * n * N * (7 * POINT + 8.0 * nu) + 8.0 * n * n * nu))
    if kind == "improve":
        return {"bytes": 32.0 * n * nu, "flops": improve}
    # and the projection; one factorisation and a few residuals for the eigenpairs
    return {"bytes": 32.0 * n * nu,
            "flops": improve + _projection_work(n, N, nu)["flops"] + 8.0 / 3.0 * float(n) ** 3}


# ---- the same quantities densely in 64 bits -----------------------------------------------

def _geometry(xyz, tri):
    v = torch.from_numpy(np.asarray(xyz, dtype=np.float64)[np.asarray(tri)]).to(DEV)
    s = math.sqrt(15.0)
    a1, b1, a2, b2 = (6 - s) / 21, (9 + 2 * s) / 21, (6 + s) / 21, (9 - 2 * s) / 21
    bary = torch.tensor([[1 / 3] * 3, [a1, a1, b1], [a1, b1, a1], [b1, a1, a1],
                         [a2, a2, b2], [a2, b2, a2], [b2, a2, a2]], dtype=torch.float64, device=DEV)
    wt = torch.tensor([9 / 40] + [(155 - s) / 1200] * 3 + [(155 + s) / 1200] * 3,
                      dtype=torch.float64, device=DEV)
    cr = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    twice = torch.linalg.vector_norm(cr, dim=1)
    edges = torch.stack([v[:, (e + 1) % 3] - v[:, e] for e in range(3)], 1)
    return {"v": v, "c": v.mean(1), "nrm": cr / twice[:, None], "twice": twice,
            "diam": torch.linalg.vector_norm(edges, dim=2).amax(1),
            "q": torch.einsum("qe,led->lqd", bary, v), "w": 0.5 * twice[:, None] * wt}


def _legendre(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.from_numpy(x).to(DEV), torch.from_numpy(w).to(DEV)


def _kernel(d, nrm, k, op):
    """c_G g + c_H dg/dn at y - x = d (.., 3), without the 1 / 4 pi."""
    r = torch.linalg.vector_norm(d, dim=-1)
    e = torch.exp(-k.imag * r) / r
    g = torch.complex(e * torch.cos(k.real * r), e * torch.sin(k.real * r))
    cg, ch = complex(op[0]), complex(op[1])
    if ch == 0:
        return g if cg == 1 else g * cg
    s = (d * nrm).sum(-1) / (r * r)
    return g * (cg + ch * s * (1j * k * r - 1.0))


def _self(G, k, op):
    """The diagonal: c_G times the polar self integral, plus c_H / 2."""
    gx, gw = _legendre(24)
    total = torch.zeros(len(G["c"]), dtype=torch.complex128, device=DEV)
    for e in range(3):
        p, q = G["v"][:, e], G["v"][:, (e + 1) % 3]
        t = (q - p) / torch.linalg.vector_norm(q - p, dim=1, keepdim=True)
        sp, sq = ((p - G["c"]) * t).sum(1), ((q - G["c"]) * t).sum(1)
        d = torch.linalg.vector_norm(p - G["c"] - sp[:, None] * t, dim=1)
        up, uq = torch.asinh(sp / d), torch.asinh(sq / d)
        mid = torch.minimum(torch.maximum(up, torch.zeros_like(up)), uq)
        for lo, hi in ((up, mid), (mid, uq)):
            u = 0.5 * (hi + lo)[:, None] + 0.5 * (hi - lo)[:, None] * gx
            R = d[:, None] * torch.cosh(u)
            w = 1j * k * R
            small = w.abs() < 0.3
            ws = torch.where(small, w, torch.zeros_like(w))
            term, series = torch.ones_like(w), torch.ones_like(w)
            for m in range(1, 20):
                term = term * ws / (m + 1)
                series = series + term
            wl = torch.where(small, torch.ones_like(w), w)
            h = torch.where(small, series, (torch.exp(wl) - 1.0) / wl)
            total += (0.5 * (hi - lo)[:, None] * gw * d[:, None] * h).sum(1)
    return complex(op[0]) * total / (4 * math.pi) + 0.5 * complex(op[1])


def _near_pairs(G):
    rows, cols = [], []
    for r in torch.arange(len(G["c"]), device=DEV).split(1024):
        dist = torch.cdist(G["c"][r], G["c"], compute_mode="donot_use_mm_for_euclid_dist")
        i, l = (dist < 2.0 * torch.maximum(G["diam"][r][:, None], G["diam"][None, :])).nonzero(as_tuple=True)
        rows.append(r[i])
        cols.append(l)
    i, l = torch.cat(rows), torch.cat(cols)
    return i[i != l], l[i != l]


def _near_values(G, i, l, k, op):
    """8 x 8 conical rule of the pairs (i, l), collapsed at the vertex nearest x_i."""
    gx, gw = _legendre(8)
    v, x = G["v"][l], G["c"][i]
    a = torch.linalg.vector_norm(v - x[:, None], dim=2).argmin(1)
    pick = lambda o: v[torch.arange(len(a), device=DEV), (a + o) % 3]
    A, B, C = pick(0), pick(1), pick(2)
    s = (0.5 * (gx + 1.0))[:, None, None]
    t = (0.5 * (gx + 1.0))[None, :, None]
    y = (A[:, None, None] + s * (B - A)[:, None, None] + s * t * (C - B)[:, None, None])
    wt = 0.25 * gw[:, None] * gw[None, :] * s[..., 0]
    val = _kernel(y - x[:, None, None], G["nrm"][l][:, None, None], k, op)
    return (val * wt).sum((1, 2)) * G["twice"][l] / (4 * math.pi)


def _matrices(xyz, tri, ks, op, near, rows=256):
    """Yields (r0, r1, [A(k)[r0:r1] for k in ks])."""
    G = _geometry(xyz, tri)
    n = len(G["c"])
    selfs = [_self(G, k, op) for k in ks]
    if near:
        ni, nl = _near_pairs(G)
    for r0 in range(0, n, rows):
        r1 = min(n, r0 + rows)
        d = G["q"][None] - G["c"][r0:r1, None, None]
        idx = torch.arange(r0, r1, device=DEV)
        if near:
            here = (ni >= r0) & (ni < r1)
            pi, pl = ni[here], nl[here]
        out = []
        for k, sf in zip(ks, selfs):
            A = (_kernel(d, G["nrm"][None, :, None], k, op) * G["w"]).sum(2) / (4 * math.pi)
            if near:
                for s in range(0, len(pi), 200000):
                    e = slice(s, s + 200000)
                    A[pi[e] - r0, pl[e]] = _near_values(G, pi[e], pl[e], k, op)
            A[idx - r0, idx] = sf[r0:r1]
            out.append(A)
        yield r0, r1, out


def _nodes(centre, a, b, N):
    th = math.pi * (2 * np.arange(N) + 1) / N
    return (centre + a * np.cos(th) + 1j * b * np.sin(th),
            (b * np.cos(th) + 1j * a * np.sin(th)) / N)


def _orthonormal(V):
    Q, R = torch.linalg.qr(V)
    return Q * torch.sgn(torch.diagonal(R))


def _project_exact(xyz, tri, V, z, w, op, near):
    n = len(tri)
    Y = torch.empty((len(z), n, V.shape[1]), dtype=torch.complex128, device=DEV)
    for r0, r1, As in _matrices(xyz, tri, [complex(k) for k in z], op, near,
                                rows=max(8, min(256, 400000 // n))):
        for j, A in enumerate(As):
            Y[j, r0:r1] = A @ V
    wt = torch.from_numpy(w).to(DEV)
    return wt[:, None, None] * (V.mH[None] @ Y), Y


def exact(case, seed):
    kind = case["kind"]
    if kind == "orth":
        return _orthonormal(_columns(seed, case["n"], case["nu"]))
    if kind == "batch":
        out = []
        for k, (m, axes, N, centre) in enumerate(_problems(case)):
            if (12.0 * m * m) ** 2 * N > 2e8:   # the larger bodies would take too long
                out.append(None)
                continue
            xyz, tri = _mesh("ell", m, axes)
            z, w = _nodes(centre, 0.8, 0.8, N)
            V = _columns(1000 * seed + k, len(tri), case["nu"])
            out.append(_project_exact(xyz, tri, V, z, w, OPERATOR["single"], 0)[0])
        return out
    xyz, tri = _mesh(case["shape"], case["size"])
    n = len(tri)
    if kind == "residual":
        if float(n) * n * case["m"] > 4e8:
            return None
        lam, X = _pairs(case, seed, n)
        R = torch.empty_like(X)
        for r0, r1, As in _matrices(xyz, tri, [complex(k) for k in lam], OPERATOR["single"], case["near"],
                                    rows=max(8, 400000 // n)):
            for c, A in enumerate(As):
                R[r0:r1, c] = A @ X[:, c]
        rel = torch.linalg.vector_norm(R, dim=0) / torch.linalg.vector_norm(X, dim=0)
        return rel.cpu().numpy(), R
    z, w = _nodes(case["centre"], case["a"], case["b"], case["N"])
    if kind == "step":
        if float(n) * n * case["N"] > 4e8:
            return None
        V = _orthonormal(_columns(seed, n, case["nu"]))
        B, Y = _project_exact(xyz, tri, V, z, w, OPERATOR[case["op"]], case["near"])
        return {"V": V, "B": B, "Y": Y} if case["av"] else {"V": V, "B": B}
    if kind == "improve":
        return _improve_exact(case, xyz, tri, _columns(seed, n, case["nu"]), z, w)
    return _solve_exact(case, xyz, tri)


def _improve_exact(case, xyz, tri, U, z, w):
    n, N, s = len(tri), len(z), _shift(case)
    if float(n) * n * N > 4e8:
        return None
    c = w / (z - s)
    ks = [complex(k) for k in z]
    rows = max(8, min(256, 400000 // n))
    S = torch.zeros((n, n), dtype=torch.complex128, device=DEV)
    v = torch.stack([U / (k - s) for k in ks])
    lu = None
    for _ in range(case["q"]):
        rhs = torch.zeros_like(U)
        for r0, r1, As in _matrices(xyz, tri, ks, OPERATOR["single"], 0, rows=rows):
            for j, A in enumerate(As):
                if lu is None:
                    S[r0:r1] += c[j] * A
                rhs[r0:r1] += c[j] * (A @ v[j])
        if lu is None:
            lu = torch.linalg.lu_factor(S)
        u = torch.linalg.lu_solve(*lu, rhs)
        v = torch.stack([(v[j] - u) / (ks[j] - s) for j in range(N)])
        norm = torch.linalg.vector_norm(v, dim=(0, 1))
        v, u = v / norm, u / norm
    return u


def _solve_exact(case, xyz, tri):
    """Eigenpairs inside the ellipse: contour moments of A(z)^-1, then Newton's method."""
    op, n = OPERATOR["single"], len(tri)

    def dense(ks):
        out = [torch.empty((n, n), dtype=torch.complex128, device=DEV) for _ in ks]
        for r0, r1, As in _matrices(xyz, tri, ks, op, 0, rows=max(8, 400000 // n)):
            for M, A in zip(out, As):
                M[r0:r1] = A
        return out

    z, w = _nodes(case["centre"], case["a"], case["b"], 64)
    P = _gauss(7, n, 24)
    A0, A1 = torch.zeros_like(P), torch.zeros_like(P)
    for k, wt in zip(z, w):
        X = torch.linalg.solve(dense([complex(k)])[0], P)
        A0 += complex(wt) * X
        A1 += complex(wt * (k - case["centre"])) * X
    U, s, Wh = torch.linalg.svd(A0, full_matrices=False)
    r = int((s > 1e-8 * s[0]).sum())
    if r == 0:
        return None
    U, s, W = U[:, :r], s[:r], Wh[:r].mH
    ev, Q = torch.linalg.eig((U.mH @ A1 @ W) / s)
    lam = ev.cpu().numpy() + case["centre"]
    keep = [i for i in range(r) if ((lam[i].real - case["centre"]) / case["a"]) ** 2
            + (lam[i].imag / case["b"]) ** 2 < 1.0]
    keep.sort(key=lambda i: lam[i].real)
    probe = _probe(n)
    ls, xs = [], []
    for i in keep:
        k, x = complex(lam[i]), U @ Q[:, i]
        x = x / (probe.conj() @ x)
        for _ in range(6):
            A, Ap, Am = dense([k, k + 1e-4, k - 1e-4])
            J = torch.zeros((n + 1, n + 1), dtype=torch.complex128, device=DEV)
            J[:n, :n], J[:n, n], J[n, :n] = A, (Ap @ x - Am @ x) / 2e-4, probe.conj()
            rhs = torch.cat([A @ x, torch.zeros(1, dtype=torch.complex128, device=DEV)])
            step = torch.linalg.solve(J, rhs)
            x, k = x - step[:n], k - complex(step[n].item())
        ls.append(k)
        xs.append(x)
    return {"lam": np.array(ls), "X": torch.stack(xs, 1)}
