"""The work a user of this library has it do, as a list of timed cases.

Each case is one pass through the public entry points: an operator applied
to a field (BP1.0, BP3.5, BP3.0, BP1.0 and BP3.0 in one pass) in one of its
precisions, the geometric factors of a mesh, a batch of meshes of mixed
degree, a Helmholtz solve, or a round of solve requests through the server.
Meshes are jittered boxes of trilinear hexahedra of the unit cube, fields
are U[-1, 1] per node or a smooth product of sines, as in the repository's
tests and benchmark.  `draw` gives more cases over the same ranges (degree 1
to 15, box sizes that are rarely round numbers).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1711_00903_gb300 as fem

LAMBDA = 1.0


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest call in use: the mass matvec of the paper's 512-element
        # mesh, a few microseconds, resident in L2
        {"name": "mass_n3_small", "kind": "mass", "N": 3, "nx": 8, "ny": 8, "nz": 8, "field": "random"},
        # setup of a mesh: the geometric factors of all three operators
        {"name": "factors_n7", "kind": "factors", "N": 7, "nx": 32, "ny": 32, "nz": 32},
        # the collocated Helmholtz matvec of the benchmark mesh
        {"name": "poisson_n7", "kind": "poisson", "prec": "f64", "N": 7, "nx": 32, "ny": 32, "nz": 32, "field": "random"},
        # the mass and the dealiased Helmholtz matvec of one field, as a time
        # step with a mass term applies them, on a smooth field
        {"name": "mass_dealiased_n7", "kind": "both", "N": 7, "nx": 32, "ny": 32, "nz": 32, "field": "smooth"},
        # mass matvec at high, even degree (odd line lengths), odd element count
        {"name": "mass_n12", "kind": "mass", "N": 12, "nx": 17, "ny": 17, "nz": 17, "field": "random"},
        # dealiased matvec at low degree, ragged element count
        {"name": "dealiased_n4", "kind": "dealiased", "prec": "f64", "N": 4, "nx": 23, "ny": 21, "nz": 19, "field": "random"},
        # the highest degree the library takes, few elements
        {"name": "poisson_n15", "kind": "poisson", "prec": "f64", "N": 15, "nx": 13, "ny": 13, "nz": 13, "field": "smooth"},
        # single-precision operators, as an FP32 code or an inner solver calls them
        {"name": "poisson_f32_n10", "kind": "poisson", "prec": "f32", "N": 10, "nx": 25, "ny": 25, "nz": 25, "field": "random"},
        {"name": "dealiased_f16_n7", "kind": "dealiased", "prec": "f16", "N": 7, "nx": 32, "ny": 32, "nz": 32, "field": "random"},
        # a Helmholtz solve in the mode the library recommends (FP64 defect
        # correction around FP16 factors), to a tight residual
        {"name": "solve_mixed16_n7", "kind": "solve", "op": "poisson", "mode": "mixed16", "N": 7, "nx": 16, "ny": 16, "nz": 16},
        # many independent meshes of mixed degree in one launch
        {"name": "batch_24", "kind": "batch", "meshes": 24, "nmin": 2, "nmax": 10, "emax": 4096},
        # a round of solve requests from host memory, FP64 and mixed
        {"name": "serve_6", "kind": "serve", "requests": 6, "nmin": 3, "nmax": 9, "emax": 1728},
    ]


MOST_DOFS = 32768 * 512  # of the largest listed matvec


def _draw_box(rng, lo, hi):
    """Box sizes with about lo..hi elements in all, log-uniform."""
    e = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nx = max(1, round(e ** (1 / 3) * rng.uniform(0.7, 1.4)))
    ny = max(1, round(e ** (1 / 3) * rng.uniform(0.7, 1.4)))
    return nx, ny, max(1, min(int(hi // (nx * ny)), round(e / (nx * ny))))


def draw(rng):
    kind = rng.choice(["mass", "poisson", "poisson", "dealiased", "dealiased", "both", "factors", "solve", "batch", "serve"])
    if kind == "batch":
        return {"kind": kind, "meshes": rng.randint(4, 24), "nmin": rng.randint(1, 4), "nmax": rng.randint(5, 10),
                "emax": rng.randint(256, 4096)}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(2, 6), "nmin": rng.randint(3, 5), "nmax": rng.randint(6, 9),
                "emax": rng.randint(600, 1728)}
    if kind == "solve":
        N = rng.randint(2, 9)
        nx, ny, nz = _draw_box(rng, 64, 4096 * 512 / (N + 1) ** 3)
        return {"kind": kind, "op": rng.choice(["poisson", "dealiased"]), "mode": rng.choice(["fp64", "mixed", "mixed16"]),
                "N": N, "nx": min(nx, 16), "ny": min(ny, 16), "nz": min(nz, 16)}
    N = rng.randint(1, 15)
    points = (N + 2) ** 3 if kind in ("dealiased", "both", "factors") else (N + 1) ** 3
    nx, ny, nz = _draw_box(rng, 64, min(40000, MOST_DOFS / points))
    c = {"kind": kind, "N": N, "nx": nx, "ny": ny, "nz": nz}
    if kind in ("poisson", "dealiased"):
        c["prec"] = rng.choice(["f64", "f64", "f32", "f16"])
    if kind != "factors":
        c["field"] = rng.choice(["random", "smooth"])
    return c


# --------------------------------------------------------------- the inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _mesh(nx, ny, nz, seed):
    """Vertices (E, 8, 3) of a box mesh of the unit cube whose interior
    vertices are moved by up to a tenth of the spacing."""
    f = dict(dtype=torch.float64, device="cuda")
    z, y, x = torch.meshgrid(torch.linspace(0, 1, nz + 1, **f), torch.linspace(0, 1, ny + 1, **f),
                             torch.linspace(0, 1, nx + 1, **f), indexing="ij")
    P = torch.stack([x, y, z], -1)
    d = 2 * torch.rand(P.shape, generator=_gen(seed), **f) - 1
    d *= 0.1 * torch.tensor([1 / nx, 1 / ny, 1 / nz], **f)
    P[1:-1, 1:-1, 1:-1] += d[1:-1, 1:-1, 1:-1]
    corners = [P[t:nz + t, s:ny + s, r:nx + r] for t in (0, 1) for s in (0, 1) for r in (0, 1)]
    return torch.stack(corners, -2).reshape(nx * ny * nz, 8, 3).contiguous()


def _rule(N):
    """GLL nodes and weights, Gauss nodes and weights (numpy, 64 bits)."""
    n = N + 1
    L = np.polynomial.legendre.Legendre.basis(N)
    r = np.concatenate([[-1.0], np.sort(L.deriv().roots().real), [1.0]])
    c = np.zeros(N + 1)
    c[N] = 1.0
    for _ in range(3):  # Newton steps on P_N' at the interior nodes
        x = r[1:-1]
        p, dp = np.polynomial.legendre.legval(x, c), np.polynomial.legendre.legval(x, np.polynomial.legendre.legder(c))
        r[1:-1] = x - dp * (1 - x * x) / (2 * x * dp - N * n * p)
    r = 0.5 * (r - r[::-1])
    w = 2.0 / (N * n * np.polynomial.legendre.legval(r, c) ** 2)
    return r, w, *np.polynomial.legendre.leggauss(N + 2)


def _lagrange(x, at):
    """Values of the Lagrange basis of the nodes x at the points `at`."""
    V = np.ones((len(at), len(x)))
    for i in range(len(x)):
        for j in range(len(x)):
            if j != i:
                V[:, i] *= (at - x[j]) / (x[i] - x[j])
    return V


def _derivative(x):
    """Differentiation matrix of the nodes x."""
    D = np.zeros((len(x), len(x)))
    c = np.array([np.prod(x[i] - np.delete(x, i)) for i in range(len(x))])
    for a in range(len(x)):
        for i in range(len(x)):
            if a != i:
                D[a, i] = c[a] / (c[i] * (x[a] - x[i]))
        D[a, a] = -D[a].sum()
    return D


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _coordinates(verts, x):
    """Coordinates (E, q, q, q, 3) of the trilinear elements at the tensor points x, [t][s][r]."""
    x = _cuda(x)
    h = torch.stack([(1 - x) / 2, (1 + x) / 2], -1)  # (q, 2)
    v = verts.reshape(-1, 2, 2, 2, 3)
    return torch.einsum("etsrd,kt,js,ir->ekjid", v, h, h, h)


def _field(case, verts, seed):
    E, n = verts.shape[0], case["N"] + 1
    if case.get("field") == "random":
        return 2 * torch.rand(E, n ** 3, generator=_gen(seed + 1000003), dtype=torch.float64, device="cuda") - 1
    return _smooth(verts, case["N"], seed)


def _smooth(verts, N, seed):
    """Nodal values of a product of sines (zero on the boundary of the cube),
    its amplitude and wave numbers from the seed."""
    kx, ky, kz = 1 + seed % 3, 1 + (seed // 3) % 2, 1 + (seed // 6) % 2
    X = _coordinates(verts, _rule(N)[0])
    u = (1 + (seed % 17) / 16) * torch.sin(kx * math.pi * X[..., 0]) * torch.sin(ky * math.pi * X[..., 1]) * torch.sin(kz * math.pi * X[..., 2])
    return u.reshape(verts.shape[0], -1).contiguous()


def _gauss(kind):
    return kind in ("dealiased", "both")


def _draw_sizes(case, seed_of, count):
    """(N, nx, ny, nz) of the meshes of a batch or of the requests of a
    serving round: the same for every seed, so that a case has one size."""
    r = np.random.RandomState(seed_of)
    got = []
    for _ in range(count):
        N = int(r.randint(case["nmin"], case["nmax"] + 1))
        e = math.exp(r.uniform(math.log(64), math.log(case["emax"])))
        a = max(1, int(round(e ** (1 / 3))))
        b = max(1, int(round(math.sqrt(e / a))))
        got.append((N, a, b, max(1, int(e // (a * b)))))
    return got


def _factors(basis, verts, op):
    return fem.fem_mesh_geofacs(basis, fem.FEM_GEO_BP30 if op == "dealiased" else fem.FEM_GEO_BP35, verts)


def _apply(op):
    return fem.fem_bp30_apply if op == "dealiased" else fem.fem_bp35_apply


_OPS = {"poisson": fem.FEM_OP_BP35, "dealiased": fem.FEM_OP_BP30}
_MODES = {"fp64": fem.FEM_PCG_FP64, "mixed": fem.FEM_PCG_MIXED, "mixed16": fem.FEM_PCG_MIXED16}
_PRECS = {"f64": fem.FEM_PREC_F64, "f32": fem.FEM_PREC_F32, "f16": fem.FEM_PREC_F16G}


def _half_scale(G):
    """The power of two that brings the largest factor just below 2^14."""
    return 2.0 ** (14 - math.frexp(float(G.abs().max()))[1])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        basis, items = {}, []
        for k, (N, nx, ny, nz) in enumerate(_draw_sizes(case, 11, case["meshes"])):
            if N not in basis:
                basis[N] = fem.fem_basis_setup(N)
            b = basis[N]
            verts = _mesh(nx, ny, nz, seed + k)
            q = _field({"N": N, "field": "random"}, verts, seed + k)
            op = "dealiased" if k % 2 else "poisson"
            items.append((_OPS[op], b, _factors(b, verts, op), LAMBDA, q, torch.empty_like(q)))
        batch = fem.fem_batch_create(items)
        # a configuration kept from an earlier run of the tuner
        batch.config = {"threads": 512, "group": 2, "order": 0, "layout": 0}
        return {"kind": kind, "batch": batch, "outs": [i[5] for i in items]}
    if kind == "serve":
        reqs = []
        for k, (N, nx, ny, nz) in enumerate(_draw_sizes(case, 12, case["requests"])):
            b, verts = fem.fem_basis_setup(N), _mesh(nx, ny, nz, seed + k)
            op = "dealiased" if k % 3 == 1 else "poisson"
            rhs = _apply(op)(b, _factors(b, verts, op), LAMBDA, _smooth(verts, N, seed + k))
            reqs.append((_OPS[op], N, verts.cpu().numpy(), rhs.cpu().numpy(), LAMBDA, fem.FEM_PCG_MIXED16 if k % 2 else fem.FEM_PCG_FP64, 1e-12))
        return {"kind": kind, "server": fem.Server(), "requests": reqs}
    b = fem.fem_basis_setup(case["N"])
    verts = _mesh(case["nx"], case["ny"], case["nz"], seed)
    E = verts.shape[0]
    s = {"kind": kind, "basis": b}
    if kind == "factors":
        empty = lambda k: torch.empty(fem.geo_shape(b, k, E), dtype=torch.float64, device="cuda")  # noqa: E731
        return s | {"verts": verts, "wJ": empty(fem.FEM_GEO_BP1), "G35": empty(fem.FEM_GEO_BP35), "G30": empty(fem.FEM_GEO_BP30)}
    if kind == "solve":
        G = _factors(b, verts, case["op"])
        rhs = _apply(case["op"])(b, G, LAMBDA, _smooth(verts, case["N"], seed))
        return s | {"solver": fem.fem_pcg_create(b, G, LAMBDA, _MODES[case["mode"]], op=_OPS[case["op"]]), "rhs": rhs}
    q = _field(case, verts, seed)
    if kind == "mass":
        return s | {"wJ": fem.fem_mesh_geofacs(b, fem.FEM_GEO_BP1, verts), "q": q, "out": torch.empty_like(q)}
    G = fem.fem_mesh_geofacs(b, fem.FEM_GEO_BP30 if _gauss(kind) else fem.FEM_GEO_BP35, verts)
    if kind == "both":
        return s | {"G": G, "q": q, "out_m": torch.empty_like(q), "out_a": torch.empty_like(q)}
    ginv = None
    if case["prec"] != "f64":
        q = q.float()
        if case["prec"] == "f16":
            scale = _half_scale(G)
            G, ginv = (G * scale).half(), torch.tensor([1 / scale], dtype=torch.float64, device="cuda")
        else:
            G = G.float()
    return s | {"prec": _PRECS[case["prec"]], "G": G, "ginv": ginv, "q": q, "out": torch.empty_like(q)}


# ----------------------------------------------------------------- one pass

def run(s):
    kind = s["kind"]
    if kind == "mass":
        return fem.fem_bp1_apply(s["basis"], s["wJ"], s["q"], out=s["out"])
    if kind == "poisson":
        return fem.fem_bp35_apply_ex(s["basis"], s["prec"], s["G"], LAMBDA, s["q"], ginv=s["ginv"], out=s["out"])
    if kind == "dealiased":
        return fem.fem_bp30_apply_ex(s["basis"], s["prec"], s["G"], LAMBDA, s["q"], ginv=s["ginv"], out=s["out"])
    if kind == "both":
        return fem.fem_bp1_bp30_apply(s["basis"], s["G"], LAMBDA, s["q"], out_m=s["out_m"], out_a=s["out_a"])
    if kind == "factors":
        return fem.fem_mesh_geofacs_set(s["basis"], s["verts"], wJ=s["wJ"], G35=s["G35"], G30=s["G30"])
    if kind == "solve":
        return s["solver"].solve(s["rhs"], tol=1e-12)[0]
    if kind == "batch":
        s["batch"].apply()
        return s["outs"]
    ids = [s["server"].submit(*r) for r in s["requests"]]
    s["server"].drain()
    for rid, _ in ids:
        s["server"].forget(rid)
    return [x for _, x in ids]


# --------------------------------------------------- what a pass cannot skip

def _matvec_work(kind, N, E, word=8, gword=8):
    """Bytes (field and factors in, result out) and flops (2 per multiply-add
    of the sum-factorised contractions) of one matvec."""
    n, m = N + 1, N + 2
    interp = 4 * (m * n ** 3 + m * m * n * n + m ** 3 * n)
    if kind == "mass":
        return E * (2 * n ** 3 * word + m ** 3 * gword), E * (interp + m ** 3)
    if kind == "poisson":
        return E * n ** 3 * (2 * word + 7 * gword), E * (12 * n ** 4 + 18 * n ** 3)
    if kind == "both":
        return E * (3 * n ** 3 * word + 7 * m ** 3 * gword), E * (1.5 * interp + m ** 3 + 12 * m ** 4 + 18 * m ** 3)
    return E * (2 * n ** 3 * word + 7 * m ** 3 * gword), E * (interp + 12 * m ** 4 + 18 * m ** 3)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        pairs = [_matvec_work("dealiased" if k % 2 else "poisson", N, nx * ny * nz)
                 for k, (N, nx, ny, nz) in enumerate(_draw_sizes(case, 11, case["meshes"]))]
        return {"bytes": sum(p[0] for p in pairs), "flops": sum(p[1] for p in pairs)}
    if kind == "serve":  # the requests in, the solutions out; one matvec and its factors each
        got = {"bytes": 0, "flops": 0}
        for k, (N, nx, ny, nz) in enumerate(_draw_sizes(case, 12, case["requests"])):
            E, n = nx * ny * nz, N + 1
            got["bytes"] += E * (24 + 2 * n ** 3) * 8
            got["flops"] += _matvec_work("dealiased" if k % 3 == 1 else "poisson", N, E)[1]
        return got
    E, N = case["nx"] * case["ny"] * case["nz"], case["N"]
    n, m = N + 1, N + 2
    if kind == "factors":
        return {"bytes": E * 8 * (24 + 7 * n ** 3 + 8 * m ** 3), "flops": E * 76 * (n ** 3 + m ** 3)}
    if kind == "solve":  # the factors and the right-hand side in, the solution out, one matvec
        b, f = _matvec_work(case["op"], N, E)
        return {"bytes": b, "flops": f}
    word = 8 if case.get("prec", "f64") == "f64" else 4
    b, f = _matvec_work(kind, N, E, word, {"f64": 8, "f32": 4, "f16": 2}[case.get("prec", "f64")])
    return {"bytes": b, "flops": f}


# ----------------------------------------------- the same in plain 64 bits

def _exact_factors(verts, x, w):
    """(Grr, Grs, Grt, Gss, Gst, Gtt, wJ) as (E, 7, q^3), point r fastest."""
    h = np.stack([(1 - x) / 2, (1 + x) / 2], -1)
    d = np.stack([-0.5 * np.ones_like(x), 0.5 * np.ones_like(x)], -1)
    H, Dh, v = _cuda(h), _cuda(d), verts.reshape(-1, 2, 2, 2, 3)
    J = torch.stack([torch.einsum("etsrd,kt,js,ir->ekjid", v, *m) for m in ((H, H, Dh), (H, Dh, H), (Dh, H, H))], -1)
    xr, xs, xt = J.unbind(-1)
    C = torch.stack([torch.linalg.cross(xs, xt), torch.linalg.cross(xt, xr), torch.linalg.cross(xr, xs)], -2)
    det = (xr * C[..., 0, :]).sum(-1)
    W = _cuda(w)
    W = W[:, None, None] * W[:, None] * W
    G = torch.einsum("ekjiad,ekjibd->abekji", C, C) * (W / det)
    planes = [G[0, 0], G[0, 1], G[0, 2], G[1, 1], G[1, 2], G[2, 2], W * det]
    return torch.stack(planes, 1).reshape(verts.shape[0], 7, -1)


def _along(A, u):
    """A applied along r, s and t of u (E, t, s, r)."""
    return torch.einsum("ai,ekji->ekja", A, u), torch.einsum("bj,ekji->ekbi", A, u), torch.einsum("ck,ekji->ecji", A, u)


def _all3(A, u):
    return torch.einsum("ck,ekba->ecba", A, torch.einsum("bj,ekja->ekba", A, torch.einsum("ai,ekji->ekja", A, u)))


def _stiff(D, G, u):
    """D^T G D u + LAMBDA wJ u at the points of G."""
    q = u.shape[-1]
    g = G.reshape(-1, 7, q, q, q)
    ur, us, ut = _along(D, u)
    wr = g[:, 0] * ur + g[:, 1] * us + g[:, 2] * ut
    ws = g[:, 1] * ur + g[:, 3] * us + g[:, 4] * ut
    wt = g[:, 2] * ur + g[:, 4] * us + g[:, 5] * ut
    T = D.T.contiguous()
    return _along(T, wr)[0] + _along(T, ws)[1] + _along(T, wt)[2] + LAMBDA * g[:, 6] * u


def _round_factors(G, prec):
    if prec == "f32":
        return G.float().double()
    if prec == "f16":
        s = _half_scale(G)
        return (G * s).half().double() / s
    return G


def _exact_matvec(kind, prec, N, verts, q):
    """The operator on every element, a few thousand elements at a time."""
    r, w, rt, wt = _rule(N)
    n, E = N + 1, verts.shape[0]
    I = _cuda(_lagrange(r, rt))
    D, Dt = _cuda(_derivative(r)), _cuda(_derivative(rt))
    x, wx = (r, w) if kind == "poisson" else (rt, wt)
    out = torch.empty(E, n ** 3, dtype=torch.float64, device="cuda")
    out_m = torch.empty_like(out)
    top = None
    if prec == "f16":  # the scale of the halves is that of the whole mesh
        top = max(float(_exact_factors(verts[e:e + 2048], x, wx).abs().max()) for e in range(0, E, 2048))
    for e in range(0, E, 2048):
        G = _exact_factors(verts[e:e + 2048], x, wx)
        u = q[e:e + 2048].double().reshape(-1, n, n, n)
        if prec == "f16":
            s = 2.0 ** (14 - math.frexp(top)[1])
            G = (G * s).half().double() / s
        else:
            G = _round_factors(G, prec)
        if kind == "poisson":
            out[e:e + 2048] = _stiff(D, G, u).reshape(-1, n ** 3)
            continue
        ug, IT = _all3(I, u), I.T.contiguous()
        if kind in ("mass", "both"):
            out_m[e:e + 2048] = _all3(IT, G[:, 6].reshape(ug.shape) * ug).reshape(-1, n ** 3)
        if kind in ("dealiased", "both"):
            out[e:e + 2048] = _all3(IT, _stiff(Dt, G, ug)).reshape(-1, n ** 3)
    return out_m if kind == "mass" else (out_m, out) if kind == "both" else out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        got = []
        for k, (N, nx, ny, nz) in enumerate(_draw_sizes(case, 11, case["meshes"])):
            verts = _mesh(nx, ny, nz, seed + k)
            q = _field({"N": N, "field": "random"}, verts, seed + k)
            got.append(_exact_matvec("dealiased" if k % 2 else "poisson", "f64", N, verts, q))
        return got
    if kind == "serve":  # the right-hand sides are A u: the solutions are u
        return [_smooth(_mesh(nx, ny, nz, seed + k), N, seed + k).cpu().numpy()
                for k, (N, nx, ny, nz) in enumerate(_draw_sizes(case, 12, case["requests"]))]
    N = case["N"]
    verts = _mesh(case["nx"], case["ny"], case["nz"], seed)
    if kind == "factors":
        r, w, rt, wt = _rule(N)
        parts = [(_exact_factors(verts[e:e + 4096], r, w), _exact_factors(verts[e:e + 4096], rt, wt))
                 for e in range(0, verts.shape[0], 4096)]
        G35, G30 = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
        return G30[:, 6].contiguous(), G35, G30
    if kind == "solve":
        return _smooth(verts, N, seed)
    q = _field(case, verts, seed)
    if case.get("prec", "f64") != "f64":
        q = q.float()
    return _exact_matvec(kind, case.get("prec", "f64"), N, verts, q)
