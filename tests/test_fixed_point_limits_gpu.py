"""Where 64-bit fixed point, scaled per element, would hold fewer digits than
FP64 arithmetic: elements with nearly parallel edges (geometric factors) and
flat elements (operators).  Against references in extended precision
(np.longdouble: 64 bits of mantissa or more)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble
U = 2.0 ** -53
BOX = np.array([[(c >> d) & 1 for d in range(3)] for c in range(8)], dtype=float)
PAIRS = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


def _fem():
    import paper_1711_00903_gb300 as fem
    return fem


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _rotation(rng):
    r = np.linalg.qr(rng.standard_normal((3, 3)))[0]
    return r * np.sign(np.linalg.det(r))


def _columns(cols):
    """The parallelepiped with these edge vectors, right-handed."""
    cols = np.asarray(cols)
    return BOX @ (cols if np.linalg.det(cols) > 0 else cols[[1, 0, 2]])


def _parallel_elements():
    """Rotated boxes sheared by 10 to 1e5, columns (1, +-a, +-a), two columns
    that differ by 1e-3 to 1e-7, rotated flat elements."""
    rng = np.random.default_rng(17)
    v = []
    for s in (3, 10, 100, 1e3, 1e4, 1e5):
        for _ in range(3):
            v.append(BOX @ np.array([[1, s, 0], [0, 1, 0], [0, 0, 1.0]]).T @ _rotation(rng).T)
    for a in (0.3, 0.1, 0.04, 0.02, 0.012):
        for _ in range(4):
            v.append(_columns([[1, *(rng.choice([-1, 1], 2) * a * rng.uniform(0.7, 1.3, 2))] for _ in range(3)]))
    for e in (1e-3, 1e-6, 1e-7):
        for _ in range(3):
            c = rng.uniform(0.5, 1, 3)
            v.append(_columns([c, c + e * rng.uniform(-1, 1, 3), rng.uniform(-1, 1, 3)]))
    for a in (10, 1e3):
        v.append((BOX + 0.1 * rng.uniform(-1, 1, (8, 3))) * [1, 1, 1 / a] @ _rotation(rng).T)
    return np.ascontiguousarray(np.array(v))


def _factors(verts, x, w):
    """Factors and, with u = 2^-53, the first-order bound of an evaluation in
    FP64: 8 u per column component (edge differences and bilinear form, on
    absolute values), 2 u per product of a cofactor, 6 u for the determinant,
    the quotient and the weights, 4 u for the sum of three products."""
    x, w = x.astype(LD), w.astype(LD)
    h, d = np.stack([(1 - x) / 2, (1 + x) / 2], -1), np.stack([0 * x - 0.5, 0 * x + 0.5], -1)
    v = verts.astype(LD).reshape(-1, 2, 2, 2, 3)

    def columns(v, d):
        return [np.einsum("etsrd,kt,js,ir->ekjid", v, *m) for m in ((h, h, d), (h, d, h), (d, h, h))]

    X = columns(v, d)
    e = [np.abs(np.diff(v, axis=a)).sum((1, 2, 3)) for a in (3, 2, 1)]  # |edges| along r, s, t
    A = [0.5 * a[:, None, None, None, :] + 0 * X[0] for a in e]         # of the columns' components
    cross = lambda a, b: np.stack([a[..., 1] * b[..., 2] + a[..., 2] * b[..., 1],  # noqa: E731
                                   a[..., 2] * b[..., 0] + a[..., 0] * b[..., 2],
                                   a[..., 0] * b[..., 1] + a[..., 1] * b[..., 0]], -1)
    nxt = ((1, 2), (2, 0), (0, 1))
    C = [np.cross(X[i], X[j]) for i, j in nxt]
    dC = [U * (8 * (cross(A[i], abs(X[j])) + cross(abs(X[i]), A[j])) + 2 * cross(abs(X[i]), abs(X[j]))) for i, j in nxt]
    det = (X[0] * C[0]).sum(-1)
    ddet = (abs(X[0]) * dC[0] + 8 * U * A[0] * abs(C[0]) + 4 * U * abs(X[0] * C[0])).sum(-1)
    W = w[:, None, None] * w[:, None] * w
    G, bar = [], []
    for a, b in PAIRS:
        g = (C[a] * C[b]).sum(-1) * W / det
        G.append(g)
        bar.append(W / abs(det) * (dC[a] * abs(C[b]) + abs(C[a]) * dC[b] + 4 * U * abs(C[a] * C[b])).sum(-1)
                   + abs(g) * (ddet / abs(det) + 6 * U))
    G.append(W * det)
    bar.append(W * ddet + 6 * U * abs(G[-1]))
    shape = (verts.shape[0], 7, -1)
    return np.stack(G, 1).reshape(shape), np.stack(bar, 1).reshape(shape)


@pytest.mark.parametrize("N", [1, 2, 7, 15])
def test_factors_of_nearly_parallel_edges(N):
    """Each factor within the error that an evaluation in FP64 may have."""
    fem = _fem()
    b, verts = fem.fem_basis_setup(N), _parallel_elements()
    t = fem.fem_basis_host_tables(N)
    for kind, x, w in ((fem.FEM_GEO_BP35, "r", "w"), (fem.FEM_GEO_BP30, "rt", "wt")):
        got = fem.fem_mesh_geofacs(b, kind, _dev(verts)).cpu().numpy()
        ref, bar = _factors(verts, t[x], t[w])
        assert np.all(abs(got - ref) <= bar)
    wj = fem.fem_mesh_geofacs(b, fem.FEM_GEO_BP1, _dev(verts)).cpu().numpy()
    np.testing.assert_array_equal(wj, got[:, 6])


# ------------------------------------------------------------ flat elements

def _along(A, u, axis):
    return np.moveaxis(np.tensordot(A, u, axes=(1, axis)), 0, axis)


def _all3(A, u):
    return _along(A, _along(A, _along(A, u, 3), 2), 1)


def _symmetric(A, s):
    A = A.astype(LD)
    return (A + s * A[::-1, ::-1]) / 2


def _stiff(T, G, u, d):
    """T G d + 0.37 wJ u of the derivatives d (along r, s, t)."""
    g = G.reshape(-1, 7, *u.shape[1:])
    w = [sum(g[:, k] * x for k, x in zip(row, d)) for row in ((0, 1, 2), (1, 3, 4), (2, 4, 5))]
    return _along(T, w[0], 3) + _along(T, w[1], 2) + _along(T, w[2], 1) + LD(0.37) * g[:, 6] * u


def _folded(A):
    """Absolute values of an operator as even-odd folded lines add them up."""
    return abs(A) + abs(A[:, ::-1])


def _flat_reference(op, t, G, q, exact):
    """The operator and the bound 2 (1.5 n + 17) 2^-53 |D^T| |G| |d| of FP64
    lines folded even-odd (n / 2 + 3 roundings a contraction, 8 in the chain
    rule and the sums), with |d| the derivatives themselves along the directions
    in `exact` (FP64 takes them without an error of the field's size) and |D|
    |q| along the others."""
    n = t["D"].shape[0]
    I, D = _symmetric(t["I"], 1), _symmetric(t["D" if op == "bp35" else "Dt"], -1)
    u, G = q.astype(LD).reshape(-1, n, n, n), G.astype(LD)
    if op == "bp30":
        u = _all3(I, u)
    d = [_along(D, u, a) for a in (3, 2, 1)]
    m = [abs(x) if a in exact else _along(_folded(D), abs(u), 3 - a) for a, x in enumerate(d)]
    ref, bar = _stiff(D.T, G, u, d), _stiff(_folded(D.T), abs(G), abs(u), m)
    if op == "bp30":
        ref, bar = _all3(I.T.copy(), ref), _all3(_folded(I.T), bar)
    chain = 1.5 if op == "bp35" else 4.5
    return ref.reshape(q.shape), (2 * (chain * n + 17) * U * bar).reshape(q.shape)


def _flat_fields(rng, n, thin):
    """Constant across the thin direction; constant; with a slope of 1 to 1e-9
    across the thin direction; random; zero but for a face."""
    axis = 3 - thin
    shape = [8, n, n, n]
    shape[axis] = 1
    flat = np.broadcast_to(rng.uniform(-1, 1, shape), (8, n, n, n))
    x = np.linspace(0, 1, n).reshape([-1 if a == axis else 1 for a in range(4)])
    q = flat + np.array([0, 0, 1, 1e-3, 1e-6, 1e-9, 0, 0]).reshape(8, 1, 1, 1) * x
    q[1] = 0.7
    q[6] = rng.uniform(-1, 1, (n, n, n))
    q[7] = 0.0
    q[7, 0] = rng.uniform(-1, 1, (n, n))
    return np.ascontiguousarray(q.reshape(8, -1))


@pytest.mark.parametrize("op,N", [("bp35", 1), ("bp35", 2), ("bp35", 3), ("bp35", 7), ("bp30", 1), ("bp30", 2),
                                  ("bp30", 7)])
@pytest.mark.parametrize("thin", [0, 1, 2])
def test_flat_elements_keep_the_small_factors(op, N, thin):
    """Each node within the error that an evaluation in FP64 may have, on
    axis-aligned and slightly skewed elements of aspect 1 to 1e6 (and a long
    one), where the smallest factors are aspect^-2 of the largest.  FP64 takes
    the derivative of a constant line without an error at two and three points
    (of any line at two)."""
    fem, rng = _fem(), np.random.default_rng(100 * N + thin)
    b = fem.fem_basis_setup(N)
    t = fem.fem_basis_host_tables(N)
    kind, apply = (fem.FEM_GEO_BP35, fem.fem_bp35_apply) if op == "bp35" else (fem.FEM_GEO_BP30, fem.fem_bp30_apply)
    for aspect in (1, 10, 100, 1e3, 1e4, 1e6, 1e9, 1e-3):
        scale = np.ones(3)
        scale[thin] = 1 / aspect
        for skew in (0, 0.05):
            verts = np.ascontiguousarray((BOX + skew * rng.uniform(-1, 1, (8, 8, 3))) * scale)
            q = _flat_fields(rng, N + 1, thin)
            G = fem.fem_mesh_geofacs(b, kind, _dev(verts))
            got = apply(b, G, 0.37, _dev(q)).cpu().numpy()
            for rows, exact in ((slice(0, 2), (thin,)), (slice(2, 8), ())):
                if op == "bp35" and N == 1:
                    exact = (0, 1, 2)
                elif N > (2 if op == "bp35" else 1):
                    exact = ()
                ref, bar = _flat_reference(op, t, G.cpu().numpy()[rows], q[rows], exact)
                assert np.all(abs(got[rows] - ref) <= bar)


# ------------------------------------------------- elements that stay in FP64

def _fastest(f):
    """Least time of ten calls, us."""
    import torch
    f()
    t = []
    for _ in range(10):
        a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        z.record()
        z.synchronize()
        t.append(a.elapsed_time(z) * 1e3)
    return min(t)


def _fp64_rate():
    """FP64 instructions (of a lane) per us, measured."""
    probe, flops = _fem().fem_fma_probe(2000)
    return flops / 2 / _fastest(lambda: _fem().fem_fma_probe(2000, out=probe))


def _left_handed(N, n):
    import fem_synth
    return _dev(fem_synth.box_mesh(n, n, n, seed=N)[:, [1, 0, 3, 2, 5, 4, 7, 6]])


@pytest.mark.parametrize("op", ["bp1", "bp35", "bp30", "bp1_bp30"])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_a_mesh_of_fp64_elements_runs_at_the_fp64_rate(op, N):
    """Every element of a left-handed mesh is left to FP64.  Twice the time that
    the even-odd lines' instructions take at the FP64 rate measured here, and
    the launch: the pipe is 0.8 to 0.9 busy in kernels made for it, and up to a
    quarter of the lanes idle where n^2 or m^2 lines do not fill warps."""
    import torch

    import bench
    fem = _fem()
    verts = _left_handed(N, 32)
    E = verts.shape[0]
    b = fem.fem_basis_setup(N)
    kind = {"bp1": fem.FEM_GEO_BP1, "bp35": fem.FEM_GEO_BP35}.get(op, fem.FEM_GEO_BP30)
    G = fem.fem_mesh_geofacs(b, kind, verts)
    q = torch.rand(E, (N + 1) ** 3, dtype=torch.float64, device="cuda")
    out, out_m = torch.empty_like(q), torch.empty_like(q)
    call = {"bp1": lambda: fem.fem_bp1_apply(b, G, q, out=out), "bp35": lambda: fem.fem_bp35_apply(b, G, 1.0, q, out=out),
            "bp30": lambda: fem.fem_bp30_apply(b, G, 1.0, q, out=out),
            "bp1_bp30": lambda: fem.fem_bp1_bp30_apply(b, G, 1.0, q, out_m=out_m, out_a=out)}[op]

    assert _fastest(call) <= 2 * E * bench.alg_counts(N)[1][op] / _fp64_rate() + 10


def test_factors_of_fp64_elements_run_at_the_fp64_rate():
    """All factors of a left-handed mesh at N = 7: at most 1.16 times their FP64
    instructions' time (64 and 243 of 256 lanes have a column, a pipe 0.9 busy)
    and two launches: elements are left to FP64 before their points are computed
    in fixed point."""
    import torch

    import bench
    fem, N = _fem(), 7
    verts = _left_handed(N, 20)
    E, b = verts.shape[0], fem.fem_basis_setup(N)
    wJ, G35, G30 = (torch.empty(fem.geo_shape(b, k, E), dtype=torch.float64, device="cuda")
                    for k in (fem.FEM_GEO_BP1, fem.FEM_GEO_BP35, fem.FEM_GEO_BP30))
    inst = bench.alg_counts(N)[1]
    t = _fastest(lambda: fem.fem_mesh_geofacs_set(b, verts, wJ=wJ, G35=G35, G30=G30))
    assert t <= 1.16 * E * (inst["geofacs_bp35"] + inst["geofacs_bp30_bp1"]) / _fp64_rate() + 20
