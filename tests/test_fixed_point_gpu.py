"""The FP64 operators on the integer pipe (csrc/fx.cuh) where their rules
change hands: element scales from 2^-900 to 2^900, elements that hold values
of many magnitudes, zeros, spikes, NaN and Inf (which go through FP64 lines),
flat and indefinite factors, every degree, element counts around the block
sizes.  Against the oracle, node by node.

Bar: |y - y_oracle| <= 8 (1.5 n + 17) 2^-53 b, with b the same operator on
absolute values and on operators folded even-odd as FP64 lines evaluate them,
(|A[a][i]| + |A[a][Q-1-i]|) for A[a][i]: an FP64 evaluation makes at most
about n/2 + 3 roundings per contraction on the longest chain (three
contractions in BP3.5, six in BP1.0, nine in BP3.0: 1.5 n, 3 n, 4.5 n), 8 in
the chain rule and the sums, for each side, times 4 for what the two
evaluations order differently."""
import numpy as np
import pytest

import fem_synth
import oracle

pytestmark = pytest.mark.gpu


def _fem():
    import paper_1711_00903_gb300 as fem
    return fem


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _along(A, u, axis):
    return np.moveaxis(np.tensordot(A, u, axes=(1, axis)), 0, axis)


def _folded_abs(A):
    return np.abs(A) + np.abs(A[:, ::-1])


def _stiff_abs(D, G, u):
    k = u.shape[-1]
    g = np.abs(G).reshape(-1, 7, k, k, k)
    D, DT = _folded_abs(D), _folded_abs(D.T)
    ur, us, ut = _along(D, u, 3), _along(D, u, 2), _along(D, u, 1)
    wr = g[:, 0] * ur + g[:, 1] * us + g[:, 2] * ut
    ws = g[:, 1] * ur + g[:, 3] * us + g[:, 4] * ut
    wt = g[:, 2] * ur + g[:, 4] * us + g[:, 5] * ut
    return _along(DT, wr, 3) + _along(DT, ws, 2) + _along(DT, wt, 1), g[:, 6]


class Op:
    """BP3.5 with its factors, oracle and bound."""

    chain = 1.5

    def __init__(self, N):
        self.N, self.n, self.b = N, N + 1, oracle.Basis(N)

    def factors(self, verts):
        return oracle.geofacs(self.N, 2, verts)[0]

    def oracle(self, geo, q):
        return oracle.bp35(self.N, geo, 0.37, q)

    def apply(self, geo, q):
        fem = _fem()
        return fem.fem_bp35_apply(fem.fem_basis_setup(self.N), _dev(geo), 0.37, _dev(q)).cpu().numpy()

    def bound(self, geo, q):
        u = np.abs(q).reshape(-1, self.n, self.n, self.n)
        s, wj = _stiff_abs(self.b.D, geo, u)
        return (s + 0.37 * wj * u).reshape(q.shape)

    @property
    def tol(self):
        return 8 * (self.chain * self.n + 17) * 2.0 ** -53


class Dealiased(Op):
    """BP3.0: nine contractions on the longest chain."""

    chain = 4.5

    def factors(self, verts):
        return oracle.geofacs(self.N, 3, verts)[0]

    def oracle(self, geo, q):
        return oracle.bp30(self.N, geo, 0.37, q)

    def apply(self, geo, q):
        fem = _fem()
        return fem.fem_bp30_apply(fem.fem_basis_setup(self.N), _dev(geo), 0.37, _dev(q)).cpu().numpy()

    def _interp(self, q):
        u, I = np.abs(q).reshape(-1, self.n, self.n, self.n), _folded_abs(self.b.I)
        return _along(I, _along(I, _along(I, u, 3), 2), 1)

    def _project(self, g, shape):
        IT = _folded_abs(self.b.I.T)
        return _along(IT, _along(IT, _along(IT, g, 3), 2), 1).reshape(shape)

    def bound(self, geo, q):
        u = self._interp(q)
        s, wj = _stiff_abs(self.b.Dt, geo, u)
        return self._project(s + 0.37 * wj * u, q.shape)


class Mass(Dealiased):
    """BP1.0: six contractions; its factors are the seventh plane."""

    chain = 3.0

    def factors(self, verts):
        return oracle.geofacs(self.N, 1, verts)[0]

    def oracle(self, geo, q):
        return oracle.bp1(self.N, geo, q)

    def apply(self, geo, q):
        fem = _fem()
        return fem.fem_bp1_apply(fem.fem_basis_setup(self.N), _dev(geo), _dev(q)).cpu().numpy()

    def bound(self, geo, q):
        u = self._interp(q)
        return self._project(np.abs(geo).reshape(u.shape) * u, q.shape)


OPS = {"bp35": Op, "bp30": Dealiased, "bp1": Mass}


def _check(op, geo, q):
    got, ref = op.apply(geo, q), op.oracle(geo, q)
    np.testing.assert_array_equal(np.isfinite(got), np.isfinite(ref))
    fine = np.isfinite(ref)
    with np.errstate(invalid="ignore", over="ignore"):
        assert np.all(np.abs(got - ref)[fine] <= (op.tol * op.bound(geo, q))[fine])
    return got


def _elements(op, seed=5):
    """Eleven elements: ordinary ones and each kind that changes the path."""
    rng = np.random.default_rng(seed)
    verts = fem_synth.box_mesh(3, 2, 2, seed=seed)[:11].copy()
    geo = op.factors(verts)
    NP = op.n ** 3
    q = rng.uniform(-1, 1, (11, NP))
    i = np.arange(NP)
    q[1] = 0.0
    q[2, rng.integers(NP)] = 1e12                                       # one value far above the rest
    q[3] *= 10.0 ** -(2.0 * (i % op.n + (i // op.n) % op.n + i // op.n ** 2))  # decay in every direction
    q[4] = 0.0
    q[4, rng.integers(NP)] = 1.0                                        # a unit vector
    q[5, rng.integers(NP)] = np.nan
    q[6, rng.integers(NP)] = np.inf
    q[7] *= 2.0 ** 900
    q[8] *= 2.0 ** -900
    geo[9] = -geo[9]                                                    # not positive definite
    q[10].reshape(op.n, op.n, op.n)[0, 0, :] = 1e-17                    # an edge of near-zeros
    return geo, q


@pytest.mark.parametrize("name", sorted(OPS))
@pytest.mark.parametrize("N", range(1, 16))
def test_elements_of_every_kind(name, N):
    op = OPS[name](N)
    geo, q = _elements(op)
    got = _check(op, geo, q)
    # an element's result does not depend on its neighbours in the block
    for e in (0, 3, 10):
        np.testing.assert_array_equal(op.apply(geo[e:e + 1], q[e:e + 1])[0], got[e])


@pytest.mark.parametrize("N", range(1, 16))
def test_one_pass_is_both_operators(N):
    """BP1.0 and BP3.0 in one pass: the bits of each alone, whichever path an element takes."""
    op, mass = Dealiased(N), Mass(N)
    geo, q = _elements(op)
    fem = _fem()
    m, a = fem.fem_bp1_bp30_apply(fem.fem_basis_setup(N), _dev(geo), 0.37, _dev(q))
    np.testing.assert_array_equal(a.cpu().numpy(), op.apply(geo, q))
    np.testing.assert_array_equal(m.cpu().numpy(), mass.apply(np.ascontiguousarray(geo[:, 6]), q))


@pytest.mark.parametrize("name", sorted(OPS))
@pytest.mark.parametrize("N", [1, 4, 7, 10, 15])
def test_flat_and_scaled_elements(name, N):
    op = OPS[name](N)
    rng = np.random.default_rng(N)
    verts = fem_synth.box_mesh(3, 1, 1, seed=N)
    q = rng.uniform(-1, 1, (3, op.n ** 3))
    for scale in ((1, 1, 1e-4), (1e3, 1, 1), (1e-3, 1e-3, 1e-3)):
        _check(op, op.factors(np.ascontiguousarray(verts * np.array(scale))), q)
    geo = op.factors(verts)
    got = op.apply(geo, q)
    for k in (-200, 40, 200):  # a power of two scales the result exactly
        np.testing.assert_array_equal(op.apply(geo, np.ldexp(q, k)), np.ldexp(got, k))
        np.testing.assert_array_equal(op.apply(np.ldexp(geo, k), q), np.ldexp(got, k))


@pytest.mark.parametrize("name", sorted(OPS))
@pytest.mark.parametrize("N", [1, 2, 3, 5, 6, 8, 9, 12])
def test_element_counts_around_the_blocks(name, N):
    op = OPS[name](N)
    verts = fem_synth.box_mesh(5, 5, 3, seed=N)
    geo = op.factors(verts)
    q = np.random.default_rng(N).uniform(-1, 1, (75, op.n ** 3))
    full = _check(op, geo, q)
    for E in (1, 2, 3, 7, 31, 32, 33):
        np.testing.assert_array_equal(op.apply(geo[:E], q[:E]), full[:E])


def _hexahedra():
    """An ordinary element, a box, a sheared, a rotated and a strongly
    distorted one, one with a skew of 1e-5, a flat, a large, a tiny and an
    inverted one."""
    rng = np.random.default_rng(3)
    box = np.array([[(c >> d) & 1 for d in range(3)] for c in range(8)], dtype=float)
    jitter = rng.uniform(-1, 1, (8, 3))
    rot = np.linalg.qr(rng.standard_normal((3, 3)))[0]
    rot *= np.sign(np.linalg.det(rot))
    shear = np.array([[1, 0.7, -0.4], [0, 1, 0.8], [0, 0, 1.0]])
    v = [box + 0.1 * jitter, box, box @ shear.T, (box + 0.05 * jitter) @ rot.T, box + 0.2 * jitter,
         box + 1e-5 * jitter, box * [1, 1, 1e-3] + 1e-5 * jitter, 2.0 ** 90 * (box + 0.1 * jitter),
         2.0 ** -90 * (box + 0.1 * jitter), (box + 0.1 * jitter)[[1, 0, 3, 2, 5, 4, 7, 6]]]
    return np.ascontiguousarray(np.array(v))


@pytest.mark.parametrize("N", [1, 2, 4, 7, 8, 9, 15])
def test_factors_of_elements_of_every_kind(N):
    """Geometric factors, fixed-point or FP64 by element: each within 1e-13 of
    the oracle relative to sqrt(Gaa Gbb) (about 40 roundings at a cancellation
    of up to 20 in the determinant) times the ratio of the element's largest
    coordinate to its shortest edge (the columns of the map are differences of
    coordinates, which the oracle rounds at the coordinates' size), wJ the same
    bits from every entry point, and the same bits for an element alone."""
    fem = _fem()
    b, verts = fem.fem_basis_setup(N), _hexahedra()
    edges = np.stack([verts[:, i] - verts[:, j] for i, j in ((1, 0), (2, 0), (4, 0), (7, 6), (7, 5), (7, 3))], 1)
    ratio = np.abs(verts).max((1, 2)) / np.linalg.norm(edges, axis=2).min(1)
    for kind in (fem.FEM_GEO_BP35, fem.FEM_GEO_BP30):
        got = fem.fem_mesh_geofacs(b, kind, _dev(verts)).cpu().numpy()
        ref = oracle.geofacs(N, kind, verts)[0]
        d = np.sqrt(np.abs(ref[:, [0, 3, 5]]))
        scale = np.stack([d[:, 0] ** 2, d[:, 0] * d[:, 1], d[:, 0] * d[:, 2], d[:, 1] ** 2, d[:, 1] * d[:, 2],
                          d[:, 2] ** 2, np.abs(ref[:, 6])], 1)
        assert np.all(np.abs(got - ref) <= 1e-13 * ratio[:, None, None] * scale)
        for e in (1, 5, 9):
            np.testing.assert_array_equal(fem.fem_mesh_geofacs(b, kind, _dev(verts[e:e + 1])).cpu().numpy()[0], got[e])
    wj = fem.fem_mesh_geofacs(b, fem.FEM_GEO_BP1, _dev(verts)).cpu().numpy()
    np.testing.assert_array_equal(wj, got[:, 6])
