"""FP64 contractions in fixed point on inputs whose factors differ by many orders of magnitude:
every entry within a few ulps of the sum of its own |terms|, as FP64 multiply-adds give it, not
of the cell's largest.

The terms run down to the products behind the cofactors: with U[a][c] the sum of the magnitudes
of the products of cofactor (c, a) of J over |det J|, row a, entry c of K = J^-1 errs by below 8
ulps of U (the cofactor's two products and difference 2, the determinant 4, reciprocal and
product 2), so the terms of an entry are formed with U in the place of |K| (once in a product of
two, the other factor K).

Entries of the reference tensor that are zero but for rounding (below 2^-45 of their row's
largest) are held to 2^-59 of that; what this changes is allowed for, entry by entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synthetic import mesh as M  # noqa: E402

pytestmark = pytest.mark.gpu
LD = np.longdouble
ULP = 2.0 ** -53


def _geometry(x):
    """K, U (as above) and |det J| in extended precision, x [E, d+1, d]."""
    J = (x[:, 1:] - x[:, :1]).transpose(0, 2, 1).astype(LD)
    d = J.shape[1]
    if d == 2:
        adj = np.stack([np.stack([J[:, 1, 1], -J[:, 0, 1]], -1), np.stack([-J[:, 1, 0], J[:, 0, 0]], -1)], -2)
        terms = np.abs(adj)
    else:
        adj, terms = np.empty_like(J), np.empty_like(J)
        for a in range(3):
            for c in range(3):
                p = J[:, (c + 1) % 3, (a + 1) % 3] * J[:, (c + 2) % 3, (a + 2) % 3]
                q = J[:, (c + 1) % 3, (a + 2) % 3] * J[:, (c + 2) % 3, (a + 1) % 3]
                adj[:, a, c], terms[:, a, c] = p - q, np.abs(p) + np.abs(q)
    det = np.einsum("ec,ec->e", adj[:, 0], J[:, :, 0])
    return adj / det[:, None, None], terms / np.abs(det)[:, None, None], np.abs(det)


def _corners(d, n_elem, shear, seed=3):
    """Corner simplices J = I + lower triangle of entries of size `shear` (zero: K = I)."""
    r = np.random.default_rng(seed)
    J = np.eye(d) + shear * np.tril(r.uniform(0.5, 1.0, (n_elem, d, d)) * r.choice([-1, 1], (n_elem, d, d)), -1)
    x = np.zeros((n_elem, d + 1, d))
    x[:, 1:] = J.transpose(0, 2, 1)
    return x


def _on_gpu(x):
    n, v, d = x.shape
    ids = np.arange(n * v, dtype=np.int32).reshape(n, v)
    return torch.as_tensor(ids, device="cuda"), torch.as_tensor(x.reshape(-1, d).copy(), device="cuda")


def _noise(rows):
    """2^-59 of each row's largest entry where an entry is zero but for rounding, else 0."""
    top = np.abs(rows).max(1, keepdims=True)
    return np.where((rows != 0) & (np.abs(rows) < 2.0 ** -45 * top), 2.0 ** -59 * top, 0.0)


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("q", [1, 2, 3, 4])
@pytest.mark.parametrize("shear", [0.0, 2.0 ** -5, 2.0 ** -7, 2.0 ** -14, 2.0 ** -27, 2.0 ** -45])
def test_poisson_sheared_corners(d, q, shear):
    """Off-diagonal entries of G_K far below the diagonal ones. The contraction adds at most 7
    ulps to the 24 of G_K (two entries of K, three products and their sum, the determinant)."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.POISSON, F.TRIANGLE if d == 2 else F.TETRAHEDRON, q)
    x = _corners(d, 101, shear)
    A = F.tabulate(form, *_on_gpu(x)).cpu().numpy()
    assert F.status_poll() == 0
    K, U, det = _geometry(x)
    n = form.n_local
    A0 = form.reference_tensor().reshape(n, n, d, d)
    pairs = [(a, b) for a in range(d) for b in range(a, d)]
    A0 = np.stack([A0[:, :, a, b] + (A0[:, :, b, a] if a != b else 0.0) for a, b in pairs])
    A0 = np.triu(A0) + np.triu(A0, 1).transpose(0, 2, 1)  # entries i1 <= i2, mirrored
    rows = A0.reshape(len(pairs), -1).T  # [n n][pairs]
    G = np.stack([det * (K[:, a] * K[:, b]).sum(1) for a, b in pairs], 1)
    I = np.stack([det * (U[:, a] * np.abs(K[:, b]) + np.abs(K[:, a]) * U[:, b]).sum(1) for a, b in pairs], 1)
    ref = (G @ rows.T.astype(LD)).reshape(A.shape)
    tol = (I @ (32 * ULP * np.abs(rows) + _noise(rows)).T).reshape(A.shape)
    assert (np.abs(A - ref) <= tol).all()


def _aligned(n_elem, stretch=(1.0, 2.0, 0.5)):
    return _corners(3, n_elem, 0.0) * np.array(stretch)


def _jittered(n_elem):
    m = M.unit_cube_tets(3, 0.15, 5)
    return m.vertices[m.cells[np.arange(n_elem) % m.n_elem]]


def _coefficients(kind, n_elem, ns):
    r = np.random.default_rng(8)
    w = r.standard_normal((n_elem, 3, ns))
    if kind == "wall":  # no slip on a part of the nodes
        return w * (r.random((n_elem, 1, ns)) < 0.5)
    if kind == "one node":
        return w * (np.arange(ns) == r.integers(0, ns, n_elem)[:, None])[:, None]
    if kind == "nodes":
        return w * np.exp2(r.uniform(-60, 0, (n_elem, 1, ns)))
    return w * np.array(kind)[:, None]


@pytest.mark.parametrize("q", [1, 2])
@pytest.mark.parametrize("cells", [_aligned, _jittered])
@pytest.mark.parametrize("kind", [(1.0, 1.0, 1.0), (1.0, 1e-4, 1.0), (1.0, 1e-8, 0.0), (1e-12, 1.0, 1e-18), "wall",
                                  "one node", "nodes"])
def test_convection_coefficients(q, cells, kind):
    """Coefficients of very different size between components or nodes: a sum of at most 30
    terms (31 ulps), each the product of K (8 ulps of U), w and |det J| (4) summed over three
    components (4)."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.NS_CONVECTION, F.TETRAHEDRON, q)
    n = form.n_local
    ns, n_elem = n // 3, 131
    x, w = cells(n_elem), _coefficients(kind, n_elem, n // 3)
    c, v = _on_gpu(x)
    A = F.tabulate(form, c, v, coeffs=torch.as_tensor(w.reshape(n_elem, n), device="cuda"))
    assert F.status_poll() == 0
    A = A.cpu().numpy().reshape(n_elem, 3, ns, 3, ns)
    K, U, det = _geometry(x)
    R = form.reference_tensor().reshape(n, n, n, 3)[:ns, :ns, :ns].reshape(ns * ns, ns * 3)
    H = det[:, None, None] * np.einsum("eac,ect->eta", K, w.astype(LD))
    T = det[:, None, None] * np.einsum("eac,ect->eta", U, np.abs(w).astype(LD))
    ref = (H.reshape(n_elem, -1) @ R.T.astype(LD)).reshape(n_elem, ns, ns)
    tol = 48 * ULP * (T.reshape(n_elem, -1) @ np.abs(R).T.astype(LD)).reshape(n_elem, ns, ns)
    for i in range(3):
        for j in range(3):
            if i == j:
                assert (np.abs(A[:, i, :, i] - ref) <= tol).all()
            else:
                assert not A[:, i, :, j].any()


@pytest.mark.parametrize("q", [1, 2, 3])
@pytest.mark.parametrize("cells", [_aligned, _jittered, lambda n: _corners(3, n, 2.0 ** -12),
                                   lambda n: _corners(3, n, 2.0 ** -27)], ids=["aligned", "jittered", "-12", "-27"])
@pytest.mark.parametrize("lmbda", [1.25, 1e-4, 1e-8, 1e-13, 0.0, 1e4])
def test_elasticity_small_factors(q, cells, lmbda):
    """lambda far below mu, and entries of K far below the others: a sum of 9 terms (10 ulps),
    each a sum of three products (3) of two entries of K (16), a Lame parameter and |det J| (6)."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.ELASTICITY, F.TETRAHEDRON, q, 1.0, lmbda)
    n = form.n_local
    ns, n_elem = n // 3, 67
    x = cells(n_elem)
    A = F.tabulate(form, *_on_gpu(x)).cpu().numpy().reshape(n_elem, 3, ns, 3, ns)
    assert F.status_poll() == 0
    K, U, det = _geometry(x)
    rows = F.Form(F.POISSON, F.TETRAHEDRON, q).reference_tensor().reshape(ns * ns, 9)
    weight, X = 40 * ULP * np.abs(rows) + _noise(rows), np.abs(K)
    for i in range(3):
        for j in range(3):
            B = K[:, :, None, j] * K[:, None, :, i] + lmbda * K[:, :, None, i] * K[:, None, :, j]
            T = (U[:, :, None, j] * X[:, None, :, i] + X[:, :, None, j] * U[:, None, :, i] +
                 lmbda * (U[:, :, None, i] * X[:, None, :, j] + X[:, :, None, i] * U[:, None, :, j]))
            if i == j:
                B = B + np.einsum("eac,ebc->eab", K, K)
                T = T + np.einsum("eac,ebc->eab", U, X) + np.einsum("eac,ebc->eab", X, U)
            B, T = (B * det[:, None, None]).reshape(-1, 9), (T * det[:, None, None]).reshape(-1, 9)
            err = np.abs(A[:, i, :, j].reshape(n_elem, -1) - B @ rows.T.astype(LD))
            assert (err <= T @ weight.T).all()


def _upstream(kind, form, n_elem):
    r = np.random.default_rng(6)
    n = form.n_local
    x = r.standard_normal((n_elem, n, n))
    if kind == "rank one":
        return r.standard_normal((n_elem, n, 1)) * r.standard_normal((n_elem, 1, n))
    if kind == "diagonal":
        return x * np.eye(n)
    if kind == "wide":
        return x * np.exp2(r.uniform(-60, 0, x.shape))
    e, i, j = np.arange(n_elem), r.integers(0, n, n_elem), r.integers(0, n, n_elem)
    if kind == "one entry":
        y = np.zeros_like(x)
        y[e, i, j] = x[e, i, j]
        return y
    x[e, i, j] *= kind
    return x


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("q", [1, 2, 3, 4])
@pytest.mark.parametrize("kind", ["normal", "rank one", "diagonal", "wide", "one entry", 1e6, 1e12, 1e20])
@pytest.mark.parametrize("regular", [True, False])
def test_adjoint_upstream_spread(d, q, kind, regular):
    """Each component of dL/dvertices by its own terms, upstream entries of very different size.
    Gbar is a sum of n^2 terms: roundings of at most an ulp of the sum of |terms| each, which
    random signs add to below 2n ulps. The formula's products take two entries of K more (48
    ulps with their sums)."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.POISSON, F.TRIANGLE if d == 2 else F.TETRAHEDRON, q)
    n, n_elem = form.n_local, 70
    dA = _upstream(1.0 if kind == "normal" else kind, form, n_elem)
    if regular:
        x = _corners(d, n_elem, 0.0)
    else:
        m = M.unit_square_triangles(6, 0.2, 4) if d == 2 else M.unit_cube_tets(3, 0.15, 4)
        x = m.vertices[m.cells[np.arange(n_elem) % m.n_elem]]
    got = F.tabulate_adjoint(form, *_on_gpu(x), torch.as_tensor(dA, device="cuda")).cpu().numpy().reshape(x.shape)
    assert F.status_poll() == 0
    K, U, det = _geometry(x)
    A0 = form.reference_tensor().astype(LD)
    G = (dA.reshape(n_elem, -1).astype(LD) @ A0).reshape(-1, d, d)
    S = (np.abs(dA).reshape(n_elem, -1).astype(LD) @ np.abs(A0)).reshape(-1, d, d)

    def gradient(G, K, sign):  # dL/dvertices; sign +1: the sum of the terms' magnitudes
        G, KT = G + G.transpose(0, 2, 1), K.transpose(0, 2, 1)
        c = np.einsum("eab,eak,ebk->e", G, K, K)[:, None, None] / 2
        dJ = det[:, None, None] * (c * KT + sign * (KT @ G @ K @ KT))
        return np.concatenate([sign * dJ.sum(2)[:, None], dJ.transpose(0, 2, 1)], 1)

    tol = (2 * n + 48) * ULP * gradient(S, np.maximum(U, np.abs(K)), 1)
    assert (np.abs(got - gradient(G, K, -1)) <= tol).all()


@pytest.mark.parametrize("q", [1, 2, 3])
@pytest.mark.parametrize("power", [-690, -705, -880, 880])
def test_elasticity_far_from_one(q, power):
    """mu and lambda times a power of two: the same tensors times that power, on either side of
    the range of the fixed point, up to the two contractions' roundings (20 ulps of the largest)."""
    import paper_1112_0402_gb300 as F

    x = np.concatenate([_jittered(60), _aligned(7)])
    args = _on_gpu(x)
    A = F.tabulate(F.Form(F.ELASTICITY, F.TETRAHEDRON, q, 1.0, 1.25), *args).cpu().numpy()
    scale = 2.0 ** power
    B = F.tabulate(F.Form(F.ELASTICITY, F.TETRAHEDRON, q, scale, 1.25 * scale), *args).cpu().numpy() / scale
    assert F.status_poll() == 0
    assert (np.abs(B - A) <= 20 * ULP * np.abs(A).max((1, 2), keepdims=True)).all()


@pytest.mark.parametrize("q", [1, 2, 4])
@pytest.mark.parametrize("power", [-690, -705, -880, 880])
def test_adjoint_far_from_one(q, power):
    """The same of dA: the gradient scales, up to roundings (n^2 ulps of the largest component)."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.POISSON, F.TETRAHEDRON, q)
    args = _on_gpu(_jittered(60))
    dA = _upstream(1.0, form, 60)
    got = [F.tabulate_adjoint(form, *args, torch.as_tensor(dA * s, device="cuda")).cpu().numpy().reshape(60, -1) / s
           for s in (1.0, 2.0 ** power)]
    assert F.status_poll() == 0
    assert (np.abs(got[1] - got[0]) <= form.n_local ** 2 * 4 * ULP * np.abs(got[0]).max(1, keepdims=True)).all()
