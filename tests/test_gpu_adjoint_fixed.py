"""The adjoint kernel's fixed-point contraction: every degree, sizes at which batches and
tiles end, gradients without symmetry, zero, huge, tiny, infinite and NaN upstream values.

Bound: Gbar errs by at most n^2 ulps of sum |A0||dA| (the fixed point by less: 2^-54 of
max|A0| max|dA| a term against 2^-53 of the partial sums), the FP64 geometry and the chain
rule by below 64 ulps of the formula's sum of |terms|, with |K_a| in place of the entries of
row a of J^-1; (n^2 + 64) 2^-53 of that sum, taken with max|A0| max|dA| n^2 for |Gbar|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synthetic import mesh as M  # noqa: E402

pytestmark = pytest.mark.gpu


def _case(d, q, n_elem, scale=1.0, seed=4):
    import paper_1112_0402_gb300 as F

    form = F.Form(F.POISSON, F.TRIANGLE if d == 2 else F.TETRAHEDRON, q)
    m = M.unit_square_triangles(6, 0.2, seed) if d == 2 else M.unit_cube_tets(3, 0.15, seed)
    x = m.vertices[m.cells[np.arange(n_elem) % m.n_elem]]
    ids = np.arange(n_elem * (d + 1), dtype=np.int32).reshape(n_elem, d + 1)
    dA = np.random.default_rng(seed).standard_normal((n_elem, form.n_local, form.n_local)) * scale
    return F, form, x, ids, dA


def _run(F, form, x, ids, dA):
    dv = F.tabulate_adjoint(form, torch.as_tensor(ids, device="cuda"),
                            torch.as_tensor(x.reshape(-1, x.shape[2]).copy(), device="cuda"),
                            torch.as_tensor(dA, device="cuda"))
    assert F.status_poll() == 0
    return dv.cpu().numpy().reshape(x.shape)


def _reference(form, x, dA):
    d = form.dim
    A0 = form.reference_tensor().astype(np.longdouble)
    x = x.astype(np.longdouble)
    J = (x[:, 1:] - x[:, :1]).transpose(0, 2, 1)
    if d == 2:
        adj = np.stack([np.stack([J[:, 1, 1], -J[:, 0, 1]], -1), np.stack([-J[:, 1, 0], J[:, 0, 0]], -1)], -2)
    else:
        adj = np.stack([np.cross(J[:, :, (a + 1) % 3], J[:, :, (a + 2) % 3]) for a in range(3)], 1)
    det = np.einsum("er,er->e", adj[:, 0], J[:, :, 0])
    K, s = adj / det[:, None, None], np.abs(det)[:, None, None]
    G = (dA.reshape(len(x), -1).astype(np.longdouble) @ A0).reshape(-1, d, d)
    KK = np.einsum("eab,ecb->eac", K, K)
    KT = K.transpose(0, 2, 1)
    dJ = s * (np.einsum("eab,eab->e", G, KK)[:, None, None] * KT - KT @ (G + G.transpose(0, 2, 1)) @ KK)
    ref = np.concatenate([-dJ.sum(2)[:, None, :], dJ.transpose(0, 2, 1)], 1)
    row = np.sqrt((K * K).sum(2)).sum(1)  # sum of |K_a|
    g = np.abs(A0).max() * np.abs(dA).reshape(len(x), -1).max(1) * A0.shape[0]
    bound = np.abs(det) * 3 * d * g * row ** 3
    return ref, (A0.shape[0] + 64) * 2.0 ** -53 * bound[:, None, None]


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("q", [1, 2, 3, 4])
@pytest.mark.parametrize("n_elem,scale", [(1, 1.0), (33, 2.0 ** -200), (130, 2.0 ** 300)])
def test_against_formula(d, q, n_elem, scale):
    F, form, x, ids, dA = _case(d, q, n_elem, scale)
    got = _run(F, form, x, ids, dA)
    ref, tol = _reference(form, x, dA)
    assert (np.abs(got - ref) <= tol).all()


def test_many_cells():
    """More cells than the resident warps take at one a batch (tiles of 32 cells)."""
    F, form, x, ids, dA = _case(3, 2, 152 * 24 * 32 + 5)
    got = _run(F, form, x, ids, dA)
    ref, tol = _reference(form, x, dA)
    assert (np.abs(got - ref) <= tol).all()


@pytest.mark.parametrize("d,q", [(2, 2), (3, 2), (3, 4)])
def test_zero_extreme_and_non_finite_gradients(d, q):
    F, form, x, ids, dA = _case(d, q, 40)
    dA[3] = 0.0
    dA[7] *= 2.0 ** 950
    dA[8] *= 2.0 ** -1000
    dA[11, 0, 0] = np.inf
    dA[20, -1, 0] = np.nan
    got = _run(F, form, x, ids, dA)
    bad = np.isin(np.arange(40), (11, 20))
    assert not np.isfinite(got[bad]).all(axis=(1, 2)).any()
    assert not got[3].any()
    ref, tol = _reference(form, x[~bad], dA[~bad])
    # a denormal step of each of the products where the gradient is tiny
    assert (np.abs(got[~bad] - ref) <= tol + 2.0 ** -1060).all()
