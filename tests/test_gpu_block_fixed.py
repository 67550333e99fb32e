"""FP64 element tensors of the vector forms by the block algorithm, whose contraction runs in
fixed point, against the dense FP64 contraction: both sides of the rules that send cells to
the FP64 multiply-adds (stretched cells, lambda far above mu), every kernel, ragged tiles.

Bound: an entry is a sum of at most 90 (convection) or 81 terms A0 G, each evaluation errs by
at most that many ulps of the sum of |terms|, plus below 32 for the FP64 geometry, and the
fixed point by below 2^-50 of max|A0| max|G|: 256 ulps of max|A0| sum_alpha B, where B bounds
|G| by the lengths of the rows of J^-1."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synthetic import mesh as M  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretch", [(1, 1, 1), (2, 1, 8), (1, 1, 64)])
@pytest.mark.parametrize("kind,q,n_elem", [("convection", 1, 1), ("convection", 1, 131), ("convection", 2, 67),
                                           ("elasticity", 1, 131), ("elasticity", 2, 66), ("elasticity", 3, 65)])
@pytest.mark.parametrize("lmbda", [1.25, 1.0e4])
def test_block_matches_dense(kind, q, n_elem, stretch, lmbda):
    import paper_1112_0402_gb300 as F

    if kind == "convection" and lmbda != 1.25:
        pytest.skip("no Lame parameter")
    code = F.NS_CONVECTION if kind == "convection" else F.ELASTICITY
    block = F.Form(code, F.TETRAHEDRON, q, 1.0, lmbda)
    dense = F.Form(code, F.TETRAHEDRON, q, 1.0, lmbda, algorithm=F.ALG_DENSE)
    m = M.unit_cube_tets(3, 0.15, 5)
    x = m.vertices[m.cells[np.arange(n_elem) % m.n_elem]] * np.array(stretch, dtype=np.float64)
    ids = np.arange(4 * n_elem, dtype=np.int32).reshape(n_elem, 4)
    rng = np.random.default_rng(9)
    w = rng.standard_normal((n_elem, block.n_local)) if kind == "convection" else None
    args = [torch.as_tensor(ids, device="cuda"), torch.as_tensor(x.reshape(-1, 3).copy(), device="cuda")]
    kw = {"coeffs": None if w is None else torch.as_tensor(w, device="cuda")}
    A, B = F.tabulate(block, *args, **kw), F.tabulate(dense, *args, **kw)
    J = (x[:, 1:] - x[:, :1]).transpose(0, 2, 1)
    K, det = np.linalg.inv(J), np.abs(np.linalg.det(J))
    rows = np.sqrt((K * K).sum(2))  # |K_a|
    if kind == "convection":
        total = det * rows.sum(1) * np.abs(w).sum(1)
    else:
        total = 9 * det * (2.0 + lmbda) * rows.sum(1) ** 2
    tol = 256 * 2.0 ** -53 * np.abs(block.reference_tensor()).max() * total
    diff = (A - B).abs().reshape(n_elem, -1).amax(1).cpu().numpy()
    assert (diff <= tol).all()
    n = block.n_local
    nnz = n_elem * n * n
    slot = torch.randperm(nnz, generator=torch.Generator().manual_seed(3)).to(torch.int32).reshape(n_elem, n, n).cuda()
    val = torch.zeros(nnz, dtype=torch.float64, device="cuda")
    F.assemble(block, args[0], args[1], slot, val, **kw)
    assert F.status_poll() == 0
    # the same contraction; results may leave the fixed point by another of its two exact
    # roundings (ties to even or away from zero)
    got = val[slot.long().reshape(-1)].reshape(A.shape)
    assert ((got - A).abs() <= 2.0 ** -52 * A.abs()).all()


def test_uniform_and_zero_coefficients():
    """w constant along an axis (whole geometry columns zero) and w = 0."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.NS_CONVECTION, F.TETRAHEDRON, 2)
    m = M.unit_cube_tets(2, 0.0, 1)
    c, v = torch.as_tensor(m.cells, device="cuda"), torch.as_tensor(m.vertices, device="cuda")
    w = torch.zeros((m.n_elem, 30), dtype=torch.float64, device="cuda")
    assert not F.tabulate(form, c, v, coeffs=w).any()
    w[:, 10:20] = 3.0  # w = (0, 3, 0)
    A = F.tabulate(form, c, v, coeffs=w)
    dense = F.tabulate(F.Form(F.NS_CONVECTION, F.TETRAHEDRON, 2, algorithm=F.ALG_DENSE), c, v, coeffs=w)
    scale = dense.abs().amax()
    assert (A - dense).abs().amax() <= 256 * 2.0 ** -53 * scale * 30
    assert F.status_poll() == 0
