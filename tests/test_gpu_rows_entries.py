"""Every entry of the row-owner sums on the smallest meshes (chunks of fewer pairs than warps),
within the fixed point's own bound: an entry of m contributions errs by at most m u / 2 (FP32:
u / 2 <= 2^-30 B; FP64: truncation, u <= 2^-60 B) against the fused assembly of the same
contributions, with B the largest max|A0[i1]| sum|G_K| times the most pairs of a row, and the
FP64 atomics and the rounding of the result by m + 1 ulps of the contributions. That is below
5e-6 of the largest element entry for FP32; 99% of the entries are above 1e-4 of it, so a
contribution left out, doubled or put elsewhere shows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synthetic import mesh as M  # noqa: E402
from synthetic import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("d,q", [(d, q) for d in (2, 3) for q in (1, 2, 3, 4)])
@pytest.mark.parametrize("n", [1, 2, 3])
def test_entries_of_small_meshes(d, q, n, precision):
    import paper_1112_0402_gb300 as F

    m = M.unit_square_triangles(n, 0.15, 3) if d == 2 else M.unit_cube_tets(n, 0.15, 3)
    p = W.make_problem(m, W.MASS, q)
    rp, col, slot = F.csr_pattern(p.dofmap, p.n_dof)
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    cell = F.TRIANGLE if d == 2 else F.TETRAHEDRON
    cells, verts, slots = dev(m.cells), dev(m.vertices), dev(slot)
    plan = F.RowPlan(dev(p.dofmap), p.n_dof, dev(rp), dev(col))
    contributions = np.bincount(slot.reshape(-1), minlength=col.size)
    x = m.vertices[m.cells]
    J = (x[:, 1:] - x[:, :1]).transpose(0, 2, 1)
    det, K = np.abs(np.linalg.det(J)), np.linalg.inv(J)
    G = det[:, None, None] * (K @ K.transpose(0, 2, 1))
    size = {F.MASS: det.max(), F.POISSON: np.abs(G).sum((1, 2)).max()}
    for kind in (F.MASS, F.POISSON):
        form = F.Form(kind, cell, q)
        got, ref = (torch.full((col.size,), v, dtype=torch.float64, device="cuda") for v in (3.0, 0.0))
        F.assemble_rows(form, plan, cells, verts, got, precision=precision)
        F.assemble(form, cells, verts, slots, ref, precision=precision)
        A0 = form.reference_tensor()
        if kind == F.POISSON:  # the kernels' columns are the pairs (a, b) and (b, a) summed
            A0 = A0.reshape(-1, d, d)
            A0 = A0 + np.triu(A0, 1).transpose(0, 2, 1) + np.tril(A0, -1).transpose(0, 2, 1)
        B = 1.001 * np.abs(A0).max() * size[kind] * plan.max_incidence
        unit = (2.0 ** -30 if precision == "fp32" else 2.0 ** -60) * B
        tol = contributions * unit + (contributions + 1) * 2.0 ** -52 * B / plan.max_incidence
        assert (np.abs((got - ref).cpu().numpy()) <= tol).all()
    assert F.status_poll() == 0
