"""Row-owner assembly over the smallest meshes (chunks of fewer pairs than warps, one class
run per pair), every element, and under graph capture. Reference: the fused assembly, which
adds the same FP32 (or FP64) contributions with FP64 atomics; the fixed-point sums differ
from it by at most m 2^-30 B (FP32) or m 2^-61 B plus rounding (FP64), B below the number of
cells times the largest contribution bound, max|A0| sum|G| <= n_alpha * max|A0| * max|G|, and
the FP64 contributions themselves by their own rounding, 2^-50 of the same bound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synthetic import mesh as M  # noqa: E402
from synthetic import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _setup(d, q, n):
    import paper_1112_0402_gb300 as F

    m = M.unit_square_triangles(n, 0.15, 3) if d == 2 else M.unit_cube_tets(n, 0.15, 3)
    p = W.make_problem(m, W.MASS, q)
    rp, col, slot = F.csr_pattern(p.dofmap, p.n_dof)
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    cell = F.TRIANGLE if d == 2 else F.TETRAHEDRON
    forms = [F.Form(F.MASS, cell, q), F.Form(F.POISSON, cell, q)]
    plan = F.RowPlan(dev(p.dofmap), p.n_dof, dev(rp), dev(col))
    return F, forms, plan, dev(m.cells), dev(m.vertices), dev(slot), col.size


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("d,q", [(d, q) for d in (2, 3) for q in (1, 2, 3, 4)])
@pytest.mark.parametrize("n", [1, 2])
def test_small_meshes(d, q, n, precision):
    F, forms, plan, cells, verts, slot, nnz = _setup(d, q, n)
    vals = [torch.full((nnz,), 3.0, dtype=torch.float64, device="cuda") for _ in range(2)]
    F.assemble_rows_pair(*forms, plan, cells, verts, *vals, precision=precision)
    for form, val in zip(forms, vals):
        ref = torch.zeros(nnz, dtype=torch.float64, device="cuda")
        F.assemble(form, cells, verts, slot, ref, precision=precision)
        single = torch.full((nnz,), 5.0, dtype=torch.float64, device="cuda")
        F.assemble_rows(form, plan, cells, verts, single, precision=precision)
        assert torch.equal(single, val)
        A = F.tabulate(form, cells, verts).abs().amax().item()
        m = plan.max_incidence
        # max|A0| sum|G| is within 2^12 of the largest |A| (the diagonal entries of A0 differ by
        # less than that for these forms)
        unit = 2.0 ** -30 if precision == "fp32" else 2.0 ** -50
        assert (val - ref).abs().amax().item() <= m * m * 2.0 ** 12 * unit * A
    assert F.status_poll() == 0


@pytest.mark.parametrize("q", [2, 4])
def test_captured_and_replayed(q):
    F, forms, plan, cells, verts, slot, nnz = _setup(3, q, 4)
    a, b = (torch.zeros(nnz, dtype=torch.float64, device="cuda") for _ in range(2))
    F.assemble_rows_pair(*forms, plan, cells, verts, a, b)
    want = [a.clone(), b.clone()]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        F.assemble_rows_pair(*forms, plan, cells, verts, a, b)
        F.assemble_rows_pair(*forms, plan, cells, verts, a, b)
    for _ in range(3):
        a.fill_(1.0)
        b.fill_(2.0)
        graph.replay()
    assert torch.equal(a, want[0]) and torch.equal(b, want[1])
    assert F.status_poll() == 0
