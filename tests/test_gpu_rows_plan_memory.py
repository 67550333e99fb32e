"""The row plan's device memory: what the header states, from the plan's own counts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synthetic import mesh as M  # noqa: E402
from synthetic import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [1, 4])
def test_device_bytes(q):
    """Per cell n_local (2 n_local + 4) bytes of pairs and positions and eight doubles of geometry
    scratch; per dof 8 bytes; the rest (chunk tables, class runs, alignment) below 1 KB a chunk."""
    import paper_1112_0402_gb300 as F

    p = W.make_problem(M.unit_cube_tets(4, 0.15, 3), W.MASS, q)
    rp, col, _ = F.csr_pattern(p.dofmap, p.n_dof, with_slots=False)
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    plan = F.RowPlan(dev(p.dofmap), p.n_dof, dev(rp), dev(col))
    n_elem, n = p.dofmap.shape
    least = n_elem * (n * (2 * n + 4) + 64) + p.n_dof * 8
    assert least <= plan.device_bytes <= least + plan.n_chunks * 1024 + 64
