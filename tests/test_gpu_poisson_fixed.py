"""FP64 Poisson element tensors, whose contraction runs in fixed point: every entry against
A0 : G_K in extended precision, on both sides of the rule that sends stretched cells to the
FP64 multiply-adds, at the sizes where tiles and chunks end.

Bound per entry: the FP64 geometry errs by a few ulps of |K_a||K_b||det J| per G entry (the
cells are a jittered simplex times powers of two, which scale J exactly, so its conditioning
is that of the unstretched cell: cofactor, determinant and product roundings, below 32
ulps), and the contraction by at most 7 ulps of the sum of |terms|; 64 * 2^-53 covers both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from synthetic import mesh as M  # noqa: E402

pytestmark = pytest.mark.gpu


def _cells(d, n_elem, stretch, scale, seed=11):
    """n_elem jittered simplices (their own vertices each), axes scaled by powers of two."""
    m = M.unit_square_triangles(8, 0.2, seed) if d == 2 else M.unit_cube_tets(4, 0.15, seed)
    x = m.vertices[m.cells[np.arange(n_elem) % m.n_elem]]  # [E, d+1, d]
    x = x * (np.array(stretch[:d], dtype=np.float64) * scale)
    ids = np.arange(n_elem * (d + 1), dtype=np.int32).reshape(n_elem, d + 1)
    return ids, np.ascontiguousarray(x.reshape(-1, d))


def _reference(form, ids, verts):
    """A0 : G_K in extended precision and the bound's sums of |terms|."""
    d = form.dim
    x = verts[ids].astype(np.longdouble)
    J = (x[:, 1:] - x[:, :1]).transpose(0, 2, 1)
    if d == 2:
        adj = np.stack([np.stack([J[:, 1, 1], -J[:, 0, 1]], -1), np.stack([-J[:, 1, 0], J[:, 0, 0]], -1)], -2)
    else:
        adj = np.stack([np.cross(J[:, :, (a + 1) % 3], J[:, :, (a + 2) % 3]) for a in range(3)], 1)
    det = np.einsum("er,er->e", adj[:, 0], J[:, :, 0])
    K = adj / det[:, None, None]
    G = np.abs(det)[:, None, None] * np.einsum("eab,ecb->eac", K, K)
    norm = np.sqrt(np.einsum("eab,eab->ea", K, K))
    B = np.abs(det)[:, None, None] * norm[:, :, None] * norm[:, None, :]
    # A0 as the kernels hold it: symmetric columns (a, b) + (b, a) summed, entries i1 <= i2
    # mirrored (its rounding noise on entries that are zero in exact arithmetic included)
    n = form.n_local
    A0 = form.reference_tensor().reshape(n, n, d, d)
    A0 = np.stack([A0[:, :, a, b] + (A0[:, :, b, a] if a != b else 0.0) for a in range(d) for b in range(a, d)])
    A0 = (np.triu(A0) + np.triu(A0, 1).transpose(0, 2, 1)).astype(np.longdouble)
    pairs = [(a, b) for a in range(d) for b in range(a, d)]
    ref = sum(G[:, a, b, None, None] * A0[k] for k, (a, b) in enumerate(pairs))
    return ref, sum(B[:, a, b, None, None] * np.abs(A0[k]) for k, (a, b) in enumerate(pairs))


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("q", [1, 2, 3, 4])
@pytest.mark.parametrize("stretch,scale", [((1, 1, 1), 1.0), ((1, 2, 4), 1.0), ((1, 1, 8), 2.0 ** -60),
                                           ((1, 16, 1), 2.0 ** 60), ((1, 1024, 32), 1.0), ((1, 1, 1), 2.0 ** -300)])
def test_every_entry(d, q, stretch, scale):
    import paper_1112_0402_gb300 as F

    form = F.Form(F.POISSON, F.TRIANGLE if d == 2 else F.TETRAHEDRON, q)
    ids, verts = _cells(d, 133, stretch, scale)
    A = F.tabulate(form, torch.as_tensor(ids, device="cuda"), torch.as_tensor(verts, device="cuda")).cpu().numpy()
    # the degeneracy test squares edge lengths in FP32: cells of 2^-300 are below its range
    # and flagged, their values are as computed
    assert F.status_poll() == (F.FLAG_DEGENERATE if scale < 2.0 ** -100 else 0)
    ref, bound = _reference(form, ids, verts)
    assert (np.abs(A - ref) <= 64 * 2.0 ** -53 * bound).all()
    assert (A == A.transpose(0, 2, 1)).all()


@pytest.mark.parametrize("d,q,n_elem", [(2, 1, 1), (2, 1, 125), (2, 4, 97), (3, 1, 101), (3, 2, 95), (3, 3, 7),
                                        (3, 4, 1), (3, 4, 97)])
def test_chunk_ends_and_assembly(d, q, n_elem):
    """Ragged tiles and chunks; nothing past the last cell is written; the assembly adds the
    tabulated values (exactly: every slot receives one value); a bad slot is skipped."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.POISSON, F.TRIANGLE if d == 2 else F.TETRAHEDRON, q)
    n = form.n_local
    ids, verts = _cells(d, n_elem, (1, 1, 1), 1.0)
    c, v = torch.as_tensor(ids, device="cuda"), torch.as_tensor(verts, device="cuda")
    whole = torch.full((n_elem + 1, n, n), 7.0, dtype=torch.float64, device="cuda")
    A = F.tabulate(form, c, v, out=whole[:n_elem])
    assert (whole[n_elem] == 7.0).all()
    ref, bound = _reference(form, ids, verts)
    assert (np.abs(A.cpu().numpy() - ref) <= 64 * 2.0 ** -53 * bound).all()
    nnz = n_elem * n * n
    slot = torch.randperm(nnz, generator=torch.Generator().manual_seed(3)).to(torch.int32).reshape(n_elem, n, n).cuda()
    val = torch.zeros(nnz, dtype=torch.float64, device="cuda")
    F.assemble(form, c, v, slot, val)
    assert F.status_poll() == 0
    assert torch.equal(val[slot.long().reshape(-1)], A.reshape(-1))
    slot[0, 0, 0] = nnz
    val.zero_()
    F.assemble(form, c, v, slot, val)
    assert F.status_poll() == F.FLAG_BOUNDS
    assert torch.equal(val[slot.long().reshape(-1)[1:]], A.reshape(-1)[1:])


def test_degenerate_and_stretched_cells_beside_regular_ones():
    """A flat cell gives non-finite values and the flag; its neighbours in the tile, regular
    and stretched, keep theirs."""
    import paper_1112_0402_gb300 as F

    form = F.Form(F.POISSON, F.TETRAHEDRON, 2)
    ids, verts = _cells(3, 40, (1, 1, 1), 1.0)
    verts[ids[5]] *= np.array([1.0, 64.0, 1.0])
    verts[ids[9], 2] = 0.25
    c, v = torch.as_tensor(ids, device="cuda"), torch.as_tensor(verts, device="cuda")
    A = F.tabulate(form, c, v).cpu().numpy()
    assert F.status_poll() == F.FLAG_DEGENERATE
    assert not np.isfinite(A[9]).any()
    live = np.arange(40) != 9
    ref, bound = _reference(form, ids[live], verts)
    assert (np.abs(A[live] - ref) <= 64 * 2.0 ** -53 * bound).all()
