"""Galerkin product and kept entries of the smoothing on the forms their kernels take
apart: FP32 and FP64 bases, one and three components, two and three dimensions, bases
that do not start on a 16-byte boundary, coarse blocks cut short by the grid; operators
whose rows are too long to stage (a stencil of 81 points).

Sums of at most a few thousand FP64 products of one sign pattern per entry: 1e-12 of the
largest entry. The FP32 basis is exact in FP64, so the bound is the same. The smoothing
on the long rows runs 6 passes of sums of at most 81 products: 1e-12."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from synth.darcy import darcy_2d_case, darcy_3d_case  # noqa: E402
from synth.elastic import elastic_3d_case  # noqa: E402
from test_gpu_fixed import _host  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1912_06934_gb300 as M
    return M


CASES = {
    "3d": lambda: darcy_3d_case(dims=(21, 13, 10), H=(8, 5, 4)),
    "2d": lambda: darcy_2d_case(n=37, H=8),
    "elastic": lambda: elastic_3d_case(ne=7, H=4),
}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shift", [0, 1])
def test_coarse_operator(M, case, prec, shift):
    c = CASES[case]()
    bd = c["ncomp"]
    g = M.grid(c["dims"], c["H"], centering=c["centering"], ncomp=bd)
    A = M.Mat.from_host(c["indptr"], c["indices"], c["data"], bdim=bd)
    o = M.opts(tol=0.0, max_iter=8, **(dict(smoother=M.msrsb.MSRSB_SMOOTH_GS, pre=1, post=1) if bd == 3 else {}))
    h = M.msrsb_setup(A, g, o)
    ids, P, _ = h.get_setup()
    h.destroy()
    P = P.to(torch.float32 if prec else torch.float64)
    buf = torch.zeros(P.numel() + shift, dtype=P.dtype, device="cuda")
    Ps = buf[shift:]
    Ps.copy_(P.reshape(-1))
    rowptr, colidx, val = M.msrsb_coarse_op(A, g, ids, Ps, prec)
    ids, P = ids.cpu().numpy(), P.double().cpu().numpy()
    nc = len(rowptr) - 1
    r, s = np.nonzero(ids >= 0)
    Pf = sp.csr_matrix((np.concatenate([P[l][r, s] for l in range(bd)]),
                        (np.concatenate([bd * r + l for l in range(bd)]),
                         np.concatenate([bd * ids[r, s] + l for l in range(bd)]))), shape=(ids.shape[0] * bd, nc * bd))
    n = ids.shape[0] * bd
    Af = (sp.csr_matrix((c["data"], c["indices"], c["indptr"]), shape=(n, n)) if bd == 1 else
          sp.bsr_matrix((np.asarray(c["data"]).reshape(-1, 3, 3), c["indices"], c["indptr"]), shape=(n, n)).tocsr())
    ref = (Pf.T @ Af @ Pf).toarray()
    got = sp.bsr_matrix((val.cpu().numpy(), colidx.cpu().numpy(), rowptr.cpu().numpy()),
                        shape=(nc * bd, nc * bd)).toarray()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("dims", [(40, 23), (9, 64)], ids=str)
def test_smoothing_of_long_rows(M, dims):
    nx, ny = dims
    n = nx * ny
    rng = np.random.default_rng(2)
    y, x = np.divmod(np.arange(n), nx)
    rows, cols = [], []
    for dy in range(-4, 5):
        for dx in range(-4, 5):
            ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny)
            rows.append(np.nonzero(ok)[0])
            cols.append(rows[-1] + dx + nx * dy)
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    A = sp.csr_matrix((np.where(rows == cols, 0.0, -rng.uniform(0.1, 1.0, len(rows))), (rows, cols)), shape=(n, n))
    A = (A - sp.diags(np.asarray(A.sum(axis=1)).ravel())).tocsr()
    A.sort_indices()
    g = M.grid(dims, (8, 8))
    _, _, ids, skel = M.msrsb_partition(g)
    W = ids.shape[1]
    part = ids.cpu().numpy()
    P0 = np.where(part >= 0, 1.0, 0.0) / np.maximum((part >= 0).sum(axis=1, keepdims=True), 1)
    P = torch.as_tensor(P0, device="cuda").contiguous()
    M.msrsb_build_basis(M.Mat.from_host(A.indptr, A.indices, A.data), ids, skel, W, M.basis_opts(0.9, 0.0, 10, 6), 0, P)
    ref = _host(A, part, P0, 0.9, 6, np.float64)
    assert np.abs(P.cpu().numpy() - ref).max() <= 1e-12
