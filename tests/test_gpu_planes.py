"""Coarse solver over planes on plane sizes where its factorisation can go
wrong: fewer columns than CTAs in a cluster, one more and one less than a warp's
or a CTA's rows, several rows per thread, one or two planes, 2D, 3x3 blocks.

With the smoother off, one application is P A_c^-1 P^T v; it is compared with a
host solve with the A_c and P of the same set-up (msrsb_get_setup). The scalar
operators are diagonally dominant (off-diagonals sum to half the diagonal), so
A_c is well conditioned and two backward stable solves agree to a small multiple
of roundoff: 1e-11. The elastic block's A_c has a condition number below 1e6
(12 coarse steps, contrast e^2): 1e-9."""
import itertools

import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from synth.elastic import elastic_3d_case  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1912_06934_gb300 as M
    return M


def _matrix(dims, seed):
    rng = np.random.default_rng(seed)
    d, n = len(dims), int(np.prod(dims))
    pos = np.indices(dims).reshape(d, -1, order="F")
    st = np.cumprod((1,) + tuple(dims[:-1]))
    rows, cols, vals = [], [], []
    for o in itertools.product((-1, 0, 1), repeat=d):
        if not any(o):
            continue
        ok = np.ones(n, dtype=bool)
        for a in range(d):
            ok &= (pos[a] + o[a] >= 0) & (pos[a] + o[a] < dims[a])
        i = np.nonzero(ok)[0]
        rows.append(i)
        cols.append(i + int(np.dot(o, st)))
        vals.append(-rng.uniform(0.1, 1.0, size=len(i)))
    A = sp.csr_matrix((np.concatenate(vals), (np.concatenate(rows), np.concatenate(cols))), shape=(n, n))
    A = (A + sp.diags(2.0 * np.asarray(abs(A).sum(axis=1)).ravel())).tocsr()
    A.sort_indices()
    return A


def _check(M, h, bd, tol, seed):
    ids, P, Ac = (t.cpu().numpy() for t in h.get_setup())
    n = ids.shape[0]
    v = np.random.default_rng(seed).standard_normal(n * bd)
    z = h.apply(torch.as_tensor(v, device="cuda")).cpu().numpy()
    r, s = np.nonzero(ids >= 0)
    Pf = sp.csr_matrix((np.concatenate([P[l][r, s] for l in range(bd)]),
                        (np.concatenate([bd * r + l for l in range(bd)]),
                         np.concatenate([bd * ids[r, s] + l for l in range(bd)]))), shape=(n * bd, Ac.shape[0]))
    ref = Pf @ np.linalg.solve(Ac, Pf.T @ v)
    assert np.linalg.norm(z - ref) <= tol * np.linalg.norm(ref)


# coarse nodes per axis; the plane is all but the last
@pytest.mark.parametrize("nb", [(1, 2), (5, 1), (16, 3), (33, 4), (640, 3), (1, 1, 2), (3, 5, 3), (17, 1, 4), (8, 8, 3),
                                (13, 5, 4), (43, 3, 3), (16, 16, 3), (19, 14, 4), (22, 18, 3), (24, 25, 2)], ids=str)
def test_plane_solver_matches_host(M, nb):
    dims = tuple(2 * b for b in nb)
    A = _matrix(dims, 5)
    h = M.msrsb_setup(M.Mat.from_host(A.indptr, A.indices, A.data), M.grid(dims, (2,) * len(nb)),
                      M.opts(smoother=M.msrsb.MSRSB_SMOOTH_NONE, post=0, tol=0.0, max_iter=5))
    _check(M, h, 1, 1e-11, 6)
    h.destroy()


@pytest.mark.parametrize("ne,H", [((9, 7, 6), 3), ((24, 18, 12), 3)], ids=str)
def test_plane_solver_matches_host_elastic(M, ne, H):
    c = elastic_3d_case(ne=ne, H=H)
    h = M.msrsb_setup(M.Mat.from_host(c["indptr"], c["indices"], c["data"], bdim=3),
                      M.grid(c["dims"], c["H"], centering=1, ncomp=3),
                      M.opts(smoother=M.msrsb.MSRSB_SMOOTH_NONE, post=0, tol=0.0, max_iter=5,
                             krylov=M.msrsb.MSRSB_PCG))
    _check(M, h, 3, 1e-9, 7)
    h.destroy()


# more than 1024 coarse unknowns, where the plane factors are kept and applied (not
# the explicit inverse): planes of 1 and 3 rows, odd rows (no 16-byte copies), rows
# that do not fit the staged copies, chains of many planes. Tolerance as above.
@pytest.mark.parametrize("nb", [(1, 1030), (3, 345), (11, 11, 9), (27, 5, 8), (16, 13, 5), (258, 4), (520, 5)], ids=str)
def test_kept_planes_match_host(M, nb):
    dims = tuple(2 * b for b in nb)
    A = _matrix(dims, 7)
    h = M.msrsb_setup(M.Mat.from_host(A.indptr, A.indices, A.data), M.grid(dims, (2,) * len(nb)),
                      M.opts(smoother=M.msrsb.MSRSB_SMOOTH_NONE, post=0, tol=0.0, max_iter=5))
    _check(M, h, 1, 1e-11, 8)
    h.destroy()
