"""Line-block ILU(0) sweeps on the shapes where their layout can go wrong: lines
of one point less and more than a warp's segments, single lines and blocks,
odd heights and depths, patterns with missing entries (the sweeps store a
coefficient for every stencil offset, zero where the pattern has none).

One application of the smoother alone (no coarse stage) against the oracle's
sequential substitution in the same order. The matrices are diagonally dominant
(each row's off-diagonals sum to half its diagonal), so the substitutions
contract and the error stays a small multiple of the unit roundoff: 1e-10
relative in FP64 (as every application is checked), 1e-5 with FP32 factors (27
products a row of roundoff 6e-8 each, a factor of 6 in hand)."""
import itertools

import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from oracle import msrsb as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1912_06934_gb300 as M
    return M


def _matrix(dims, keep, seed):
    """Non-symmetric stencil matrix: every neighbour entry is there with
    probability `keep`, off-diagonals negative, rows diagonally dominant."""
    rng = np.random.default_rng(seed)
    d, n = len(dims), int(np.prod(dims))
    pos = np.indices(dims).reshape(d, -1, order="F")
    st = np.cumprod((1,) + tuple(dims[:-1]))
    rows, cols, vals = [], [], []
    for o in itertools.product((-1, 0, 1), repeat=d):
        if not any(o):
            continue
        ok = (rng.uniform(size=n) < keep)
        for a in range(d):
            ok &= (pos[a] + o[a] >= 0) & (pos[a] + o[a] < dims[a])
        i = np.nonzero(ok)[0]
        rows.append(i)
        cols.append(i + int(np.dot(o, st)))
        vals.append(-rng.uniform(0.1, 1.0, size=len(i)))
    A = sp.csr_matrix((np.concatenate(vals), (np.concatenate(rows), np.concatenate(cols))), shape=(n, n))
    A = (A + sp.diags(2.0 * np.asarray(abs(A).sum(axis=1)).ravel() + 0.1)).tocsr()
    A.sort_indices()
    return A


DIMS = [(64, 64), (33, 7), (31, 5), (256, 6), (200, 3), (5, 1), (64, 6, 5), (63, 5, 7), (65, 4, 4), (97, 5, 3),
        (128, 3, 5), (129, 4, 3), (193, 3, 3), (256, 5, 4), (1, 6, 5), (2, 9, 1), (40, 1, 6)]


@pytest.mark.parametrize("dims", DIMS, ids=str)
@pytest.mark.parametrize("keep", [1.0, 0.4])
@pytest.mark.parametrize("prec", [0, 1])
def test_sweeps_match_the_oracle(M, dims, keep, prec):
    A = _matrix(dims, keep, 3 + sum(dims))
    h = M.msrsb_setup(M.Mat.from_host(A.indptr, A.indices, A.data), M.grid(dims, (8,) * len(dims)),
                      M.opts(prec=prec, no_coarse=1, tol=0.0, max_iter=2))
    v = np.random.default_rng(7).standard_normal(A.shape[0])
    z = h.apply(torch.as_tensor(v, device="cuda")).cpu().numpy()
    h.destroy()
    order, colour, _, _ = O.line_block_order(dims)
    zr = O.ColouredSmoother(A, colour, "ilu0", order=order).solve(v)
    assert np.linalg.norm(z - zr) <= (1e-10, 1e-5)[prec] * np.linalg.norm(zr)


@pytest.mark.parametrize("dims", [(100, 6), (33, 5, 6), (96, 4, 5), (128, 5, 3)], ids=str)
@pytest.mark.parametrize("prec,k", [(0, 3), (1, 2), (1, 5)])
def test_lockstep_sweeps_equal_single_ones(M, dims, prec, k):
    A = _matrix(dims, 0.8, 11)
    h = M.msrsb_setup(M.Mat.from_host(A.indptr, A.indices, A.data), M.grid(dims, (8,) * len(dims)),
                      M.opts(prec=prec, tol=1e-3, max_iter=20))
    B = torch.as_tensor(np.random.default_rng(5).standard_normal((k, A.shape[0])), device="cuda")
    out = h.solve_multi(B, rtol=1e-8, maxit=100)
    for r in range(k):
        one = h.solve(B[r].clone(), rtol=1e-8, maxit=100)
        assert out["iters"][r] == one["iters"] and torch.equal(out["x"][r], one["x"])
    h.destroy()
