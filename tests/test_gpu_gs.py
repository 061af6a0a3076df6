"""Block Gauss-Seidel sweeps alone (no coarse stage) against the oracle's, forward,
backward and both, on node grids with odd and even edges down to two
elements (rows with most neighbours missing) and with missing entries in the
pattern: the sweeps keep every colour's blocks in padded groups.

The oracle forms v - A z before the backward sweep, the sweeps fold it into the
colours; the difference is roundoff amplified by the blocks' condition (contrast
e^2 here), 1e-10 relative in FP64 and 1e-4 with FP32 blocks."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from oracle import msrsb as O  # noqa: E402
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


@pytest.mark.parametrize("ne", [(1, 1, 2), (1, 4, 2), (4, 3, 5), (7, 6, 6), (12, 9, 8)], ids=str)
@pytest.mark.parametrize("pre,post", [(1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("thin", [False, True])
@pytest.mark.parametrize("prec", [0, 1])
def test_sweeps_match_the_oracle(M, ne, pre, post, thin, prec):
    c = elastic_3d_case(ne=ne, H=2)
    A = sp.bsr_matrix((c["data"], c["indices"], c["indptr"]))
    if thin:  # drop a third of the off-diagonal blocks
        r = np.repeat(np.arange(len(c["indptr"]) - 1), np.diff(c["indptr"]))
        keep = (r == c["indices"]) | (np.random.default_rng(1).uniform(size=len(r)) > 1 / 3)
        ptr = np.concatenate([[0], np.cumsum(np.bincount(r[keep], minlength=len(c["indptr"]) - 1))])
        A = sp.bsr_matrix((c["data"][keep], c["indices"][keep], ptr))
    h = M.msrsb_setup(M.Mat.from_host(A.indptr, A.indices, A.data, bdim=3),
                      M.grid(c["dims"], c["H"], centering=1, ncomp=3),
                      M.opts(smoother=M.msrsb.MSRSB_SMOOTH_GS, pre=pre, post=post, no_coarse=1, tol=0.0, max_iter=2,
                             krylov=M.msrsb.MSRSB_PCG, prec=prec))
    v = np.random.default_rng(2).standard_normal(A.shape[0])
    vd = torch.as_tensor(v, device="cuda")
    h.apply(torch.full_like(vd, float("nan")))  # what an earlier vector left behind must not matter
    z = h.apply(vd).cpu().numpy()
    h.destroy()
    col = O.parity_colours(c["dims"])
    S = A.tocsr()
    ref = np.zeros_like(v)
    if pre:
        ref = O.ColouredSmoother(S, col, "gs_fwd", bdim=3).solve(v)
    if post:
        ref = ref + O.ColouredSmoother(S, col, "gs_bwd", bdim=3).solve(v - S @ ref)
    assert np.linalg.norm(z - ref) <= (1e-10, 1e-4)[prec] * np.linalg.norm(ref)
