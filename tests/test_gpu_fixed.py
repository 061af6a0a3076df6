"""FP64 restricted smoothing in fixed point (M-matrix operators, relaxations up to
0.7, initial bases whose rows sum to 1) against the same passes in extended
precision on the host, beside the FP64 passes.

The FP64 passes are reached with twice the indicator as the initial basis: its
rows sum to 2, so the fixed-point passes do not take it, and the first pass's
rescaling removes the factor exactly. Both results are rounded to FP64 on return,
so the fixed-point result may be no further from the reference than the FP64 one.
What the fixed-point passes do not serve (positive off-diagonals, larger
relaxations, rows that do not sum to 1) is compared with the host in FP64: 1e-12
after 12 passes of sums of 27 products."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from synth.darcy import darcy_2d_case, darcy_3d_case  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    "3d": lambda: darcy_3d_case(dims=(20, 18, 13), H=(8, 6, 4)),
    "3d_sigma1": lambda: darcy_3d_case(dims=(33, 9, 17), H=(5, 4, 8), sigma=1.0, seed=4),
    "2d": lambda: darcy_2d_case(n=45, H=8),
}


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1912_06934_gb300 as M
    return M


def _host(Ah, ids, P, omega, passes, dt):
    """Alg. 1 passes on the host in dt: P (n, W) in colour slots."""
    n, W = ids.shape
    ip, ix = Ah.indptr, Ah.indices
    a = Ah.data.astype(dt)
    rows = np.repeat(np.arange(n), np.diff(ip))
    match = (ids[rows] == ids[ix]) & (ids[rows] >= 0)
    d = np.zeros(n, dtype=dt)
    d[rows[rows == ix]] = a[rows == ix]
    scale = np.where(d != 0, dt(omega) / np.where(d != 0, d, 1), 0)
    P = np.where(ids >= 0, P, 0).astype(dt)
    for _ in range(passes):
        acc = np.zeros((n, W), dtype=dt)
        np.add.at(acc, rows, np.where(match, a[:, None] * P[ix], dt(0)))
        P = np.where(ids >= 0, P - scale[:, None] * acc, 0)
        P = P / P.sum(axis=1, keepdims=True)
    return P


def _setup(M, c):
    A = M.Mat.from_host(c["indptr"], c["indices"], c["data"])
    ahat, _ = M.msrsb_filter(A)
    part, _, p_ids, skel = M.msrsb_partition(M.grid(c["dims"], c["H"]))
    P0 = ((p_ids >= 0) & (p_ids == part[:, None])).to(torch.float64).contiguous()
    return A, ahat, p_ids, skel, P0


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("omega", [2.0 / 3.0, 0.3])
def test_fixed_point_is_no_less_exact(M, case, omega):
    c = CASES[case]()
    A, ahat, p_ids, skel, P0 = _setup(M, c)
    Ah = M.Mat(A.rowptr, A.colidx, ahat)
    W, passes = p_ids.shape[1], 60
    out = []
    for f in (1.0, 2.0):
        P = (f * P0).contiguous()
        it, e = M.msrsb_build_basis(Ah, p_ids, skel, W, M.basis_opts(omega, 0.0, 10, passes), 0, P)
        assert it == passes
        out.append((P.cpu().numpy(), e))
    ids = p_ids.cpu().numpy()
    Hh = sp.csr_matrix((ahat.cpu().numpy(), c["indices"], c["indptr"]))
    ref = _host(Hh, ids, P0.cpu().numpy(), omega, passes, np.longdouble)
    far = [float(np.sqrt(((P - ref) ** 2).sum())) for P, _ in out]
    big = [float(np.abs(P - ref).max()) for P, _ in out]
    print(case, omega, "2-norm of the error: fixed %.3g FP64 %.3g; largest %.3g %.3g" % (*far, *big))
    assert far[0] <= far[1] and big[0] <= big[1]
    assert abs(out[0][1] - out[1][1]) <= 1e-14
    assert np.all(out[0][0][ids < 0] == 0.0)


@pytest.mark.parametrize("what", ["unfiltered", "omega", "rows"])
def test_other_inputs_keep_the_floating_passes(M, what):
    c = darcy_3d_case(dims=(20, 18, 13), H=(8, 6, 4))
    A, ahat, p_ids, skel, P0 = _setup(M, c)
    omega = 0.9 if what == "omega" else 0.5
    if what == "rows":
        P0 = (P0 + 0.25 * torch.rand(P0.shape, device="cuda", dtype=torch.float64)) * (p_ids >= 0)
    val = A.val if what == "unfiltered" else ahat
    P = P0.clone()
    M.msrsb_build_basis(M.Mat(A.rowptr, A.colidx, val), p_ids, skel, p_ids.shape[1],
                        M.basis_opts(omega, 0.0, 10, 12), 0, P)
    ref = _host(sp.csr_matrix((val.cpu().numpy(), c["indices"], c["indptr"])), p_ids.cpu().numpy(), P0.cpu().numpy(),
                omega, 12, np.float64)
    assert np.abs(P.cpu().numpy() - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())
