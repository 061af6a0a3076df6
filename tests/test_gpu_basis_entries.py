"""Entries of a basis built by msrsb_build_basis, one by one: small ones keep the
precision of their type, slots that no product has reached are exactly 0, and a
refused call leaves the caller's basis as it was.

Bound of an entry's relative error. With weights w_ik = omega |a_ik| / D_ii of an
M-matrix a pass is P_i' = (1 - omega) P_i + sum w_ik P_k, divided by its row's sum:
non-negative terms only, so relative errors of the inputs do not grow. It is
evaluated as P_i - (omega / D_ii) (D_ii P_i - sum |a_ik| P_k), whose terms add up to
at most (1 + omega) / (1 - omega) = 5 times the result; with up to 27 products, the
update and the scaling's 8 additions and division that is 5 (27 + 5) + 8 + 3 < 172
units of roundoff u = 2^-53 a pass."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from synth.darcy import darcy_2d_case, darcy_3d_case  # noqa: E402

pytestmark = pytest.mark.gpu

OMEGA = 2.0 / 3.0
CASES = {
    "3d": lambda: darcy_3d_case(dims=(20, 18, 13), H=(8, 6, 4)),
    "3d_sigma3": lambda: darcy_3d_case(dims=(33, 9, 17), H=(5, 4, 8), sigma=3.0, seed=4),
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


# blocks wide enough that the passes of the test below have not crossed them
FAR = {
    "3d_far": lambda: darcy_3d_case(dims=(39, 26, 13), H=(13, 13, 13), sigma=1.0, seed=4),
    "3d_far_sigma3": lambda: darcy_3d_case(dims=(39, 26, 13), H=(13, 13, 13), sigma=3.0, seed=4),
    "2d_far": lambda: darcy_2d_case(n=45, H=15),
}


def _inputs(M, case, prec):
    c = {**CASES, **FAR}[case]()
    A = M.Mat.from_host(c["indptr"], c["indices"], c["data"])
    ahat, _ = M.msrsb_filter(A)
    part, _, p_ids, skel = M.msrsb_partition(M.grid(c["dims"], c["H"]))
    dt = torch.float64 if prec == 0 else torch.float32
    P = ((p_ids >= 0) & (p_ids == part[:, None])).to(dt).contiguous()
    return M.Mat(A.rowptr, A.colidx, ahat), sp.csr_matrix((ahat.cpu().numpy(), c["indices"], c["indptr"])), p_ids, skel, P


def _reference(Ah, ids, P, passes):
    """The passes as sums of non-negative terms, in extended precision."""
    ld = np.longdouble
    n = ids.shape[0]
    rows = np.repeat(np.arange(n), np.diff(Ah.indptr))
    match = (ids[rows] == ids[Ah.indices]) & (ids[rows] >= 0)
    off = rows != Ah.indices
    d = np.zeros(n, dtype=ld)
    d[rows[~off]] = Ah.data[~off]
    w = np.where(off, -ld(OMEGA) * Ah.data.astype(ld) / np.where(d[rows] != 0, d[rows], 1), 0)
    P = np.where(ids >= 0, P, 0).astype(ld)
    keep = np.where(d != 0, 1 - ld(OMEGA), ld(1))[:, None]
    for _ in range(passes):
        T = keep * P
        np.add.at(T, rows, np.where(match, w[:, None] * P[Ah.indices], ld(0)))
        T[ids < 0] = 0
        P = T / T.sum(axis=1, keepdims=True)
    return P


def _run(M, Ah, p_ids, skel, P, prec, passes):
    it, _ = M.msrsb_build_basis(Ah, p_ids, skel, p_ids.shape[1], M.basis_opts(OMEGA, 0.0, 10, passes), prec, P)
    assert it == passes
    return P.cpu().numpy()


@pytest.mark.parametrize("case,passes", [(c, 30) for c in CASES] + [(c, 5) for c in FAR])
def test_small_entries_keep_their_precision(M, case, passes):
    Ah, Hh, p_ids, skel, P0 = _inputs(M, case, 0)
    ref = _reference(Hh, p_ids.cpu().numpy(), P0.cpu().numpy(), passes)
    P = _run(M, Ah, p_ids, skel, P0.clone(), 0, passes)
    on = ref > 0
    far = float(np.max(np.abs(P[on] - ref[on]) / ref[on]))
    print(case, "smallest entry %.3g, largest relative error %.3g" % (float(ref[on].min()), far))
    assert float(ref[on].min()) < (1e-9 if passes == 5 else 1e-3)  # there are small entries to look at
    assert far <= 172 * passes * 2.0 ** -53


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("case", list(CASES))
def test_unreached_slots_are_zero(M, case, prec):
    Ah, Hh, p_ids, skel, P0 = _inputs(M, case, prec)
    ids = p_ids.cpu().numpy()
    for passes in (1, 3):
        ref = _reference(Hh, ids, P0.cpu().numpy(), passes)
        P = _run(M, Ah, p_ids, skel, P0.clone(), prec, passes)
        assert np.any((ref == 0) & (ids >= 0))
        assert np.all(P[ref == 0] == 0)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bad", [dict(n_it=0), dict(max_iter=-1), dict(W=2)])
def test_a_refused_call_leaves_the_basis(M, prec, bad):
    Ah, _, p_ids, skel, P0 = _inputs(M, "3d", prec)
    o = dict(omega=OMEGA, tol=0.0, n_it=10, max_iter=12)
    W = bad.get("W", p_ids.shape[1])
    o.update({k: v for k, v in bad.items() if k != "W"})
    P = P0.clone()
    with pytest.raises(M.MsrsbError) as err:
        M.msrsb_build_basis(Ah, p_ids, skel, W, M.basis_opts(**o), prec, P)
    assert err.value.status == 1  # MSRSB_EINVAL
    torch.cuda.synchronize()
    assert torch.equal(P.view(torch.uint8), P0.view(torch.uint8))
