"""The end of a GMRES cycle (the triangular solves that give the update, several rows a
thread beyond 256 columns) and the scaling of its first vector.

A weak preconditioner makes cycles long. A wrong update would leave the true residual
above the estimate that ended the cycle, so that the solver would need another one: with
a restart length above the iterations needed, the solve must end in its first cycle with
a true residual within rtol (the solver's own test), which is formed again here in FP64:
2 rtol leaves room for its rounding (the operator's condition number times 1e-16 is
below rtol). Scaling b by a power of two scales every quantity exactly, so that the
solution must be the scaled one bit for bit."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from synth.darcy import darcy_3d_case  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1912_06934_gb300 as M
    return M


@pytest.mark.parametrize("dims,restart", [((16, 16, 16), 200), ((24, 24, 24), 512)])
def test_cycle_update(M, dims, restart):
    c = darcy_3d_case(dims=dims, H=8, seed=9)
    A = sp.csr_matrix((c["data"], c["indices"], c["indptr"]))
    h = M.msrsb_setup(M.Mat.from_host(c["indptr"], c["indices"], c["data"]), M.grid(c["dims"], c["H"]),
                      M.opts(smoother=M.msrsb.MSRSB_SMOOTH_L1JAC, no_coarse=1, restart=restart, tol=0.0, max_iter=2))
    b = A @ np.random.default_rng(4).standard_normal(A.shape[0])
    out = h.solve(torch.as_tensor(b, device="cuda"), rtol=1e-9, maxit=2000)
    x = out["x"].cpu().numpy()
    assert np.linalg.norm(b - A @ x) <= 2e-9 * np.linalg.norm(b)
    assert (256 if restart == 512 else 32) < out["iters"] <= restart
    big = h.solve(torch.as_tensor(b * 2.0 ** 40, device="cuda"), rtol=1e-9, maxit=2000)
    assert big["iters"] == out["iters"] and np.array_equal(big["x"].cpu().numpy(), x * 2.0 ** 40)
    h.destroy()
