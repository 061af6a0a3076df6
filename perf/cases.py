"""Cases that stand for the work a user has this framework do: building the
coarse space, setting up the two-level preconditioner, applying it, solving
with it (one right-hand side, several, from host memory) and differentiating
the Darcy model through it, in 2D and 3D, on pressure (scalar, MPFA-O) and
displacement (3x3 block, Q1 elements) operators, in both precisions.

Operators are assembled here with torch in 64 bits from a seeded coefficient
field: MPFA-O on unit cells (2D: pressure fixed left and right; 3D: no flow
outside and a well in two opposite corners) and Q1 hexahedral elasticity
(bottom fixed, unit traction on top), the inputs of this repository's own
workloads. All grids are x fastest.
"""
import itertools
import math

import numpy as np
import torch

import paper_1912_06934_gb300 as M
from paper_1912_06934_gb300.adjoint import msrsb_mpfa_solve_diff

B = M.msrsb
DEV = "cuda"
F64 = torch.float64
OMEGA, TOL, N_IT, MAX_PASSES = 2.0 / 3.0, 1e-3, 10, 100  # Alg. 1 as the workloads run it
RTOL, MAXIT = 1e-8, 500


def _case(name, kind, model, dims, h, prec, sigma=0.0, nrhs=1):
    c = dict(kind=kind, model=model, nx=dims[0], ny=dims[1], nz=dims[2] if len(dims) == 3 else 1, h=h, prec=prec,
             sigma=sigma, nrhs=nrhs)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one application inside a user's own Krylov method on the smallest
        # workload: launches and dependent steps only
        _case("apply_darcy2d_64_f64", "apply", "darcy2d", (64, 64), 8, "f64"),
        # a small plane problem, solved again and again with a kept handle
        _case("solve_darcy2d_100x140_f64", "solve", "darcy2d", (100, 140), 5, "f64"),
        # the coarse space alone (filter, restricted smoothing, Galerkin
        # product) on a grid that the blocks do not divide
        _case("coarse_space_darcy3d_61x47x53_f64", "basis", "darcy3d", (61, 47, 53), 8, "f64", 3.0),
        # the headline workload: set-up in the mixed form ...
        _case("setup_darcy3d_64_mixed", "setup", "darcy3d", (64, 64, 64), 8, "mixed", 3.0),
        # ... and the whole call from and to host buffers, as a simulator that
        # keeps its matrices on the host makes it
        _case("host_darcy3d_64_mixed", "host", "darcy3d", (64, 64, 64), 8, "mixed", 3.0),
        # the plain 64-bit form of it, the default precision
        _case("solve_darcy3d_64_f64", "solve", "darcy3d", (64, 64, 64), 8, "f64", 3.0),
        # the largest flow problem: a new operator, and one more right-hand
        # side for a kept one (a time step)
        _case("setup_darcy3d_128_mixed", "setup", "darcy3d", (128, 128, 128), 8, "mixed", 2.0),
        _case("solve_darcy3d_128_mixed", "solve", "darcy3d", (128, 128, 128), 8, "mixed", 2.0),
        # mechanics, 352,947 unknowns: block Gauss-Seidel and PCG
        _case("setup_elastic_48_mixed", "setup", "elastic", (48, 48, 48), 6, "mixed"),
        _case("solve_elastic_48_mixed", "solve", "elastic", (48, 48, 48), 6, "mixed"),
        # an ensemble member: 8 right-hand sides of one operator together
        _case("multi8_darcy3d_80_mixed", "multi", "darcy3d", (80, 80, 80), 8, "mixed", 3.0, 8),
        # inversion for ln k: assembly, forward solve, adjoint solve, gradient
        _case("adjoint_darcy3d_64_f64", "adjoint", "darcy3d", (64, 64, 64), 8, "f64", 2.0),
    ]


def draw(rng):
    def edge(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def edges3(lo, hi):
        e = edge(lo, hi)  # the axes within a factor of about 1.3 of one another
        return tuple(max(lo, min(hi, int(round(e * rng.uniform(0.87, 1.13))))) for _ in range(3))

    kind = rng.choice(["apply", "solve2", "solve3", "solve3", "solve_el", "basis", "setup", "setup", "setup_el",
                       "host", "multi", "adjoint"])
    prec = rng.choice(["f64", "mixed"])
    h3 = rng.choice([6, 8, 8, 10])
    sigma = round(rng.uniform(1.0, 3.0), 2)
    if prec == "mixed" and kind in ("solve3", "setup"):
        h3 = max(h3, 8)  # on the largest grids smaller blocks make another problem of the coarse system
    if kind == "apply":
        return _case(None, kind, "darcy2d", (edge(32, 250), edge(32, 250)), rng.randint(4, 10), "f64")
    if kind == "solve2":
        return _case(None, "solve", "darcy2d", (edge(32, 250), edge(32, 250)), rng.randint(4, 10), prec)
    if kind == "solve3":
        return _case(None, "solve", "darcy3d", edges3(20, 126 if prec == "mixed" else 90), h3, prec, sigma)
    if kind in ("solve_el", "setup_el"):
        return _case(None, kind[:5], "elastic", edges3(8, 47), rng.choice([4, 6, 6]) if kind == "solve_el" else 6, prec)
    if kind == "basis":
        return _case(None, kind, "darcy3d", edges3(16, 64), h3, prec, sigma)
    if kind == "setup":
        return _case(None, kind, "darcy3d", edges3(20, 126 if prec == "mixed" else 90), h3, prec, sigma)
    if kind == "host":
        return _case(None, kind, "darcy3d", edges3(20, 80), h3, prec, sigma)
    if kind == "multi":
        return _case(None, kind, "darcy3d", edges3(20, 78), h3, "mixed", sigma, rng.randint(2, 8))
    return _case(None, kind, "darcy3d", edges3(16, 62), h3, prec, min(sigma, 2.0))


# ---- inputs --------------------------------------------------------------------


def _cells(case):
    """Cells (or elements) per axis, x first."""
    return (case["nx"], case["ny"]) if case["model"] == "darcy2d" else (case["nx"], case["ny"], case["nz"])


def _points(case):
    """Fine points per axis: cells, or the nodes of the elements."""
    c = _cells(case)
    return tuple(e + 1 for e in c) if case["model"] == "elastic" else c


def _bdim(case):
    return 3 if case["model"] == "elastic" else 1


def _field(dims, corr, gen):
    """Gaussian random field of unit variance, covariance exp(-(r/corr)^2),
    shape dims reversed (x last): white noise on a padded box, convolved with
    exp(-2 x^2 / corr^2)."""
    pad = int(math.ceil(3 * corr))
    big = [d + 2 * pad for d in reversed(dims)]
    w = torch.fft.fftn(torch.randn(big, generator=gen, device=DEV, dtype=F64))
    for ax, size in enumerate(big):
        t = torch.arange(size, device=DEV, dtype=F64)
        t = torch.minimum(t, size - t)
        k = torch.where(t <= pad, torch.exp(-2.0 * t * t / (corr * corr)), torch.zeros_like(t))
        w = w * torch.fft.fft(k).reshape([-1 if a == ax else 1 for a in range(len(big))])
    f = torch.fft.ifftn(w).real[tuple(slice(pad, pad + d) for d in reversed(dims))]
    f = f - f.mean()
    return (f / f.std()).contiguous()


def _tensor(d):
    """The unit permeability tensor: 10:1 along rotated axes."""
    if d == 2:
        a = math.radians(30.0)
        R = np.array([[math.cos(a), -math.sin(a)], [math.sin(a), math.cos(a)]])
        return R @ np.diag([1.0, 0.1]) @ R.T
    a, b = math.radians(20.0), math.radians(35.0)
    R = np.array([[math.cos(a), -math.sin(a), 0], [math.sin(a), math.cos(a), 0], [0, 0, 1]]) @ \
        np.array([[math.cos(b), 0, math.sin(b)], [0, 1, 0], [-math.sin(b), 0, math.cos(b)]])
    return R @ np.diag([1.0, 1.0, 0.1]) @ R.T


def _log_k(case, seed):
    """ln k per cell, flat, x fastest."""
    gen = torch.Generator(DEV).manual_seed(seed)
    dims = _cells(case)
    if case["model"] == "darcy2d":
        return torch.randn(int(np.prod(dims)), generator=gen, device=DEV, dtype=F64)
    return case["sigma"] * _field(dims, 8.0, gen).reshape(-1)


def _shift(dims, off, lo, hi):
    """Slices of an array over dims (x last) for index + off, lo..hi kept."""
    return tuple(slice(lo + o, d + hi + o) for d, o in zip(reversed(dims), reversed(off)))


def _eliminate(C, R):
    """C^-1 R for many small systems; C is symmetric definite up to the sign
    of its rows, so no row exchanges are needed."""
    m = C.shape[-1]
    rows = [torch.cat((C[:, i], R[:, i]), 1) for i in range(m)]
    for k in range(m):
        rows[k] = rows[k] / rows[k][:, k:k + 1]
        for i in range(m):
            if i != k:
                rows[i] = rows[i] - rows[i][:, k:k + 1] * rows[k]
    return torch.stack([r[:, m:] for r in rows], 1)


def _mpfa(dims, logk, walls):
    """MPFA-O on unit cells, K = exp(ln k) times the unit tensor: stencil
    values (n, 3^d) and b (n). In the region of the 2^d cells around a vertex
    the pressure is linear per cell, through its pressure and the potentials at
    its d half-faces; flux continuity there eliminates the potentials. `walls`:
    pressure 1 at x = 0 and 0 at the far x side; no flow elsewhere."""
    d = len(dims)
    slots = list(itertools.product((0, 1), repeat=d))  # offsets (x first) of a region's cells
    at = {o: c for c, o in enumerate(slots)}
    nv = tuple(e + 1 for e in dims)
    V = int(np.prod(nv))
    K = torch.as_tensor(_tensor(d), device=DEV)
    pad = [1, 1] * d
    ek = torch.nn.functional.pad(torch.exp(logk).reshape(dims[::-1]), pad)
    has = torch.nn.functional.pad(torch.ones(dims[::-1], device=DEV, dtype=F64), pad)

    def view(a, o):  # cell (vertex - 1 + o) for every vertex
        return a[tuple(slice(q, q + e) for q, e in zip(reversed(o), reversed(nv)))].reshape(-1)

    sign = [[1.0 if q == 0 else -1.0 for q in o] for o in slots]
    on = [view(has, o) > 0 for o in slots]
    # flux of slot s across its half-face normal to a: sum_b U[s][a][b] (u_b - p_s)
    U = [[[-(0.5 ** (d - 2)) * view(ek, o) * K[a, b] * sign[s][b] for b in range(d)] for a in range(d)]
         for s, o in enumerate(slots)]
    faces, face_of = [], {}
    for a in range(d):
        for q in itertools.product((0, 1), repeat=d - 1):
            m, p = at[q[:a] + (0,) + q[a:]], at[q[:a] + (1,) + q[a:]]
            face_of[m, a] = face_of[p, a] = len(faces)
            faces.append((a, m, p))
    nf, nc = len(faces), len(slots)
    zero = torch.zeros(V, device=DEV, dtype=F64)
    C = [[zero] * nf for _ in range(nf)]
    R = [[zero] * (nc + 1) for _ in range(nf)]  # right-hand sides: the cells' pressures, the walls' values
    for f, (a, m, p) in enumerate(faces):
        open_m, open_p = on[m] & ~on[p], on[p] & ~on[m]
        fixed = (open_m | open_p) if walls and a == 0 else torch.zeros_like(open_m)
        for s, sg, rest in ((m, 1.0, open_m), (p, -1.0, open_p)):
            use = ((on[m] & on[p]) | (rest & ~fixed)).to(F64) * sg
            for b in range(d):
                C[f][face_of[s, b]] = C[f][face_of[s, b]] + use * U[s][a][b]
                R[f][s] = R[f][s] + use * U[s][a][b]
        C[f][f] = C[f][f] + (fixed | (~on[m] & ~on[p])).to(F64)
        if walls and a == 0:
            R[f][nc] = R[f][nc] + open_p.to(F64)
    X = _eliminate(torch.stack([torch.stack(r, 1) for r in C], 1), torch.stack([torch.stack(r, 1) for r in R], 1))
    n3 = 3 ** d
    A = [torch.zeros(dims[::-1], device=DEV, dtype=F64) for _ in range(n3)]
    rhs = torch.zeros(dims[::-1], device=DEV, dtype=F64)
    for f, (a, m, p) in enumerate(faces):
        both = on[m] & on[p]
        wall = walls and a == 0
        for s, sg in ((m, 1.0), (p, -1.0)):
            # the flux in +a direction out of (m) or into (p) the cell
            src = [torch.where(on[m], U[m][a][b], zero) for b in range(d)] if s == m else \
                [torch.where(on[m] & on[p], U[m][a][b], U[p][a][b]) for b in range(d)]
            fm = [face_of[m, b] for b in range(d)]
            fp = [face_of[p, b] for b in range(d)]
            use = both.to(F64) if not wall else (both | on[s]).to(F64)
            back = tuple(slice(1 - o, 1 - o + e) for o, e in zip(reversed(slots[s]), reversed(dims)))
            for c in range(nc + 1):
                own = both | (on[m] if s == m else torch.zeros_like(both))  # taken from the minus cell
                T = zero
                for b in range(d):
                    x = torch.where(own, X[:, fm[b], c], X[:, fp[b], c])
                    T = T + src[b] * x
                if c < nc:
                    if c == m:
                        T = T - torch.where(own, sum(src), zero)
                    if c == p:
                        T = T - torch.where(own, zero, sum(src))
                T = (sg * use * T).reshape(nv[::-1])[back]
                if c == nc:
                    rhs = rhs - T
                else:
                    q = sum((o2 - o1 + 1) * 3 ** k for k, (o1, o2) in enumerate(zip(slots[s], slots[c])))
                    A[q] = A[q] + T
    return torch.stack(A, -1).reshape(-1, n3), rhs.reshape(-1)


def _wells(A, rhs):
    """Bottom-hole-pressure wells in the first cell (1) and the last (0)."""
    mid, n = A.shape[1] // 2, A.shape[0]
    wi = torch.zeros_like(rhs)
    wi = torch.cat((A[:1, mid], wi[1:n - 1], A[n - 1:, mid]))
    A = torch.cat((A[:, :mid], (A[:, mid] + wi)[:, None], A[:, mid + 1:]), 1)
    return A, rhs + torch.cat((wi[:1], torch.zeros_like(wi[1:])))


def _elastic(ne, gen):
    """Q1 elasticity on unit cubes: block stencil (nodes, 27, 3, 3) and b."""
    E = torch.exp(math.log(1e10) + _field(ne, 6.0, gen))
    nu = 0.2 + 0.15 * torch.rand(ne[::-1], generator=gen, device=DEV, dtype=F64)
    lam, G = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    corners = [(x, y, z) for z in (0, 1) for y in (0, 1) for x in (0, 1)]
    gp = (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0))
    KL, KG = np.zeros((24, 24)), np.zeros((24, 24))
    for xi in itertools.product(gp, gp, gp):
        S = np.zeros((6, 24))
        for c, o in enumerate(corners):
            f = [x if q else 1 - x for x, q in zip(xi, o)]
            g = [1.0 if q else -1.0 for q in o]
            gx, gy, gz = g[0] * f[1] * f[2], g[1] * f[0] * f[2], g[2] * f[0] * f[1]
            S[:, 3 * c:3 * c + 3] = [[gx, 0, 0], [0, gy, 0], [0, 0, gz], [0, gz, gy], [gz, 0, gx], [gy, gx, 0]]
        KL += S.T @ np.diag([0.0] * 6) @ S + np.outer(S[:3].sum(0), S[:3].sum(0)) / 8.0
        KG += S.T @ np.diag([2.0, 2, 2, 1, 1, 1]) @ S / 8.0
    nn = tuple(e + 1 for e in ne)
    A = torch.zeros(nn[::-1] + (27, 3, 3), device=DEV, dtype=F64)
    tl, tg = torch.as_tensor(KL, device=DEV), torch.as_tensor(KG, device=DEV)
    for i, a in enumerate(corners):
        part = tuple(slice(q, q + e) for q, e in zip(reversed(a), reversed(ne)))
        for j, b in enumerate(corners):
            q = sum((b[k] - a[k] + 1) * 3 ** k for k in range(3))
            s = (slice(3 * i, 3 * i + 3), slice(3 * j, 3 * j + 3))
            A[part + (q,)] += lam[..., None, None] * tl[s] + G[..., None, None] * tg[s]
    load = torch.zeros(nn[::-1] + (3,), device=DEV, dtype=F64)
    for a in range(2):
        for b in range(2):
            load[-1, a:a + ne[1], b:b + ne[0], 2] -= 0.25
    # the bottom nodes are fixed: their rows and columns keep the diagonal only
    eye = torch.eye(3, device=DEV, dtype=F64)
    keep = A[0, :, :, 13] * eye
    A[0] = 0.0
    A[0, :, :, 13] = keep
    A[1, :, :, :9] = 0.0
    n = int(np.prod(nn))
    return A.reshape(n, 27, 3, 3), load.reshape(-1)


def _columns(dims):
    """Column of every stencil entry (n, 3^d), n where it leaves the grid."""
    d, n = len(dims), int(np.prod(dims))
    i = torch.arange(n, device=DEV)
    pos, st = [], 1
    for e in dims:
        pos.append((i // st) % e)
        st *= e
    cols = torch.empty((n, 3 ** d), dtype=torch.int64, device=DEV)
    for q in range(3 ** d):
        ok, c, st = torch.ones(n, dtype=torch.bool, device=DEV), i.clone(), 1
        for k in range(d):
            o = (q // 3 ** k) % 3 - 1
            ok &= (pos[k] + o >= 0) & (pos[k] + o < dims[k])
            c += o * st
            st *= dims[k]
        cols[:, q] = torch.where(ok, c, n)
    return cols


def _times(A, cols, x):
    """A x for a stencil operator."""
    bd = A.shape[2] if A.dim() == 4 else 1
    n = A.shape[0]
    xp = torch.cat((x.reshape(n, bd), x.new_zeros(1, bd)))[cols]  # (n, 3^d, bd)
    if bd == 1:
        return (A * xp[..., 0]).sum(1)
    return torch.einsum("nqij,nqj->ni", A, xp).reshape(-1)


def _system(case, seed):
    """(stencil operator, b, columns, ln k or None) of a case."""
    dims = _cells(case)
    if case["model"] == "elastic":
        A, b = _elastic(dims, torch.Generator(DEV).manual_seed(seed))
        return A, b, _columns(_points(case)), None
    logk = _log_k(case, seed)
    A, b = _mpfa(dims, logk, case["model"] == "darcy2d")
    if case["model"] == "darcy3d":
        A, b = _wells(A, b)
    return A, b, _columns(dims), logk


def _xi(case, seed, n):
    """Right-hand sides of an ensemble member are A xi, xi random normal."""
    gen = torch.Generator(DEV).manual_seed(seed + 7)
    return torch.randn((case["nrhs"], n), generator=gen, device=DEV, dtype=F64)


def _vector(seed, n):
    return torch.randn(n, generator=torch.Generator(DEV).manual_seed(seed + 7), device=DEV, dtype=F64)


def _observed(seed, n):
    gen = torch.Generator(DEV).manual_seed(seed + 7)
    at = torch.randperm(n, generator=gen, device=DEV)[:64].sort().values
    return at, torch.rand(64, generator=gen, device=DEV, dtype=F64)[:at.numel()]


def _csr(A, cols):
    ok = cols < A.shape[0]
    rowptr = torch.zeros(A.shape[0] + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = ok.sum(1).cumsum(0)
    return rowptr.to(torch.int32), cols[ok].to(torch.int32), A[ok].reshape(-1).contiguous()


def _options(case):
    prec = B.MSRSB_F32 if case["prec"] == "mixed" else B.MSRSB_F64
    kw = dict(omega=OMEGA, tol=TOL, n_it=N_IT, max_iter=MAX_PASSES, prec=prec)
    if case["model"] == "elastic":
        kw.update(smoother=B.MSRSB_SMOOTH_GS, pre=1, post=1, krylov=B.MSRSB_PCG)
    return M.opts(**kw)


def prepare(case, seed):
    bd, kind = _bdim(case), case["kind"]
    pts = _points(case)
    S, b, cols, logk = _system(case, seed)
    rowptr, colidx, val = _csr(S, cols)
    g = M.grid(pts, (case["h"],) * len(pts), centering=1 if bd == 3 else 0, ncomp=bd)
    A = M.Mat(rowptr, colidx, val, bd)
    st = dict(case=case, A=A, g=g, o=_options(case), b=b)
    n = b.numel()
    if kind == "apply":
        st["v"] = _vector(seed, n)
    if kind == "multi":
        st["B"] = torch.stack([_times(S, cols, x) for x in _xi(case, seed, n)])
    if kind == "host":
        st["host"] = tuple(t.cpu().pin_memory() for t in (rowptr, colidx, val))
        st["b_host"], st["x_host"] = b.cpu().pin_memory(), torch.empty(n, dtype=F64).pin_memory()
    if kind == "basis":
        st["p_ids"], st["skel"], st["part"] = (M.msrsb_partition(g)[k] for k in (2, 3, 0))
    if kind == "adjoint":
        khat = torch.as_tensor(_tensor(3), device=DEV).expand(n, 3, 3).contiguous()
        st["theta"] = logk.requires_grad_(True)
        st["model"] = (g, khat, [(0, 1.0), (n - 1, 0.0)], rowptr, colidx)
        st["at"], st["seen"] = _observed(seed, n)
    if kind in ("apply", "solve", "multi"):
        st["h"] = M.msrsb_setup(A, g, st["o"])
    return st


def run(st):
    kind, A, g, o = st["case"]["kind"], st["A"], st["g"], st["o"]
    if kind == "apply":
        return st["h"].apply(st["v"])
    if kind == "solve":
        return st["h"].solve(st["b"], rtol=RTOL, maxit=MAXIT)["x"]
    if kind == "multi":
        return st["h"].solve_multi(st["B"], rtol=RTOL, maxit=MAXIT)["x"]
    if kind == "host":
        M.msrsb.msrsb_solve_host_ptrs(*st["host"], A.bdim, g, o, st["b_host"], st["x_host"], rtol=RTOL, maxit=MAXIT)
        return st["x_host"]
    if kind == "setup":
        h = M.msrsb_setup(A, g, o)
        ids, P, Ac = h.get_setup()
        h.destroy()
        return dict(ids=ids, P=P, Ac=Ac)
    if kind == "basis":
        ahat, _ = M.msrsb_filter(A)
        # the initial basis: the indicator of the primal blocks
        P = (st["p_ids"] == st["part"][:, None]).to(torch.float32 if st["case"]["prec"] == "mixed" else F64)
        M.msrsb_build_basis(M.Mat(A.rowptr, A.colidx, ahat), st["p_ids"], st["skel"], P.shape[1],
                            M.basis_opts(OMEGA, TOL, N_IT, MAX_PASSES), o.prec, P)
        rowptr, colidx, val = M.msrsb_coarse_op(A, g, st["p_ids"], P, o.prec)
        return dict(ahat=ahat, P=P, rowptr=rowptr, colidx=colidx, Ac=val)
    # adjoint: the misfit at the observed cells and its gradient in ln k
    p = msrsb_mpfa_solve_diff(st["theta"], st["model"], o, rtol=RTOL, maxit=MAXIT, refine=2)
    J = ((p[st["at"]] - st["seen"]) ** 2).sum()
    return dict(p=p.detach(), grad=torch.autograd.grad(J, st["theta"])[0])


def work(case):
    """The operator read once and the results written once; multiply-adds of
    Alg. 1 (100 passes over half the entries, which the filter keeps), of the
    Galerkin product, of ILU(0) or the block smoother and of a solve's 40 steps
    (operator, smoother, transfer)."""
    pts, bd, kind = _points(case), _bdim(case), case["kind"]
    n, d = int(np.prod(pts)), len(pts)
    W, q = 2 ** d, 3 ** d
    nnz = float(np.prod([3 * e - 2 for e in pts]))
    nc = float(np.prod([-(-e // case["h"]) for e in pts]))
    esz = 4 if case["prec"] == "mixed" else 8
    op = nnz * (8 * bd * bd + 4)
    p_bytes, ac_bytes = n * W * bd * esz, nc * q * bd * bd * 8
    space = 2.0 * bd * MAX_PASSES * nnz / 2 * W / 2 + 2.0 * nnz * bd * bd * W
    factor = 2.0 * nnz * (q / 4 if bd == 1 else 0)
    step = 2.0 * nnz * bd * bd * (3 if bd == 1 else 4) + 4.0 * n * W * bd
    vec = 8.0 * n * bd
    if kind == "apply":
        return dict(bytes=op + 2 * vec, flops=step)
    if kind in ("solve", "multi"):
        return dict(bytes=op + 2 * vec * case["nrhs"], flops=40 * step * case["nrhs"])
    if kind == "basis":
        return dict(bytes=op + p_bytes + ac_bytes + 8 * nnz, flops=space)
    if kind == "setup":
        return dict(bytes=op + p_bytes + ac_bytes, flops=space + factor)
    if kind == "host":
        return dict(bytes=op + 2 * vec, flops=space + factor + 40 * step)
    return dict(bytes=n * 72.0 + 4 * vec, flops=2 * (space + factor) + 6 * 25 * step + 2500.0 * n)


# ---- the results in 64 bits ------------------------------------------------------


def _solve(A, cols, b, its=20000):
    """A^-1 b by conjugate gradients scaled by the diagonal (A is symmetric
    positive definite), to the limit of 64 bits."""
    bd = _bd(A)
    mid = A.shape[1] // 2
    D = (A[:, mid] if bd == 1 else torch.diagonal(A[:, mid], dim1=1, dim2=2)).reshape(-1)
    x, r = torch.zeros_like(b), b.clone()
    z = r / D
    p, rz = z.clone(), torch.dot(r, z)
    first = float(rz)
    for k in range(its):
        Ap = _times(A, cols, p)
        a = rz / torch.dot(p, Ap)
        x += a * p
        r -= a * Ap
        z = r / D
        new = torch.dot(r, z)
        p = z + (new / rz) * p
        rz = new
        if k % 50 == 49 and float(rz) <= 1e-29 * first:
            break
    return x


def _refined(A, cols, b):
    x = _solve(A, cols, b)
    return x + _solve(A, cols, b - _times(A, cols, x))


def _bd(A):
    return A.shape[2] if A.dim() == 4 else 1


class _Coarse:
    """Coarse nodes, supports in colour slots and primal blocks of a grid."""

    def __init__(self, pts, h, cen):
        self.nb, lo, cnt, node, blk = [], [], [], [], []
        n, st = int(np.prod(pts)), 1
        i = torch.arange(n, device=DEV)
        for e in pts:
            nb = -(-e // h) if cen == 0 else -(-(e - 1) // h) + 1
            c = [J * h + (min((J + 1) * h, e) - J * h - 1) // 2 if cen == 0 else min(J * h, e - 1) for J in range(nb)]
            c = torch.tensor(c, device=DEV)
            x = (i // st) % e
            at = torch.searchsorted(c, x, right=True) - 1  # last coarse node at or before x
            on = (at >= 0) & (c[at.clamp(min=0)] == x)
            two = (at >= 0) & ~on & (at + 1 < nb)
            if cen == 0:
                b = x // h
            else:
                up = (at + 1).clamp(max=nb - 1)
                b = torch.where(two & (x - c[at] > c[up] - x), up, at)
            lo.append(at.clamp(min=0))
            cnt.append(two)
            node.append(on)
            blk.append(b)
            self.nb.append(nb)
            st *= e
        d = len(pts)
        self.nc = int(np.prod(self.nb))
        self.strides = [int(np.prod(self.nb[:k])) for k in range(d)]
        self.ids = torch.full((n, 2 ** d), -1, dtype=torch.int64, device=DEV)
        self.lo = lo
        for t in itertools.product((0, 1), repeat=d):
            ok = torch.ones(n, dtype=torch.bool, device=DEV)
            J, s = torch.zeros_like(i), torch.zeros_like(i)
            for k in range(d):
                if t[k]:
                    ok &= cnt[k]
                I = lo[k] + t[k]
                J += I * self.strides[k]
                s += (I & 1) << k
            r = i[ok]
            self.ids[r, s[ok]] = J[ok]
        self.part = sum(b * w for b, w in zip(blk, self.strides))
        self.skel = torch.stack(node).any(0)


def _filter(a, mid):
    """M-matrix filter of a scalar stencil: negative off-diagonals, zero row sums."""
    f = a.clamp(max=0.0)
    f[:, mid] = 0.0
    f[:, mid] = -f.sum(1)
    return f


def _smooth(a, cols, G):
    """Alg. 1 on a scalar stencil: P in colour slots (n, 2^d)."""
    n, q = a.shape
    mid = q // 2
    f = _filter(a, mid)
    scale = torch.where(f[:, mid] != 0, OMEGA / f[:, mid], torch.zeros_like(f[:, mid]))
    P = (G.ids == G.part[:, None]).to(F64)
    valid = G.ids >= 0
    ids = torch.cat((G.ids, torch.full_like(G.ids[:1], -2)))
    for k in range(MAX_PASSES):
        Pp = torch.cat((P, torch.zeros_like(P[:1])))
        acc = torch.zeros_like(P)
        for j in range(q):
            c = cols[:, j]
            acc += f[:, j:j + 1] * torch.where(ids[c] == G.ids, Pp[c], 0.0)
        dP = torch.where(valid, -scale[:, None] * acc, 0.0)
        P = P + dP
        P = P / P.sum(1, keepdim=True)
        if k % N_IT == 0 and float(dP[~G.skel].abs().max()) <= TOL:
            break
    return P


def _galerkin(A, cols, P, G):
    """P^T A P as a coarse stencil (nc, 3^d, bd, bd); P: one (n, 2^d) per component."""
    bd, (n, q), d = _bd(A), A.shape[:2], len(G.nb)
    A4 = A.reshape(n, q, bd, bd)
    ids = torch.cat((G.ids, torch.full_like(G.ids[:1], -1)))

    def offset(J, base):  # stencil offset of coarse node J from per-axis indices
        return sum(((J // s) % m - o + 1) * 3 ** k for k, (s, m, o) in enumerate(zip(G.strides, G.nb, base)))

    out = torch.zeros((G.nc * q, bd, bd), device=DEV, dtype=F64)
    for m in range(bd):
        Pm = torch.cat((P[m], torch.zeros_like(P[m][:1])))
        for l in range(bd):
            AP = torch.zeros((n, q), device=DEV, dtype=F64)  # by offset from the row's lowest coarse node
            for j in range(q):
                c = cols[:, j]
                K = ids[c]
                for s in range(K.shape[1]):
                    ok = K[:, s] >= 0
                    v = torch.where(ok, A4[:, j, l, m] * Pm[c, s], 0.0)
                    at = torch.where(ok, offset(K[:, s], G.lo), 0)
                    AP.scatter_add_(1, at[:, None], v[:, None])
            for s in range(G.ids.shape[1]):
                J = G.ids[:, s]
                ok = J >= 0
                r = ok.nonzero()[:, 0]
                Jr = J[r]
                own = [(Jr // t) % e for t, e in zip(G.strides, G.nb)]
                for j in range(q):
                    K = [G.lo[k][r] + (j // 3 ** k) % 3 - 1 for k in range(d)]
                    w = P[l][r, s] * AP[r, j]
                    at = sum((K[k] - own[k] + 1) * 3 ** k for k in range(d))
                    near = torch.stack([(K[k] - own[k]).abs() <= 1 for k in range(d)]).all(0) & (w != 0)
                    out[:, l, m].index_add_(0, (Jr * q + at)[near], w[near])
    return out.reshape(G.nc, q, bd, bd)


def _dense(S, G):
    nc, q, bd, _ = S.shape
    cols = _columns(G.nb)
    D = torch.zeros((nc, nc + 1, bd, bd), device=DEV, dtype=F64)
    D[torch.arange(nc, device=DEV)[:, None], cols] = S
    return D[:, :nc].permute(0, 2, 1, 3).reshape(nc * bd, nc * bd)


def _ilu_lines(A, cols, pts):
    """ILU(0) of a 2D stencil operator in the smoother's order: pairs of
    x-lines coloured by parity, natural order inside a pair. Returns the
    factor's rows (dicts of column: value), the order and positions."""
    nx, ny = pts
    n = nx * ny
    vals, cl = A.cpu().numpy(), cols.cpu().numpy()
    order = sorted(range(n), key=lambda i: ((i // nx // 2) & 1, i // nx // 2, i))
    pos = np.empty(n, dtype=np.int64)
    pos[order] = np.arange(n)
    rows = [{int(c): float(v) for c, v in zip(cl[i], vals[i]) if c < n} for i in range(n)]
    for i in order:
        ri = rows[i]
        for k in sorted((k for k in ri if pos[k] < pos[i]), key=lambda k: pos[k]):
            lik = ri[k] / rows[k][k]
            ri[k] = lik
            for j, v in rows[k].items():
                if pos[j] > pos[k] and j in ri:
                    ri[j] -= lik * v
    return rows, order, pos


def _apply_exact(A, cols, pts, G, v):
    """The two-stage operator in 2D: coarse correction, then one ILU(0) sweep."""
    P = _smooth(A, cols, G)
    Ac = _dense(_galerkin(A, cols, [P], G), G)
    ok = G.ids >= 0
    ids = G.ids.clamp(min=0)
    r = torch.zeros(G.nc, device=DEV, dtype=F64).index_add_(0, ids[ok], (P * v[:, None])[ok])
    z = (torch.linalg.solve(Ac, r)[ids] * P * ok).sum(1)
    y = (v - _times(A, cols, z)).cpu().numpy()
    rows, order, pos = _ilu_lines(A, cols, pts)
    for i in order:
        y[i] -= sum(c * y[k] for k, c in rows[i].items() if pos[k] < pos[i])
    for i in reversed(order):
        y[i] = (y[i] - sum(c * y[k] for k, c in rows[i].items() if pos[k] > pos[i])) / rows[i][i]
    return z + torch.as_tensor(y, device=DEV)


def exact(case, seed):
    pts, bd, kind = _points(case), _bdim(case), case["kind"]
    A, b, cols, logk = _system(case, seed)
    n = b.numel()
    if kind in ("solve", "host"):
        x = _refined(A, cols, b)
        return x if kind == "solve" else x.cpu()
    if kind == "multi":
        return _xi(case, seed, n)
    if kind == "adjoint":
        p = _refined(A, cols, b)
        at, seen = _observed(seed, n)
        g = torch.zeros_like(p)
        g[at] = 2.0 * (p[at] - seen)
        lam = _refined(A, cols, g)
        theta = logk.requires_grad_(True)
        At, bt = _wells(*_mpfa(pts, theta, False))
        return dict(p=p, grad=torch.autograd.grad(torch.dot(lam, bt - _times(At, cols, p)), theta)[0])
    G = _Coarse(pts, case["h"], 1 if bd == 3 else 0)
    if kind == "apply":
        if n > 40000:
            return None
        return _apply_exact(A, cols, pts, G, _vector(seed, n))
    comps = [A] if bd == 1 else [A[:, :, l, l] for l in range(3)]
    P = [_smooth(a, cols, G) for a in comps]
    S = _galerkin(A, cols, P, G)
    if kind == "setup":
        return dict(ids=None, P=torch.stack(P), Ac=_dense(S, G))
    ok = cols < n
    near = _columns(G.nb) < G.nc
    return dict(ahat=_filter(A, A.shape[1] // 2)[ok], P=P[0], rowptr=None, colidx=None, Ac=S[near])
