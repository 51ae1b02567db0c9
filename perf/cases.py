"""Cases that stand for the work of this library's users, for timing one build against another.

A program computes eigenpairs of finite-element pencils: it assembles (here with the library's own problem
generator), builds a handle and solves, or it drives its own iteration with the steps that the handle offers
(sparse products, the two-level preconditioner, block inner products).  The matrices are the model problems of
this repository's configurations, tests and benchmark, with a smooth coefficient whose phases come from the seed
(as every program has a coefficient of its own); vectors are normal random blocks.
"""

import ctypes
import math

import numpy as np
import torch

from paper_2203_06327_gb300 import binding as B

PRECISIONS = {"fp64": B.FP64, "mixed": B.MIXED, "mixed_local": B.MIXED_LOCAL}


def listed():
    return [
        # the smallest call: one product of an iteration on a mesh of under two thousand dofs, ragged sides,
        # an odd number of columns; the launch is what counts
        dict(name="spmm_small", op="spmm", kind="p1_2d", nx=48, ny=36, m=12, delta=2, k=5, precision="mixed"),
        # the largest product: K X and M X on a mesh of a million dofs, beyond the L2 cache
        dict(name="spmm_2d", op="spmm", kind="p1_2d", nx=1024, ny=1024, m=64, delta=2, k=12, precision="mixed"),
        # the wide stencil (27 entries a row) and the most columns of the paper's experiments, in native FP64
        dict(name="spmm_brick_fp64", op="spmm", kind="q1_3d", nx=64, ny=64, nz=64, m=8, delta=1, k=20,
             precision="fp64"),
        # one application of the two-level preconditioner at the benchmark's size: the Schwarz-apply metric
        dict(name="precond_2d", op="precond", kind="p1_2d", nx=512, ny=512, m=32, delta=2, k=12, precision="mixed"),
        # the same for a cube of tetrahedra: three-dimensional subdomains, band windows of about 90
        dict(name="precond_3d", op="precond", kind="p1_3d", nx=64, ny=64, nz=64, m=8, delta=1, k=10,
             precision="mixed"),
        # the clamped plate: the widest windows, the FP32 preconditioner beside native FP64 products
        dict(name="precond_plate", op="precond", kind="morley_2d", nx=256, ny=256, m=32, delta=2, k=8,
             precision="mixed_local"),
        # the default precision: the preconditioner in FP64 throughout, on a mesh of 65 thousand dofs
        dict(name="precond_fp64", op="precond", kind="p1_2d", nx=256, ny=256, m=32, delta=2, k=12, precision="fp64"),
        # the Gram matrix of a Rayleigh-Ritz search space of three blocks (Eq. (3.6)) at the benchmark's size
        dict(name="gram_ritz", op="gram", n=261121, k=12, nu=3, nv=3, symmetric=True, scratch="handle"),
        # projection coefficients against three blocks with an odd number of columns (19, as in Table 1), by a
        # caller that owns all device memory; rows that end in the middle of a block
        dict(name="gram_odd", op="gram", n=65025, k=19, nu=1, nv=3, symmetric=False, scratch="none"),
        # a whole small solve on a handle that is kept: the latency of an iteration is what counts
        dict(name="solve_small", op="solve", kind="p1_2d", nx=48, ny=48, m=8, delta=2, k=6, tau=1,
             precision="mixed", subspace="3k", setup=False, steps=21),
        # the benchmark's own call: setup and solve of a problem that is on the device, 261121 dofs, 12 eigenpairs
        dict(name="solve_2d", op="solve", kind="p1_2d", nx=512, ny=512, m=32, delta=2, k=12, tau=0,
             precision="mixed", subspace="3k", setup=True, steps=38),
        # the options that a handle has by default (FP64, search space of two blocks), ragged subdomains
        dict(name="solve_default", op="solve", kind="p1_2d", nx=48, ny=40, m=8, delta=2, k=5, tau=1,
             precision="fp64", subspace="2k", setup=False, steps=60),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid_2d(rng, n_lo, n_hi, m_lo, m_hi, most_coarse=900):
    """(nx, ny, m): boxes of m cells, at least 3 x 3 of them, about n dofs, sides that differ."""
    while True:
        n, m, shape = _log_int(rng, n_lo, n_hi), rng.randint(m_lo, m_hi), rng.uniform(0.7, 1.4)
        sx, sy = round(math.sqrt(n) * shape / m), round(math.sqrt(n) / shape / m)
        if min(sx, sy) >= 3 and sx * sy <= most_coarse and sx * sy * m * m <= 1.02 * n_hi:
            return sx * m, sy * m, m


def draw(rng):
    op = rng.choice(["spmm_2d", "spmm_3d", "precond_2d", "precond_3d", "precond_plate", "precond_fp64", "gram",
                     "solve", "solve"])
    if op == "spmm_2d":
        nx, ny, m = _grid_2d(rng, 1600, 1 << 20, 12, 64)
        coarse = (nx // m - 1) * (ny // m - 1)  # more functions than columns
        return dict(op="spmm", kind="p1_2d", nx=nx, ny=ny, m=m, delta=2, k=rng.randint(3, min(16, max(3, coarse - 1))),
                    precision=rng.choice(["mixed", "fp64"]))
    if op == "spmm_3d":
        s, m = rng.randint(4, 8), rng.randint(4, 8)
        kind = rng.choice(["q1_3d", "p1_3d"])
        # bricks have the cube's exact multiplicities, and k must not cut one on the coarse grid
        return dict(op="spmm", kind=kind, nx=s * m, ny=s * m, nz=s * m, m=m, delta=1,
                    k=rng.choice([4, 7] if s < 8 else [4, 7, 20]) if kind == "q1_3d" else rng.randint(3, 20),
                    precision=rng.choice(["mixed", "fp64"]))
    if op == "precond_2d":
        nx, ny, m = _grid_2d(rng, 2500, 512 * 512, 8, 42)
        s = min(nx, ny) // m
        return dict(op="precond", kind="p1_2d", nx=nx, ny=ny, m=m, delta=rng.randint(1, 3),
                    k=rng.randint(1, max(2, min(12, s * s // 3))), precision="mixed")
    if op == "precond_3d":
        s, m = rng.randint(4, 8), rng.randint(4, 8)
        return dict(op="precond", kind="p1_3d", nx=s * m, ny=s * m, nz=s * m, m=m, delta=1, k=rng.randint(2, 10),
                    precision="mixed")
    if op == "precond_plate":
        s, m = rng.randint(4, 8), rng.randint(8, 32)
        return dict(op="precond", kind="morley_2d", nx=s * m, ny=s * m, m=m, delta=rng.randint(1, 2),
                    k=rng.choice([3, 4, 6, 8]), precision="mixed_local")  # no k that cuts a double eigenvalue
    if op == "precond_fp64":
        nx, ny, m = _grid_2d(rng, 2500, 256 * 256, 8, 32)
        s = min(nx, ny) // m
        return dict(op="precond", kind="p1_2d", nx=nx, ny=ny, m=m, delta=rng.randint(1, 2),
                    k=rng.randint(1, max(2, min(12, s * s // 3))), precision="fp64")
    if op == "gram":
        n, k = _log_int(rng, 1000, 261121), rng.randint(2, 20)
        nu = rng.randint(1, 3)
        sym = rng.random() < 0.5
        return dict(op="gram", n=n, k=k, nu=nu, nv=nu if sym else rng.randint(1, 3), symmetric=sym, scratch="none")
    mixed = rng.random() < 0.6
    m = 2 * rng.randint(4, 12 if mixed else 8)  # even: the initial grid halves the boxes
    sx, sy = rng.randint(4, 10 if mixed else 6), rng.randint(4, 10 if mixed else 6)
    case = dict(op="solve", kind="p1_2d", nx=sx * m, ny=sy * m, m=m, delta=2, tau=1,
                precision="mixed" if mixed else "fp64", subspace="3k" if mixed else rng.choice(["2k", "3k"]),
                setup=False, steps=30)
    # k such that the first shifts stay below the subdomains' own spectra, as the method needs, and that cuts no cluster
    k, low = rng.randint(2, min(12, max(2, min(sx, sy) ** 2 // 6))), _laplace(case, 14)
    while k > 1 and low[k] < 1.1 * low[k - 1]:
        k -= 1
    return dict(case, k=k)


# ---- inputs -------------------------------------------------------------------------------------------------------

def _shape(case):
    """Cells, edge lengths and boxes per axis."""
    n = [case["nx"], case["ny"]] + ([case["nz"]] if "nz" in case else [])
    length = [1.0] * len(n)
    if case["kind"] == "p1_2d":  # no two sides alike: no eigenvalue is exactly double
        length = [1.0, 1.001 * case["ny"] / case["nx"]]
    return n, length, [c // case["m"] for c in n]


def _kappa(case, length, rng):
    """1 + 0.5 times a product of sines with phases from the seed, per element (centroids)."""
    n = [case["nx"], case["ny"]] + ([case["nz"]] if "nz" in case else [])
    ph = rng.uniform(0.0, 2.0 * np.pi, len(n))
    wave = lambda d, at: np.sin(2.0 * np.pi * (np.arange(n[d]) + at) / n[d] + ph[d])  # noqa: E731
    if case["kind"] == "p1_2d":
        low = np.outer(wave(1, 1 / 3), wave(0, 2 / 3))
        high = np.outer(wave(1, 2 / 3), wave(0, 1 / 3))
        return 1.0 + 0.5 * np.stack([low, high], axis=-1)
    if case["kind"] == "p1_3d":
        return 1.0 + 0.5 * wave(2, 0.5)[:, None, None] * wave(1, 0.5)[None, :, None] * wave(0, 0.5)[None, None, :]
    return None


def _problem(case, seed):
    """The assembled pencil, coarse interpolations and subdomains (host arrays)."""
    n, length, nsub = _shape(case)
    kappa = _kappa(case, length, np.random.default_rng([seed, 1]))
    return B.problem_create(case["kind"], n, length, nsub, case["delta"], case.get("tau", 0), kappa)


def _laplace(case, k):
    """The k lowest Dirichlet eigenvalues of the Laplacian on the box."""
    _, length, _ = _shape(case)
    one = [[(math.pi * p / L) ** 2 for p in range(1, k + 2)] for L in length]
    out = one[0]
    for o in one[1:]:
        out = [a + b for a in out for b in o]
    return np.sort(np.array(out))[:k]


def _shifts(case):
    """Shifts as an iteration has them: just below the lowest k eigenvalues (0.5 bounds the coefficient; the clamped
    plate's eigenvalues are above the squares of the Laplacian's)."""
    low = _laplace(case, case["k"])
    return 0.9 * (low ** 2 if case["kind"] == "morley_2d" else 0.5 * low)


def _normal(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _inputs(case, seed):
    """Blocks of vectors: unit columns of mixed sizes, as corrections, updates and iterates are."""
    if case["op"] == "gram":
        U = [_normal(seed * 8 + b, case["n"], case["k"]) * 10.0 ** (b - 1) for b in range(case["nu"])]
        V = U if case["symmetric"] else [_normal(seed * 8 + 4 + b, case["n"], case["k"]) for b in range(case["nv"])]
        return U, V
    return None


def prepare(case, seed):
    op, k = case["op"], case["k"]
    if op == "gram":
        U, V = _inputs(case, seed)
        out = torch.empty((case["nu"] * k, case["nv"] * k), dtype=torch.float64, device="cuda")
        st = dict(case=case, U=U, V=V, out=out)
        if case["scratch"] == "handle":
            # the handle whose iteration the blocks belong to: a square of as many interior nodes
            side = math.isqrt(case["n"]) + 1
            pb = _problem(dict(kind="p1_2d", nx=side, ny=side, m=side // 16, delta=2), seed)
            st["solver"] = B.Solver.from_problem(pb, k, device="cuda", precision=B.MIXED)
        else:
            fn = B.lib.bpjd_block_gram_noalloc
            fn.argtypes = [ctypes.c_int64, ctypes.c_int32, ctypes.c_int32, ctypes.c_void_p, ctypes.c_int32,
                           ctypes.c_void_p, ctypes.c_int32, ctypes.c_void_p, ctypes.c_void_p]
            fn.restype = ctypes.c_int
            st["pu"] = (ctypes.c_void_p * len(U))(*[u.data_ptr() for u in U])
            st["pv"] = (ctypes.c_void_p * len(V))(*[v.data_ptr() for v in V])
        return st
    pb = _problem(case, seed)
    kw = dict(precision=PRECISIONS[case["precision"]])
    if op == "solve":
        kw.update(subspace=B.W_3K if case["subspace"] == "3k" else B.W_2K, max_iter=2000)
    st = dict(case=case, kw=kw)
    if op == "solve" and case["setup"]:
        st["arrays"] = [a.to("cuda") for a in (pb.K, pb.M, pb.P)] + [pb.P0.to("cuda") if pb.tau else None,
                                                                    pb.part.to("cuda")]
        return st
    sv = st["solver"] = B.Solver.from_problem(pb, k, device="cuda", **kw)
    if op == "solve":
        return st
    st["X"] = _normal(seed, sv.n, k)
    if op == "spmm":
        st["YA"], st["YM"] = torch.empty_like(st["X"]), torch.empty_like(st["X"])
    else:
        st["lam"] = torch.tensor(_shifts(case), device="cuda")
        st["Z"] = torch.empty_like(st["X"])
    return st


def run(state):
    case = state["case"]
    if case["op"] == "spmm":
        state["solver"].spmm(state["X"], state["YA"], state["YM"])
        return {"KX": state["YA"], "MX": state["YM"]}
    if case["op"] == "precond":
        state["solver"].apply_preconditioner(state["X"], state["lam"], state["Z"])
        return {"Z": state["Z"]}
    if case["op"] == "gram":
        if "solver" in state:
            state["solver"].block_gram(state["U"], state["V"], state["out"], symmetric=case["symmetric"])
        else:
            rc = B.lib.bpjd_block_gram_noalloc(case["n"], case["k"], case["nu"], state["pu"], case["nv"], state["pv"],
                                               1 if case["symmetric"] else 0, state["out"].data_ptr(),
                                               torch.cuda.current_stream().cuda_stream)
            if rc != B.OK:
                raise B.BpjdError(rc, "bpjd_block_gram_noalloc")
        return {"gram": state["out"]}
    if "arrays" in state:
        sv = B.Solver(*state["arrays"], case["k"], **state["kw"])
        lam, X, _ = sv.solve(eigvecs="device")
        sv.close()
    else:
        lam, X, _ = state["solver"].solve(eigvecs="device")
    return {"lam": lam, "X": X}


# ---- what a pass cannot do without --------------------------------------------------------------------------------

def _sizes(case):
    """(dofs, entries of K, entries of P, coarse dofs, sum of local sizes, band window, subdomains)."""
    n, _, nsub = _shape(case)
    plate = case["kind"] == "morley_2d"
    a = [2 * c - 1 if plate else c - 1 for c in n]  # dofs per axis (the plate's on the half-grid)
    dofs = math.prod(a)
    if case["kind"] == "p1_2d":
        nnz = dofs + 2 * ((a[0] - 1) * a[1] + a[0] * (a[1] - 1) + (a[0] - 1) * (a[1] - 1))
    elif case["kind"] == "p1_3d":
        nnz = dofs
        for s in range(1, 8):
            nnz += 2 * math.prod(a[d] - (s >> d & 1) for d in range(3))
    elif case["kind"] == "q1_3d":
        nnz = math.prod(3 * c - 2 for c in a)
    else:
        nnz = 11 * dofs
    coarse = math.prod(s - 1 for s in nsub) * (4 if plate else 1)
    nnzp = round(dofs * (12 if plate else 2.6 if case["kind"] == "p1_2d" else 2.3))
    wide = []
    for c, s in zip(n, nsub):
        m = c // s
        ends = [(max(0, b * m - case["delta"]), min(c, (b + 1) * m + case["delta"])) for b in range(s)]
        wide.append([(2 if plate else 1) * (hi - lo) - 1 for lo, hi in ends])
    local = math.prod(sum(w) for w in wide)
    top = [max(w) for w in wide]
    window = 2 * top[0] + 3 if plate else top[0] + 2 if len(n) == 2 else top[0] * top[1] + top[0] + 2
    return dofs, nnz, nnzp, coarse, local, window, math.prod(nsub)


def _precond_work(case):
    dofs, nnz, nnzp, coarse, local, window, _ = _sizes(case)
    k = case["k"]
    bytes_ = nnz * 20 + local * 4 + nnzp * 12 + 2 * dofs * k * 8 + coarse * coarse * 8
    flops = local * k * (window * window + 4 * window) + 4 * nnzp * k + 4 * coarse * coarse * k
    return bytes_, flops


def work(case):
    k = case["k"]
    if case["op"] == "gram":
        n, mu, mv = case["n"], case["nu"] * k, case["nv"] * k
        blocks = case["nu"] if case["symmetric"] else case["nu"] + case["nv"]
        return {"bytes": 8 * (blocks * n * k + mu * mv), "flops": n * mu * (mv + 1 if case["symmetric"] else 2 * mv)}
    dofs, nnz = _sizes(case)[:2]
    spmm = nnz * 20 + 8 * (dofs + 1) + 24 * dofs * k, 4 * nnz * k
    if case["op"] == "spmm":
        return {"bytes": spmm[0], "flops": spmm[1]}
    pre = _precond_work(case)
    if case["op"] == "precond":
        return {"bytes": pre[0], "flops": pre[1]}
    # a solve: per step one preconditioner application, the products of three blocks, the Gram matrices of the search
    # space and the new iterate and update (steps: what such a problem takes); the local factors are formed a few
    # times and read by the other steps
    nb = 3 if case["subspace"] == "3k" else 2
    mk = nb * k
    per_bytes = 3 * spmm[0] + 8 * dofs * k * (3 * nb + 6)
    per_flops = 3 * spmm[1] + 2 * dofs * mk * (mk + 1) + 8 * dofs * mk * k
    return {"bytes": case["steps"] * (per_bytes + pre[0]), "flops": case["steps"] * per_flops + 6 * pre[1]}


# ---- the same in 64 bits, without the library's solver ------------------------------------------------------------

def _csr(a):
    return torch.sparse_csr_tensor(torch.as_tensor(a.row_ptr), torch.as_tensor(a.col_idx).long(),
                                   torch.as_tensor(a.val), size=(a.n_rows, a.n_cols)).to("cuda")


def _flip(X):
    """Columns with their entry of largest size positive."""
    top = X.abs().argmax(dim=0)
    return X * torch.where(X[top, torch.arange(X.shape[1], device=X.device)] < 0, -1.0, 1.0)


def _pencil(K, M):
    """Ascending eigenvalues and M-orthonormal eigenvectors of a dense pencil."""
    L = torch.linalg.cholesky(M)
    A = torch.linalg.solve_triangular(L, K, upper=False)
    A = torch.linalg.solve_triangular(L, A.T.contiguous(), upper=False)
    w, Q = torch.linalg.eigh(0.5 * (A + A.T))
    return w, torch.linalg.solve_triangular(L.T, Q, upper=True)


def _exact_precond(case, seed):
    """Eq. (3.3): the coarse term in the coarse eigenbasis, and the sum of the local solves."""
    pb, k = _problem(case, seed), case["k"]
    n, lam = pb.K.n_rows, torch.tensor(_shifts(case), device="cuda")
    rho = _normal(seed, n, k)
    K, M, P = _csr(pb.K), _csr(pb.M), _csr(pb.P)
    Pd = P.to_dense()
    w, Phi = _pencil(Pd.T @ (K @ Pd), Pd.T @ (M @ Pd))
    c = Phi.T @ (Pd.T @ rho)
    y = c / (w[:, None] - lam[None, :])
    y[:k] = 0.0
    Z = Pd @ (Phi @ y)
    del Pd
    # the local matrices in blocks as wide as their band: block tridiagonal, factorised for all subdomains at once
    ptr, dofs = torch.as_tensor(pb.part.sub_ptr).cuda(), torch.as_tensor(pb.part.sub_dofs).cuda().long()
    sizes = ptr[1:] - ptr[:-1]
    sub = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), sizes)
    pos = torch.arange(len(dofs), device="cuda") - ptr[sub]
    key = sub * n + dofs  # ascending

    def local(A):
        """(row, column, value) of the entries inside the subdomains, rows and columns by packed position."""
        rp, ci = A.crow_indices(), A.col_indices()
        cnt = rp[dofs + 1] - rp[dofs]
        row = torch.repeat_interleave(torch.arange(len(dofs), device="cuda"), cnt)
        e = rp[dofs][row] + torch.arange(len(row), device="cuda") - (torch.cumsum(cnt, 0) - cnt)[row]
        want = sub[row] * n + ci[e]
        at = torch.searchsorted(key, want).clamp_(max=len(key) - 1)
        ok = key[at] == want
        return row[ok], at[ok], A.values()[e[ok]]

    parts = [local(A) for A in (K, M)]
    b = max(int((r - c).abs().max()) for r, c, _ in parts) + 1
    nb = -(-int(sizes.max()) // b)

    def blocks(r, c, v, diagonal):
        D = torch.zeros((nb, len(sizes), b, b), dtype=torch.float64, device="cuda")
        E = torch.zeros_like(D)  # block row j + 1, block column j
        if diagonal:  # rows past a subdomain's end
            D += torch.eye(b, dtype=torch.float64, device="cuda")
            D[pos // b, sub, pos % b, pos % b] = 0.0
        pr, pc = pos[r], pos[c]
        on, under = pr // b == pc // b, pr // b == pc // b + 1
        D[pr[on] // b, sub[r[on]], pr[on] % b, pc[on] % b] = v[on]
        E[pc[under] // b, sub[r[under]], pr[under] % b, pc[under] % b] = v[under]
        return D, E

    (DK, EK), (DM, EM) = blocks(*parts[0], True), blocks(*parts[1], False)
    tri = torch.linalg.solve_triangular
    for i in range(k):
        x = torch.zeros((nb, len(sizes), b, 1), dtype=torch.float64, device="cuda")
        x[pos // b, sub, pos % b, 0] = rho[dofs, i]
        L, S = [], []
        for j in range(nb):
            D = DK[j] - lam[i] * DM[j]
            if j:
                D -= S[-1] @ S[-1].mT
                x[j] -= S[-1] @ x[j - 1]
            L.append(torch.linalg.cholesky(D))
            x[j] = tri(L[-1], x[j], upper=False)
            S.append(tri(L[-1], (EK[j] - lam[i] * EM[j]).mT.contiguous(), upper=False).mT)
        for j in reversed(range(nb)):
            if j + 1 < nb:
                x[j] -= S[j].mT @ x[j + 1]
            x[j] = tri(L[j].mT, x[j], upper=True)
        Z[:, i].index_add_(0, dofs, x[pos // b, sub, pos % b, 0])
    return {"Z": Z}


def exact(case, seed):
    op, k = case["op"], case["k"]
    if op == "gram":
        U, V = _inputs(case, seed)
        return {"gram": torch.cat(U, dim=1).T @ torch.cat(V, dim=1)}
    if op == "spmm":
        pb = _problem(case, seed)
        X = _normal(seed, pb.K.n_rows, k)
        return {"KX": _csr(pb.K) @ X, "MX": _csr(pb.M) @ X}
    if op == "precond":
        return _exact_precond(case, seed)
    if _sizes(case)[0] > 6000:
        return None
    pb = _problem(case, seed)
    w, V = _pencil(_csr(pb.K).to_dense(), _csr(pb.M).to_dense())
    return {"lam": w[:k].cpu().numpy(), "X": _flip(V[:, :k])}
