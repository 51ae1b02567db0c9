"""Kernels at the sizes where their tiles, windows and dispatch rules end, through the C ABI."""

import ctypes as C

import numpy as np
import pytest
import scipy.linalg as la
import scipy.sparse as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2203_06327_gb300.binding")

DEV = "cuda"


def _scipy(a):
    return sp.csr_matrix((a.val, a.col_idx, a.row_ptr), shape=(a.n_rows, a.n_cols))


def _reference(pb, part, rho, lam):
    """Eq. (3.3) with dense factorisations."""
    K, M, P = _scipy(pb.K), _scipy(pb.M), _scipy(pb.P)
    k = len(lam)
    w, Phi = la.eigh((P.T @ K @ P).toarray(), (P.T @ M @ P).toarray())
    y = (Phi.T @ (P.T @ rho)) / (w[:, None] - lam[None, :])
    y[:k] = 0.0
    Z = P @ (Phi @ y)
    for l in range(part.n_sub):
        d = part.sub_dofs[part.sub_ptr[l]:part.sub_ptr[l + 1]]
        Kl, Ml = K[d][:, d].toarray(), M[d][:, d].toarray()
        for i in range(k):
            Z[d, i] += la.solve(Kl - lam[i] * Ml, rho[d, i], assume_a="pos")
    return Z


def _parts(name):
    """(problem, partition) with a given local window."""
    if name == "window1":  # every third dof of a row of the grid: diagonal local matrices
        pb = B.problem_create("p1_2d", (24, 18), (1.0, 0.751), (4, 3), 1)
        n = pb.K.n_rows
        lists = [np.arange(o, n, 3, dtype=np.int32) for o in range(3)]
        lists = [d[(d // 23) % 2 == p] for d in lists for p in (0, 1)]
    elif name == "short":  # subdomains of fewer dofs than the widest one's window
        pb = B.problem_create("p1_2d", (24, 18), (1.0, 0.751), (4, 3), 1)
        n = pb.K.n_rows
        lists = [np.arange(0, 23 * 6, dtype=np.int32), np.arange(23 * 6, 23 * 6 + 5, dtype=np.int32),
                 np.arange(n - 1, n, dtype=np.int32), np.arange(23 * 6, n, dtype=np.int32)]
    else:  # strips as wide as the domain: window nx + 1
        nx = int(name[6:]) - 1
        pb = B.problem_create("p1_2d", (nx, 12), (1.0, 12.0 / nx), (nx, 12), 1)
        n = pb.K.n_rows
        # any full-rank interpolation serves: hats along x times hats along y on the dofs' own grid
        ix, iy = np.arange(n) % (nx - 1) + 1, np.arange(n) // (nx - 1) + 1
        hat = lambda t, c: np.maximum(0.0, 1.0 - np.abs(t - c) * 4)  # noqa: E731
        cols = [hat(ix / nx, a / 4) * hat(iy / 12, b / 4) for b in (1, 2, 3) for a in (1, 2, 3)]
        pb.P = B.CsrArrays.from_scipy(sp.csr_matrix(np.array(cols).T))
        lists = [np.arange(0, (nx - 1) * 7, dtype=np.int32), np.arange((nx - 1) * 4, n, dtype=np.int32)]
    ptr = np.concatenate([[0], np.cumsum([len(d) for d in lists])]).astype(np.int64)
    return pb, B.PartitionArrays(ptr, np.concatenate(lists).astype(np.int32), None, 0)


# FP64 windows at the ends of the kernel's mappings: one row, warp edges (32, 33), the last with four
# warps (127) and the first beyond (128), the widest that fits (168); subdomains shorter than the window.
# Tolerance as for the other FP64 preconditioner checks: 1e-10 of the largest entry (condition below 1e4).
@pytest.mark.parametrize("name", ["window1", "short", "window32", "window33", "window127", "window128", "window168"])
@pytest.mark.parametrize("k", [1, 3])
def test_fp64_local_windows(name, k):
    pb, part = _parts(name)
    rng = np.random.default_rng(k)
    lam = np.linspace(1.0, 12.0, k)  # below the lowest eigenvalue (at least 2 pi^2) of the pencil and its blocks
    rho = rng.standard_normal((pb.K.n_rows, k))
    ref = _reference(pb, part, rho, lam)
    sv = B.Solver(pb.K, pb.M, pb.P, None, part, k, precision=B.FP64)
    if name.startswith("window"):
        assert sv.layout()["band_window"] == int(name[6:])
    Z = torch.empty((sv.n, k), dtype=torch.float64, device=DEV)
    sv.apply_preconditioner(torch.tensor(rho, device=DEV), torch.tensor(lam, device=DEV), Z)
    assert np.abs(Z.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
    sv.close()


# Double-word Gram products: columns around multiples of four (tiles are 4 x 4), one to four blocks, row counts
# of one row, of part of a block's 64 and of 35 blocks, the last one short.  The inputs make every operation exact, so the result has to be: V holds
# integers up to 64, U integers a (not +-1) plus b 2^-28 with b up to 15 (wholly in the low part of the split unless
# a = 0), so high products sum to integers below 2^24 in the running sum and the others to multiples of 2^-28 below
# 2^-4 in the compensation; U^T U takes the integers alone.
@pytest.mark.parametrize("n", [1, 31, 33, 2209])
@pytest.mark.parametrize("k,nu,nv,sym", [(1, 1, 1, False), (2, 3, 3, True), (3, 2, 3, False), (4, 1, 1, True),
                                         (5, 3, 3, True), (7, 3, 2, False), (12, 3, 3, True), (13, 1, 3, False),
                                         (16, 4, 4, True), (16, 4, 4, False), (21, 3, 1, False), (32, 2, 2, True)])
def test_block_gram_exact_integers(n, k, nu, nv, sym):
    rng = np.random.default_rng(n * 100 + k)
    ints = lambda: rng.integers(-64, 65, size=(n, k)).astype(np.float64)  # noqa: E731
    U = [ints() for _ in range(nu)]
    if not sym:
        U = [np.where(np.abs(u) == 1, 0, u) + rng.integers(0, 16, size=(n, k)) * 2.0 ** -28 for u in U]
    V = U if sym else [ints() for _ in range(nv)]
    Ud = [torch.tensor(u, device=DEV) for u in U]
    Vd = Ud if sym else [torch.tensor(v, device=DEV) for v in V]
    out = torch.full((nu * k, nv * k), float("nan"), dtype=torch.float64, device=DEV)
    fn = B.lib.bpjd_block_gram_noalloc
    fn.argtypes = [C.c_int64, C.c_int32, C.c_int32, C.c_void_p, C.c_int32, C.c_void_p, C.c_int32, C.c_void_p,
                   C.c_void_p]
    pu = (C.c_void_p * nu)(*[u.data_ptr() for u in Ud])
    pv = (C.c_void_p * nv)(*[v.data_ptr() for v in Vd])
    assert fn(n, k, nu, pu, nv, pv, 1 if sym else 0, out.data_ptr(), None) == B.OK
    Un, Vn = np.hstack(U), np.hstack(V)
    np.testing.assert_array_equal(out.cpu().numpy(), Un.T @ Vn)


# Products of every number of columns a lane group can serve (4 per lane, 1 to 16 lanes), odd ones and arrays
# that start 8 bytes off a 16-byte boundary (scalar accesses); tolerance as for the other SpMM checks.
@pytest.mark.parametrize("ncols", [1, 2, 3, 4, 5, 7, 8, 11, 12, 17, 20, 24, 31, 32, 33, 64])
@pytest.mark.parametrize("precision", [B.FP64, B.MIXED], ids=["fp64", "mixed"])
@pytest.mark.parametrize("offset", [0, 1])
def test_spmm_columns_and_alignment(ncols, precision, offset):
    pb = B.problem_create("p1_2d", (24, 18), (1.0, 0.751), (4, 3), 1)
    sv = B.Solver.from_problem(pb, 3, device=DEV, precision=precision)
    n = sv.n
    X = np.random.default_rng(ncols).standard_normal((n, ncols))
    bufs = [torch.full((n * ncols + offset,), float("nan"), dtype=torch.float64, device=DEV) for _ in range(3)]
    Xd, YA, YM = [b[offset:].view(n, ncols) for b in bufs]
    Xd.copy_(torch.tensor(X))
    sv.spmm(Xd, YA, YM)
    for Y, a in ((YA, pb.K), (YM, pb.M)):
        A = _scipy(a)
        assert np.all(np.abs(Y.cpu().numpy() - A @ X) <= 1e-13 * (abs(A) @ np.abs(X)) + 1e-300)
    sv.close()
