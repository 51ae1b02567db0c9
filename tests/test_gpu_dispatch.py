"""Both sides of the rules that choose a kernel or its launch shape, and the layouts behind them, through the C ABI."""

import ctypes as C

import numpy as np
import pytest
import scipy.linalg as la
import scipy.sparse as sp
import scipy.sparse.linalg as spla

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2203_06327_gb300.binding")

DEV = "cuda"


def _scipy(a):
    return sp.csr_matrix((a.val, a.col_idx, a.row_ptr), shape=(a.n_rows, a.n_cols))


def _partition(lists):
    ptr = np.concatenate([[0], np.cumsum([len(d) for d in lists])]).astype(np.int64)
    return B.PartitionArrays(ptr, np.concatenate(lists).astype(np.int32), None, 0)


def _boxes(nx, ny, m):
    """Dofs of boxes of m x m grid points of an (nx - 1) x (ny - 1) grid, row by row."""
    out = []
    for b in range(0, ny - 1, m):
        for a in range(0, nx - 1, m):
            r, c = np.arange(b, min(ny - 1, b + m)), np.arange(a, min(nx - 1, a + m))
            out.append((r[:, None] * (nx - 1) + c[None]).ravel())
    return out


def _strips(window):
    """A pencil whose grid rows are as long as the local window asks, with a full-rank interpolation."""
    nx = window - 1
    pb = B.problem_create("p1_2d", (nx, 12), (1.0, 12.0 / nx), (nx, 12), 1)
    n = pb.K.n_rows
    ix, iy = np.arange(n) % (nx - 1) + 1, np.arange(n) // (nx - 1) + 1
    hat = lambda t, c: np.maximum(0.0, 1.0 - np.abs(t - c) * 4)  # noqa: E731
    cols = [hat(ix / nx, a / 4) * hat(iy / 12, b / 4) for b in (1, 2, 3) for a in (1, 2, 3)]
    pb.P = B.CsrArrays.from_scipy(sp.csr_matrix(np.array(cols).T))
    return pb, nx - 1


def _apply(sv, rho, lam):
    Z = torch.empty(rho.shape, dtype=torch.float64, device=DEV)
    sv.apply_preconditioner(torch.tensor(rho, device=DEV), torch.tensor(lam, device=DEV), Z)
    return Z.cpu().numpy()


def _coarse(K, M, P, rho, lam):
    """The coarse term of Eq. (3.3)."""
    w, Phi = la.eigh((P.T @ K @ P).toarray(), (P.T @ M @ P).toarray())
    y = (Phi.T @ (P.T @ rho)) / (w[:, None] - lam[None, :])
    y[:len(lam)] = 0.0
    return P @ (Phi @ y)


# ---- FP64 local solves --------------------------------------------------------------------------------------------

# Narrow FP64 windows take one warp per pair from 2129 pairs on, a CTA per pair below: the same bits either way.
# A small scratch cuts the second handle's subdomains into chunks below the line.  Windows of one row, of the last
# two before the rule's end (16) and of the first ones past it, where both handles run the CTA kernel.
@pytest.mark.parametrize("m,window", [(1, 1), (4, 6), (13, 15), (14, 16), (15, 17)])
def test_fp64_narrow_windows_same_bits_either_way(m, window):
    nx = 14 * m + 2 if m > 1 else 34  # the last boxes of a row are one dof wide
    pb = B.problem_create("p1_2d", (nx, nx), (1.0, 1.0), (2, 2), 1)
    lists = _boxes(nx, nx, m)
    k = 2129 // len(lists) + 1
    assert len(lists) * k > 2128 and k <= 32
    n = pb.K.n_rows
    rng = np.random.default_rng(m)
    pb.P = B.CsrArrays.from_scipy(sp.csr_matrix(rng.uniform(0.0, 1.0, (n, k + 1))))
    rho, lam = rng.standard_normal((n, k)), np.linspace(1.0, 12.0, k)
    one = B.Solver(pb.K, pb.M, pb.P, None, _partition(lists), k, precision=B.FP64)
    assert one.layout()["band_window"] == window
    few = B.Solver(pb.K, pb.M, pb.P, None, _partition(lists), k, precision=B.FP64,
                   local_scratch_bytes=8 * m * m * k * window * (len(lists) // 3))
    np.testing.assert_array_equal(_apply(one, rho, lam), _apply(few, rho, lam))


# The widest FP64 window that is accepted, and the first one that is not.
def test_fp64_widest_window():
    for window, ok in ((168, True), (169, False)):
        pb, _ = _strips(window)
        part = _partition([np.arange(pb.K.n_rows)])
        if ok:
            assert B.Solver(pb.K, pb.M, pb.P, None, part, 2, precision=B.FP64).layout()["band_window"] == window
        else:
            with pytest.raises(B.BpjdError) as e:
                B.Solver(pb.K, pb.M, pb.P, None, part, 2, precision=B.FP64)
            assert e.value.code == B.ERR_UNSUPPORTED


# ---- FP32 local solves of the wide tiers (bands by column panels) -------------------------------------------------

# Windows at both ends of the tiers 64, 96 and 152; subdomains of 1, 5, 8 and 9 dofs (below a panel, a panel, one row
# more) between wide ones of every remainder modulo 8; M with K's pattern and a diagonal M (two passes over the bands).
# Tolerance: a banded Cholesky solve in FP32 has a relative error of at most B kappa 2^-24 (kappa of the diagonally
# scaled matrix) in the 2-norm; FP32 prolongation and restriction add 1e-6 of the largest entry.
@pytest.mark.parametrize("lumped", [False, True], ids=["consistent", "lumped"])
@pytest.mark.parametrize("window", [49, 64, 65, 96, 129, 152])
def test_wide_windows_short_subdomains(window, lumped):
    pb, row = _strips(window)
    if lumped:
        M = _scipy(pb.M)
        pb.M = B.CsrArrays.from_scipy(sp.csr_matrix(sp.diags(np.asarray(M.sum(axis=1)).ravel())))
    n = pb.K.n_rows
    lists, at = [], 0
    for extra, short in zip(range(8), (1, 5, 8, 9, 1, 5, 8, 9)):
        size = 2 * row + extra
        lists += [np.arange(at, at + size), np.arange(at + 3, at + 3 + short)]
        at += row
    lists += [np.arange(at, n), np.arange(n - 1, n)]
    k = 2
    rng = np.random.default_rng(window)
    rho, lam = rng.standard_normal((n, k)), np.array([1.0, 9.0])
    K, M, P = _scipy(pb.K), _scipy(pb.M), _scipy(pb.P)
    ref, tol = _coarse(K, M, P, rho, lam), np.zeros((n, k))
    for d in lists:
        Kl, Ml = K[d][:, d].toarray(), M[d][:, d].toarray()
        for i in range(k):
            A = Kl - lam[i] * Ml
            s = 1.0 / np.sqrt(np.diag(A))
            ev = la.eigvalsh(s[:, None] * A * s)
            w = la.solve(A, rho[d, i], assume_a="pos")
            ref[d, i] += w
            tol[d, i] += window * ev[-1] / ev[0] * 2.0 ** -24 * np.linalg.norm(w / s) * s.max()
    tol += 1e-6 * np.abs(ref).max()
    sv = B.Solver(pb.K, pb.M, pb.P, None, _partition(lists), k, precision=B.MIXED)
    assert sv.layout()["band_window"] == window
    assert np.all(np.abs(_apply(sv, rho, lam) - ref) <= tol)


# ---- Gram products ------------------------------------------------------------------------------------------------

# Several chunks to a block, the last one short, and tile counts that leave warps without one: 144 and 136 tiles
# (copies and splits by the other warps), 45 and 120, one (more slices than rows taken at a time).  Inputs as in the
# other exact test: integers, so that every operation is exact.
@pytest.mark.parametrize("n", [20000, 100003])
@pytest.mark.parametrize("k,nu,nv,sym", [(1, 1, 1, False), (4, 1, 3, False), (12, 3, 3, True), (16, 3, 3, False),
                                         (20, 3, 3, True), (32, 2, 2, True)])
def test_block_gram_chunks_exact_integers(n, k, nu, nv, sym):
    rng = np.random.default_rng(n + k)
    U = [rng.integers(-64, 65, size=(n, k)).astype(np.float64) for _ in range(nu)]
    V = U if sym else [rng.integers(-64, 65, size=(n, k)).astype(np.float64) for _ in range(nv)]
    Ud = [torch.tensor(u, device=DEV) for u in U]
    Vd = Ud if sym else [torch.tensor(v, device=DEV) for v in V]
    out = torch.full((nu * k, nv * k), float("nan"), dtype=torch.float64, device=DEV)
    fn = B.lib.bpjd_block_gram_noalloc
    fn.argtypes = [C.c_int64, C.c_int32, C.c_int32, C.c_void_p, C.c_int32, C.c_void_p, C.c_int32, C.c_void_p,
                   C.c_void_p]
    pu = (C.c_void_p * nu)(*[u.data_ptr() for u in Ud])
    pv = (C.c_void_p * nv)(*[v.data_ptr() for v in Vd])
    assert fn(n, k, nu, pu, nv, pv, 1 if sym else 0, out.data_ptr(), None) == B.OK
    np.testing.assert_array_equal(out.cpu().numpy(), np.hstack(U).T @ np.hstack(V))


# ---- sparse products ----------------------------------------------------------------------------------------------

def _band_matrix(n, rng, diagonal_m):
    """Rows of 1 to 9 entries within 8 places of the diagonal, positive definite; M of the same pattern or diagonal."""
    r = np.arange(n)
    off = [(d, r[(r + d < n) & (rng.random(n) < 0.4)]) for d in (1, 3, 5, 8)]
    i = np.concatenate([x for _, x in off])
    j = np.concatenate([x + d for d, x in off])
    make = lambda v: sp.csr_matrix(sp.coo_matrix(  # noqa: E731
        (np.concatenate([v, v, np.full(n, 10.0)]), (np.concatenate([i, j, r]), np.concatenate([j, i, r]))), (n, n)))
    K = make(rng.uniform(-1.0, 1.0, len(i)))
    return K, sp.csr_matrix(sp.diags(rng.uniform(1.0, 2.0, n))) if diagonal_m else make(rng.uniform(-1.0, 1.0, len(i)))


def _check_spmm(sv, K, M, ncols, offset):
    n = sv.n
    X = np.random.default_rng(ncols).standard_normal((n, ncols))
    bufs = [torch.full((n * ncols + offset,), float("nan"), dtype=torch.float64, device=DEV) for _ in range(3)]
    Xd, YA, YM = [b[offset:].view(n, ncols) for b in bufs]
    Xd.copy_(torch.tensor(X))
    sv.spmm(Xd, YA, YM)
    for Y, A in ((YA, K), (YM, M)):  # tolerance as for the other SpMM checks
        assert np.all(np.abs(Y.cpu().numpy() - A @ X) <= 1e-13 * (abs(A) @ np.abs(X)) + 1e-300)


# Rows of 1 to 9 entries (a remainder of every size after groups of four), two columns per lane (the smaller n and up
# to 12 columns) and four (20, 31 and 64 columns of the larger n), one matrix pass or two (diagonal M).
@pytest.mark.parametrize("n", [1999, 20001])
@pytest.mark.parametrize("diagonal_m", [False, True], ids=["shared", "two"])
@pytest.mark.parametrize("precision", [B.FP64, B.MIXED], ids=["fp64", "mixed"])
def test_spmm_row_lengths_and_columns_per_lane(n, diagonal_m, precision):
    rng = np.random.default_rng(n)
    K, M = _band_matrix(n, rng, diagonal_m)
    P = sp.csr_matrix(rng.uniform(0.0, 1.0, (n, 5)))
    part = _partition([np.arange(a, min(n, a + 500)) for a in range(0, n, 500)])
    sv = B.Solver(*[B.CsrArrays.from_scipy(a) for a in (K, M, P)], None, part, 3, precision=precision)
    for ncols in (1, 2, 3, 12, 20, 31, 64):
        for offset in (0, 1):
            _check_spmm(sv, K, M, ncols, offset)


# X split ahead from 8 million products on, where the columns fill the handle's buffer: both sides of the line (8.0
# million lie between 4 and 5 columns at 512 x 512), odd columns, fewer columns than the handle's, unaligned arrays.
@pytest.mark.parametrize("k,columns", [(5, (4, 5, 6, 8)), (4, (3, 4)), (12, (4, 8, 9, 10, 12))])
def test_spmm_split_ahead(k, columns):
    pb = B.problem_create("p1_2d", (512, 512), (1.0, 0.751 / 0.75), (8, 8), 1)
    sv = B.Solver.from_problem(pb, k, device=DEV, precision=B.MIXED)
    K, M = _scipy(pb.K), _scipy(pb.M)
    for ncols in columns:
        for offset in (0, 1):
            _check_spmm(sv, K, M, ncols, offset)


# ---- row combinations and the pair of Gram products, through solves ----------------------------------------------

# Columns around the line between two and four per thread (16) and odd ones, on few row blocks (a block of at least
# 256 threads) and on many (from 609 blocks of 64 rows on), against shift-invert Lanczos; 1e-9 as for the other solves.
@pytest.mark.parametrize("nx,ny", [(80, 64), (256, 192)], ids=["few", "many"])
@pytest.mark.parametrize("k,subspace", [(1, B.W_3K), (3, B.W_3K), (7, B.W_2K), (16, B.W_3K), (17, B.W_2K),
                                        (19, B.W_3K), (23, B.W_2K)])
def test_mixed_solve_columns(nx, ny, k, subspace):
    pb = B.problem_create("p1_2d", (nx, ny), (1.0, 0.8 * 0.983), (nx // 4, ny // 4) if nx < 100 else (16, 12), 2)
    K, M = _scipy(pb.K), _scipy(pb.M)
    ref = np.sort(spla.eigsh(sp.csc_matrix(K), k, sp.csc_matrix(M), sigma=0.0, v0=np.ones(K.shape[0]),
                             return_eigenvectors=False))
    sv = B.Solver.from_problem(pb, k, device=DEV, precision=B.MIXED, subspace=subspace)
    lam, X, st = sv.solve()
    assert st["converged"] == 1
    np.testing.assert_allclose(lam, ref, rtol=1e-9)
    np.testing.assert_allclose(X.T @ (M @ X), np.eye(k), atol=1e-10)
