"""Both sides of the rules that choose a kernel or its launch shape, and the layouts behind them, through the C ABI."""

import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
B = pytest.importorskip("paper_2203_06327_gb300.binding")

DEV = "cuda"


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
