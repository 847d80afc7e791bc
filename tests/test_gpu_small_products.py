"""GPU checks of the FP64 complex GEMM's tile sizes (8, 16, 32) at their edges and
of the MPO mix's entry paths (real entries, complex entries, more entries than
are staged in shared memory).

Tolerance: a sum of K products carries at most about K eps of the largest
row-column magnitude product; 8 K eps is allowed."""
import numpy as np
import pytest

from oracle import linsolve as ls
from tests.gpu_util import L_to_lib, R_to_lib, crandn, rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_02930_gb300 import api as a
    return a


@pytest.fixture(scope="module")
def ctx(api):
    return api.ctx_create(0)


@pytest.mark.parametrize("M,N", [(1, 1), (7, 9), (8, 8), (9, 65), (64, 256), (97, 130), (160, 150),
                                 (400, 380), (640, 500)])
@pytest.mark.parametrize("K", [1, 31, 32, 33, 100])
def test_zgemm_tiles(api, ctx, M, N, K):
    import torch
    rng = np.random.default_rng(M + 1000 * N + K)
    for tA, cA, tB, cB in ((False, False, False, False), (True, True, False, False),
                           (False, False, True, True), (True, True, True, True)):
        A = crandn(rng, *((K, M) if tA else (M, K)))
        B = crandn(rng, *((N, K) if tB else (K, N)))
        C0 = crandn(rng, M, N)
        a, b = (A.T if tA else A), (B.T if tB else B)
        a, b = (a.conj() if cA else a), (b.conj() if cB else b)
        want = (0.7 - 0.2j) * (a @ b) + (0.5 + 1j) * C0
        Cd = to_dev(C0)
        api.k_zgemm(ctx, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), Cd, mode=0,
                    alpha=0.7 - 0.2j, beta=0.5 + 1j, conjA=cA, conjB=cB, transA=tA, transB=tB)
        bound = 8 * (K + 4) * 2.0 ** -52 * (np.abs(a).max(1)[:, None] * np.abs(b).max(0)[None, :] +
                                            np.abs(C0).max())
        assert (np.abs(to_host(Cd) - want) <= bound).all()


@pytest.mark.parametrize("D,d,cplx", [(2, 2, True), (3, 4, False), (5, 4, True), (32, 2, True)])
def test_heff_with_dense_mpo(api, ctx, D, d, cplx):
    # every entry of the MPO non-zero: (D d^2)^2 terms per output block
    rng = np.random.default_rng(D + d)
    W = rng.standard_normal((D, d, d, D)) + 1j * cplx * rng.standard_normal((D, d, d, D))
    Ws = [W[:1], W, W, W[..., :1]]
    H = api.mpo_create(ctx, Ws)
    chlB, chlK, chrK, chrB = 5, 7, 33, 6
    L, R = crandn(rng, chlB, D, chlK), crandn(rng, chrB, D, chrK)
    X = crandn(rng, chlK, d, d, chrK)
    want = ls.heff_apply(L, W, W, R, X)
    Y = to_dev(np.zeros((chlB, d, d, chrB), complex))
    api.k_heff(ctx, H, 1, to_dev(L_to_lib(L)), to_dev(R_to_lib(R)), to_dev(X), Y)
    assert rel_err(to_host(Y), want) < 1e-12


@pytest.mark.parametrize("n,m", [(20, 20), (32, 32), (9, 30)])
@pytest.mark.parametrize("left", [True, False])
def test_small_product_in_place(api, ctx, n, m, left):
    # C on top of an operand, while other work takes the SMs in turns with the product's
    # blocks: a block that wrote before another had read would show
    import torch
    rng = np.random.default_rng(n + m)
    busy = torch.randn(1 << 28, dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    X = crandn(rng, n, m)
    F = crandn(rng, n, n) if left else crandn(rng, m, m)
    want = F @ X if left else X @ F
    Fd = to_dev(F)
    for _ in range(150):
        C = to_dev(X)
        with torch.cuda.stream(side):
            torch.sin(torch.sin(busy))
        api.k_zgemm(ctx, *((Fd, C) if left else (C, Fd)), C, mode=0)
        assert np.abs(to_host(C) - want).max() <= 8 * 36 * 2.0 ** -52 * np.abs(F).max() * np.abs(X).max()
