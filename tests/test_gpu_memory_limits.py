"""GPU checks under a limit on device memory: what makes a split or a batched product
faster takes memory only where there is some.  The limits are what the calls need
without it, counted from the buffers' sizes."""
import ctypes as C

import numpy as np
import pytest

from oracle import linsolve as ls, mpo as ompo
from tests.gpu_util import L_from_lib, L_to_lib, crandn, rel_err, to_dev, to_host

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_02930_gb300 import api as a
    return a


def _capped(api):
    """A context whose allocator refuses what would take it above ctx.cap bytes."""
    import torch
    from paper_2606_02930_gb300 import _lib
    ctx = api.Context.__new__(api.Context)
    ctx.cap, ctx.held, ctx.refused = 1 << 40, 0, 0

    def alloc(nbytes, user):
        if ctx.held + nbytes > ctx.cap:
            ctx.refused += 1
            return None
        ctx.held += nbytes
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0, 0)

    def free(ptr, nbytes, user):
        ctx.held -= nbytes
        torch.cuda.caching_allocator_delete(ptr)

    ctx._keep = [_lib.ite_alloc_fn(alloc), _lib.ite_free_fn(free)]
    h = C.c_void_p()
    _lib.check(_lib.lib.ite_ctx_create(0, None, ctx._keep[0], ctx._keep[1], None, C.byref(h)))
    ctx.h = h
    return ctx


def _digits(M, N, K):
    """Scratch of one FP64-class product: 8 digits of 2 bytes of 2 M + N rows of 2 K
    real terms (a multiple of 32), exponents, alignment."""
    return 16 * (2 * M + N) * (-(-2 * K // 32) * 32) + 4 * (M + N) + 1024


@pytest.mark.parametrize("m,n,right,tc", [(200, 300, True, True), (300, 200, False, True),
                                          (150, 170, True, False), (40, 90, False, False)])
@pytest.mark.parametrize("extra", [0, 1])
def test_split_runs_in_the_memory_of_its_factors(api, m, n, right, tc, extra):
    # extra 1: room for the LQ's published rows as well, not for the preconditioner
    import torch
    rng = np.random.default_rng(m)
    p = min(m, n)
    s = np.exp(-np.arange(p) * 10.0 / p)
    X = (np.linalg.qr(crandn(rng, m, p))[0] * s) @ np.linalg.qr(crandn(rng, n, p))[0].conj().T
    ctx = _capped(api)
    iso = m if right else n
    ctx.cap = (ctx.held + 16 * m * n + 16 * p * iso + 128 * p + 4096 +
               (_digits(p, n, m) if tc and right else _digits(m, p, n) if tc else 0) +
               extra * 16 * m * n)
    left, right_ = to_dev(np.zeros(m * p)), to_dev(np.zeros(p * n))
    sig = torch.zeros(p, dtype=torch.float64, device="cuda")
    for _ in range(2):
        r, _ = api.k_split(ctx, to_dev(X), m, n, p, 0.0, right, left, right_, sig, tc=tc)
        assert r == p and ctx.refused > 0
        assert np.abs(sig.cpu().numpy() - s).max() <= 16 * max(m, n) * EPS
        L, R = to_host(left).reshape(m, p), to_host(right_).reshape(p, n)
        assert np.linalg.norm(L @ R - X) <= 16 * max(m, n) * EPS * np.linalg.norm(X)


def test_environment_update_with_room_for_one_batch_entry(api):
    import torch
    chi = 120
    Ws = ompo.heisenberg_mpo(8)
    rng = np.random.default_rng(1)
    Lin, A = crandn(rng, chi, 5, chi), crandn(rng, chi, 2, chi)
    want = ls.left_env_update(Lin, A, Ws[3], A)
    got = []
    for limited in (False, True):
        ctx = _capped(api)
        H = api.mpo_create(ctx, Ws)
        api.set_kernel_precision(ctx, "fp64_tc")
        if limited:      # the two intermediates, and the digits of one product at a time
            ctx.cap = ctx.held + 2 * 16 * 5 * chi * 2 * chi + 4096 + max(
                _digits(5 * chi, 2 * chi, chi), _digits(chi, chi, 2 * chi))
        out = torch.zeros(5, chi, chi, dtype=torch.complex128, device="cuda")
        api.k_env_left(ctx, H, 3, to_dev(L_to_lib(Lin)), to_dev(A), to_dev(A), out)
        assert (ctx.refused > 0) == limited
        got.append(to_host(out))
    assert np.array_equal(got[0], got[1])
    assert rel_err(L_from_lib(got[0]), want) < 1e-12
