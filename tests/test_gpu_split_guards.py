"""GPU checks of the guards of the splits' preconditioner: each is made to act (by a
value in device memory; nothing faults or waits), and the split has to stay as exact
as it is without, on the FP64 Jacobi's work alone where the guard drops the rotation.

Tolerances: as for the splits themselves, 16 max(m, n) eps of the largest singular
value and of the block.  A Newton-Schulz step missing after V is scaled by 1.0001
would leave 1.5e-8.  The FP64 Jacobi's work is counted on the device: one sweep over
all pairs is at least 8 flops a term, and a smooth spectrum leaves it less."""
import numpy as np
import pytest

from tests.gpu_util import crandn, to_dev, to_host

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_02930_gb300 import api as a
    return a


@pytest.fixture(scope="module")
def ctx(api):
    return api.ctx_create(0)


@pytest.mark.parametrize("m,n,tc", [(70, 90, False), (16, 40, False), (200, 200, True)])
@pytest.mark.parametrize("guard", ["none", "wait", "unusable", "third_step", "correction"])
def test_split_with_a_guard_acting(api, ctx, m, n, tc, guard):
    import torch
    rng = np.random.default_rng(m + n)
    p = min(m, n)
    s = np.exp(-np.arange(p) * 10.0 / p)
    X = (np.linalg.qr(crandn(rng, m, p))[0] * s) @ np.linalg.qr(crandn(rng, n, p))[0].conj().T
    left, right = to_dev(np.zeros(m * p)), to_dev(np.zeros(p * n))
    sig = torch.zeros(p, dtype=torch.float64, device="cuda")
    api.svd_stats(ctx)
    r, _ = api.k_split_selftest(ctx, to_dev(X), m, n, p, 0.0, True, left, right, sig, tc, guard)
    flops = api.svd_stats(ctx)["jacobi_fp64_flops"]
    assert r == p
    tol = 16 * max(m, n) * EPS
    assert np.abs(sig.cpu().numpy() - s).max() <= tol
    L, R = to_host(left).reshape(m, p), to_host(right).reshape(p, n)
    assert np.linalg.norm(L @ R - X) <= tol * np.linalg.norm(X)
    assert np.abs(L.conj().T @ L - np.eye(p)).max() <= 4 * max(m, n) * EPS
    all_pairs = p * (p - 1) / 2 * 8 * m
    if guard in ("wait", "unusable", "correction"):
        assert flops >= all_pairs
    else:
        assert flops < all_pairs


def test_guard_out_of_range_is_refused(api, ctx):
    from paper_2606_02930_gb300 import _lib
    X = to_dev(np.eye(20))
    for guard in (-1, 5):
        st = _lib.lib.ite_k_split_selftest(ctx.h, X.data_ptr(), 20, 20, 20, 0.0, 1, X.data_ptr(),
                                           X.data_ptr(), None, None, None, 0, guard)
        assert st == _lib.ITE_EINVAL


def test_occupancy_is_asked_once_per_cluster_size(api, ctx):
    # 70 lengths of the rows, each with a shared memory of its own
    import torch
    from paper_2606_02930_gb300 import _lib
    out = torch.empty(5000 * 16, dtype=torch.complex128, device="cuda")
    right = torch.empty(256, dtype=torch.complex128, device="cuda")
    X = to_dev(crandn(np.random.default_rng(1), 5000, 16))
    before = _lib.lib.ite_k_occupancy_queries()
    for m in range(2400, 2400 + 70 * 32, 32):
        api.k_split(ctx, X, m, 16, 16, 0.0, True, out, right)
    assert _lib.lib.ite_k_occupancy_queries() - before <= 8


def test_fp32_sweeps_are_counted(api, ctx):
    import torch
    X = to_dev(crandn(np.random.default_rng(2), 64, 64))
    left, right = torch.empty_like(X), torch.empty_like(X)
    api.svd_sweeps32(ctx)
    for n in (64, 64, 12):          # the last has too few rows to be preconditioned
        api.k_split(ctx, X, n, n, n, 0.0, True, left, right)
    splits, mean = api.svd_sweeps32(ctx)
    assert splits == 2 and 1 <= mean <= 16
    assert api.svd_sweeps32(ctx) == (0, 0.0)
