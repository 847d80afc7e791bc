"""GPU parity of the preconditioned split (fp32 block Jacobi, FP64 corrections,
FP64 Jacobi on what is left) at the sizes where its blocks, padding and gates
change: row counts around 16 and 32, odd and rectangular blocks, groups of
equal singular values (left to the FP64 Jacobi), rank-deficient and strongly
graded blocks.

Tolerance: every transformation is unitary to rounding, so the singular values
and the product of the untruncated factors are off by a small multiple of
max(m, n) eps of the largest singular value (16 of them allowed); the kept rows
are orthogonal to the Jacobi's criterion, max(m, n) eps per pair (4 allowed)."""
import numpy as np
import pytest

from oracle import linsolve as ls
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


def _matrix(rng, m, n, kind):
    p = min(m, n)
    k = np.arange(p)
    s = {"decay": np.exp(-k * 10.0 / p), "groups": np.exp(-(k // 3) * 30.0 / p),
         "graded": np.exp(-k * 33.0 / p), "equal": np.ones(p),
         "lowrank": np.where(k < (p + 1) // 2, np.exp(-k * 8.0 / p), 0.0)}[kind]
    U, _ = np.linalg.qr(crandn(rng, m, p))
    V, _ = np.linalg.qr(crandn(rng, n, p))
    return (U * s[None, :]) @ V.conj().T


def _split(api, ctx, X, chi, cutoff, right, tc):
    import torch
    m, n = X.shape
    p = min(m, n)
    left, r_ = to_dev(np.zeros(m * p)), to_dev(np.zeros(p * n))
    sig = torch.zeros(p, dtype=torch.float64, device="cuda")
    r, disc = api.k_split(ctx, to_dev(X), m, n, chi, cutoff, right, left, r_, sig, tc=tc)
    return (r, disc, sig.cpu().numpy(), to_host(left)[:m * r].reshape(m, r),
            to_host(r_)[:r * n].reshape(r, n))


@pytest.mark.parametrize("m,n", [(15, 15), (16, 16), (17, 40), (31, 33), (33, 31), (64, 48),
                                 (65, 66), (97, 300), (300, 129), (257, 257)])
@pytest.mark.parametrize("kind", ["decay", "groups", "graded", "equal", "lowrank"])
def test_split_against_svd(api, ctx, m, n, kind):
    rng = np.random.default_rng(1000 * m + n)
    X = _matrix(rng, m, n, kind)
    S = np.linalg.svd(X, compute_uv=False)
    p, tol = min(m, n), 16 * max(m, n) * EPS
    for right, tc in ((True, False), (False, True)):
        r, disc, sig, L, R = _split(api, ctx, X, p, 0.0, right, tc)
        if kind in ("decay", "equal"):
            assert r == p
        assert np.abs(sig[:r] - S[:r]).max() <= tol * S[0]
        assert np.linalg.norm(L @ R - X) <= tol * np.linalg.norm(X) + 1e-12 * S[0]
        iso = L if right else R.conj().T
        assert np.abs(iso.conj().T @ iso - np.eye(r)).max() <= 4 * max(m, n) * EPS
        # truncated between two groups of singular values
        chi = max(1, p // 2 // 3 * 3)
        r_ref, disc_ref = ls.choose_rank(S, chi, 1e-10)
        r, disc, sig, L, R = _split(api, ctx, X, chi, 1e-10, right, tc)
        assert r == r_ref
        assert abs(disc - disc_ref) <= 1e-10 * max(disc_ref, 1e-12) + 1e-15


@pytest.mark.parametrize("seed", range(8))
def test_rows_of_very_different_weight_stay_preconditioned(api, ctx, seed):
    # squared norms down to 1e-26 of the largest: a rotation between a heavy and a
    # light row has to stay unitary, or all rows go to the FP64 Jacobi; left to it
    # are only members of groups of equal values, so it does less than the inner
    # products (8 flops a term) of one sweep over all pairs
    m, n = 274, 366
    X = _matrix(np.random.default_rng(seed), m, n, "groups")
    api.svd_stats(ctx)
    _split(api, ctx, X, 200, 1e-10, False, True)
    st = api.svd_stats(ctx)
    assert st["splits"] == 1
    assert st["jacobi_fp64_flops"] < m * (m - 1) / 2 * 8 * m


@pytest.mark.parametrize("scale", [1e-60, 1e60])
def test_split_is_invariant_under_scaling(api, ctx, scale):
    X = _matrix(np.random.default_rng(3), 70, 90, "decay")
    r0, d0, s0, L0, R0 = _split(api, ctx, X, 40, 1e-10, True, True)
    r, d, s, L, R = _split(api, ctx, scale * X, 40, 1e-10, True, True)
    assert r == r0
    assert np.abs(s[:r] / scale - s0[:r]).max() <= 16 * 90 * EPS * s0[0]
    assert np.linalg.norm(L @ R / scale - L0 @ R0) <= 1e-11 * np.linalg.norm(L0 @ R0)


def test_split_of_zero_and_non_finite_blocks(api, ctx):
    from paper_2606_02930_gb300._lib import IteError, ITE_ESINGULAR
    r, disc, sig, L, R = _split(api, ctx, np.zeros((40, 50)), 20, 1e-10, True, True)
    assert r == 1 and disc == 0.0 and not sig.any()
    X = _matrix(np.random.default_rng(5), 40, 40, "decay")
    X[3, 7] = np.nan
    with pytest.raises(IteError) as e:
        _split(api, ctx, X, 20, 1e-10, True, True)
    assert e.value.status == ITE_ESINGULAR
    # the context still works
    r, _, sig, _, _ = _split(api, ctx, np.nan_to_num(X), 40, 0.0, True, True)
    assert r == 40


@pytest.mark.parametrize("m,n", [(20, 127), (20, 129), (257, 20), (30, 513), (1025, 24), (3, 2050),
                                 (200, 1030)])
def test_split_of_long_rows(api, ctx, m, n):
    # the Householder LQ's variants by row length, and its general form beyond them
    X = _matrix(np.random.default_rng(m + n), m, n, "decay")
    S = np.linalg.svd(X, compute_uv=False)
    p, tol = min(m, n), 16 * max(m, n) * EPS
    for right in (True, False):
        r, disc, sig, L, R = _split(api, ctx, X, p, 0.0, right, True)
        assert r == p
        assert np.abs(sig - S).max() <= tol * S[0]
        assert np.linalg.norm(L @ R - X) <= tol * np.linalg.norm(X) + 1e-12 * S[0]


@pytest.mark.parametrize("chi,N", [(6, 8), (40, 14), (100, 16), (200, 18), (300, 20), (600, 22)])
def test_gauge_move_is_isometric_and_keeps_the_state(api, ctx, chi, N):
    # rows of 12 to 1200: every variant of the reflectors' accumulation
    from paper_2606_02930_gb300 import inputs
    A = inputs.random_isometric_mps(N, 2, chi, chi, kappa=chi / 4)
    psi = api.mps_create(ctx, A, chi)
    ref = api.mps_create(ctx, A, chi)
    api.mps_sample(ctx, psi, np.full(N, 0.5))
    nn = api.overlap(ctx, ref, ref).real
    assert abs(api.overlap(ctx, ref, psi) - nn) <= 64 * 2 * chi * EPS * nn
    for T in psi.tensors()[1:]:
        M = T.reshape(T.shape[0], -1)
        assert np.abs(M @ M.conj().T - np.eye(M.shape[0])).max() <= 16 * M.shape[1] * EPS
