"""GPU checks of the truncated split on graded blocks: the rows or columns of a
unitary matrix with weights over ten orders of magnitude, as a two-site block has
them when the neighbouring bond is in its Schmidt basis.

The singular values of diag(s) Q and Q diag(s) are s, to sqrt(p) eps each (rounding
Q's entries is a relative perturbation of all of them).  Row scaling leaves the
Householder LQ and the one-sided Jacobi accurate relative to each row, so the
singular values are held relatively: 16 max(m, n) eps of each value, the constant of
the absolute bound of the other splits."""
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


@pytest.mark.parametrize("m,n", [(40, 40), (140, 140), (160, 230), (230, 160), (300, 300)])
@pytest.mark.parametrize("kind", ["rows", "columns"])
def test_light_singular_values_keep_their_digits(api, ctx, m, n, kind):
    # 140 rows and more: the preconditioner's products on the tensor cores
    import torch
    rng = np.random.default_rng(m + 2 * n)
    p = min(m, n)
    s = np.exp(-np.arange(p) * 23.0 / p)
    if kind == "rows":
        X = s[:, None] * np.linalg.qr(crandn(rng, n, p))[0].conj().T
    else:
        X = np.linalg.qr(crandn(rng, m, p))[0] * s[None, :]
    m, n = X.shape
    for right in (True, False):
        for tc in (False, True):
            left, r_ = to_dev(np.zeros(m * p)), to_dev(np.zeros(p * n))
            sig = torch.zeros(p, dtype=torch.float64, device="cuda")
            r, _ = api.k_split(ctx, to_dev(X), m, n, p, 0.0, right, left, r_, sig, tc=tc)
            assert r == p
            worst = (np.abs(sig.cpu().numpy() - s) / s).max()
            print(f"{kind} {m}x{n} right={right} tc={tc}: relative error {worst:.2e}")
            assert worst <= 16 * max(m, n) * EPS
            L, R = to_host(left).reshape(m, p), to_host(r_).reshape(p, n)
            assert np.linalg.norm(L @ R - X) <= 16 * max(m, n) * EPS * np.linalg.norm(X)


@pytest.mark.parametrize("scale", [1e-60, 1e60])
def test_light_singular_values_at_the_ends_of_the_range(api, ctx, scale):
    import torch
    rng = np.random.default_rng(7)
    n = 160
    s = scale * np.exp(-np.arange(n) * 23.0 / n)
    X = to_dev(np.linalg.qr(crandn(rng, n, n))[0] * s[None, :])
    sig = torch.zeros(n, dtype=torch.float64, device="cuda")
    r, _ = api.k_split(ctx, X, n, n, n, 0.0, True, torch.empty_like(X), torch.empty_like(X), sig,
                       tc=True)
    assert r == n
    assert (np.abs(sig.cpu().numpy() - s) / s).max() <= 16 * n * EPS
