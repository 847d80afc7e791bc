"""GPU check of the fp32 rotation of the splits' block Jacobi against its formula in 64
bits, over the weights and overlaps that it meets.

Its inverse square roots are the hardware's approximations (relative error 2^-22.9),
the last two with a Newton-Raphson step.  zeta = (beta - alpha) / (2 |g|) is the product
of three of them and three roundings (below 2^-20.9 together), 1 / sqrt(1 + zeta^2) is
no more sensitive than that, and the phase of s adds one approximation: s is good to
2^-20, c to 2^-22, and 2^-19 and 2^-21 are allowed.  The error of zeta is the same
rotation's in c and s, so c^2 + |s|^2 - 1 only has the phase's and the steps' error:
2^-21."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_02930_gb300 import api as a
    return a


@pytest.mark.parametrize("weights", ["equal", "near", "any", "far"])
def test_rotation_within_its_error_bounds(api, weights):
    import torch
    from paper_2606_02930_gb300 import _lib
    rng = np.random.default_rng(len(weights))
    n = 100000
    a = 10.0 ** rng.uniform(-15, 0, n)
    b = {"equal": a, "near": a * (1 + 10.0 ** rng.uniform(-7, 0, n)),
         "any": 10.0 ** rng.uniform(-15, 0, n), "far": a * 10.0 ** rng.uniform(-32, -16, n)}[weights]
    a, b = np.float32(a), np.float32(np.clip(b, 1e-33, 1.0))
    swap = rng.random(n) < 0.5
    a, b = np.where(swap, b, a), np.where(swap, a, b)
    # overlaps above what counts as rounding (2e-7)
    h = 10.0 ** rng.uniform(-6.5, -0.01, n) * np.exp(2j * np.pi * rng.random(n))
    g = np.complex64(h * np.sqrt(np.float64(a)) * np.sqrt(np.float64(b)))
    ctx = api.ctx_create(0)
    dev = [torch.from_numpy(x).cuda() for x in (a, b, g.view(np.float32))]
    c, s = torch.zeros(n, device="cuda"), torch.zeros(2 * n, device="cuda")
    _lib.check(_lib.lib.ite_k_rotation_selftest(ctx.h, n, *(x.data_ptr() for x in (*dev, c, s))),
               ctx.h)
    c, s = c.cpu().numpy().astype(float), s.cpu().numpy().astype(float).view(complex)
    al, be, gg = a.astype(float), b.astype(float), g.astype(complex)
    ag = np.abs(gg)
    zeta = (be - al) / (2 * ag)
    t = np.where(zeta >= 0, 1.0, -1.0) / (np.abs(zeta) + np.hypot(1.0, zeta))
    c0 = 1 / np.hypot(1.0, t)
    s0 = c0 * t * gg / ag
    ec, es = np.abs(c - c0).max(), (np.abs(s - s0) / np.abs(s0)).max()
    eu = np.abs(c * c + np.abs(s) ** 2 - 1).max()
    print(f"{weights}: c 2^{np.log2(ec):.1f}, s 2^{np.log2(es):.1f}, unit 2^{np.log2(eu):.1f}")
    assert ec <= 2.0 ** -21 and es <= 2.0 ** -19 and eu <= 2.0 ** -21
