"""What a user has this library do, as measurable cases.

One implicit step is a chain of two-site updates, each made of the local solve
(GMRES on the effective Hamiltonian), a truncated SVD split and an environment
update.  The cases call these blocks through their own entry points at the
sizes of the repository's workloads (Heisenberg chains with chi 32 to 256, d =
2, D = 5; impurity blocks with d = 4, D = 6), from the launch-bound small ones
to the largest split, and two whole steps.

The factors of a split are fixed only up to a unitary on the new bond, and so
are the tensors of an MPS.  So a split case returns the product of its factors
(the merged block that the next visit of the bond forms, by the library's own
GEMM) with the kept singular values, and a step case the state's amplitudes.

Everything is plain torch on the GPU apart from the calls that are measured.
"""
import math

import numpy as np
import torch

from paper_2606_02930_gb300 import api

DEV = "cuda"
C128 = torch.complex128

# Algorithmic FLOPs of a truncated SVD of a p x q complex block per p q min(p, q)
SVD_FLOPS = 8.7e9 / 512.0 ** 3


def listed():
    return [
        # the two-site matvec of the small chain (N = 10, chi = 32): launches and latency
        dict(name="heff_small", op="heff", model="heisenberg", la=32, lb=32, rb=32, ra=32,
             prec="fp64", z=True),
        # the matvec that a step of the benchmark chain runs 1386 times
        dict(name="heff_bulk", op="heff", model="heisenberg", la=256, lb=256, rb=256, ra=256,
             prec="fp64_tc", z=True),
        # an impurity block with odd bonds on all sides, as in the fit of a right-hand side
        dict(name="heff_impurity_odd", op="heff", model="anderson", la=117, lb=93, rb=131, ra=109,
             prec="fp64_tc", z=False),
        # environment updates of the benchmark chain, one of each direction
        dict(name="env_bulk", op="env", model="heisenberg", la=256, lb=256, rb=256, ra=256,
             prec="fp64_tc"),
        # GMRES(10) of a served chain (chi = 64) in plain FP64, and of the benchmark chain
        dict(name="solve_served", op="solve", model="heisenberg", chl=64, chr=64, prec="fp64",
             dtau=0.1, m=10),
        dict(name="solve_bulk", op="solve", model="heisenberg", chl=256, chr=256, prec="fp64_tc",
             dtau=0.1, m=10),
        # a local solve converged by refinement with bf16 inner matvecs
        dict(name="solve_mixed", op="solve", model="heisenberg", chl=256, chr=256,
             prec="mixed_bf16", dtau=0.1, m=10),
        # truncated SVD splits: the small chain's block, an odd block whose singular values
        # come in triplets and whose cutoff binds, the benchmark chain's block, and a block of
        # 1024 (chi = 512 with d = 2, or chi = 256 with d = 4)
        dict(name="split_small", op="split", m=64, n=64, chi=32, cutoff=0.0, efolds=10.0, mult=1,
             right=True, tc=False),
        dict(name="split_odd", op="split", m=274, n=366, chi=200, cutoff=1e-10, efolds=30.0,
             mult=3, right=False, tc=True),
        dict(name="split_bulk", op="split", m=512, n=512, chi=256, cutoff=1e-10, efolds=12.0,
             mult=1, right=True, tc=True),
        dict(name="split_large", op="split", m=1024, n=1024, chi=512, cutoff=1e-14, efolds=16.0,
             mult=1, right=True, tc=True),
        # one whole backward-Euler step of a chain at its bond cap, as the benchmark runs it
        dict(name="step_chain", op="step", n=18, chi=96, prec="fp64_tc", scheme="be", dtau=0.05,
             seed_kappa=24.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["heff", "heff", "env", "solve", "split", "split", "split", "step"])
    if op in ("heff", "env"):
        model = rng.choice(["heisenberg", "anderson"])
        top = 300 if model == "heisenberg" else 140
        base = _log_int(rng, 16, top)
        side = [max(8, min(top, int(base * rng.uniform(0.7, 1.3)))) for _ in range(4)]
        case = dict(op=op, model=model, la=side[0], lb=side[1], rb=side[2], ra=side[3],
                    prec=rng.choice(["fp64", "fp64_tc"]))
        if op == "heff":
            case["z"] = rng.random() < 0.5
        return case
    if op == "solve":
        model = rng.choice(["heisenberg", "anderson"])
        top = 256 if model == "heisenberg" else 96
        chl = _log_int(rng, 24, top)
        chr_ = max(24, min(top, int(chl * rng.uniform(0.7, 1.3))))
        dtau = rng.uniform(0.06, 0.12) * (1.0 if model == "heisenberg" else 4.0)
        return dict(op=op, model=model, chl=chl, chr=chr_, dtau=round(dtau, 4),
                    prec=rng.choice(["fp64", "fp64_tc", "fp64_tc", "mixed_bf16"]),
                    m=rng.choice([6, 8]))
    if op == "split":
        m = _log_int(rng, 24, 1000)
        n = max(24, min(1000, int(m * rng.uniform(0.6, 1.6))))
        p = min(m, n)
        return dict(op=op, m=m, n=n, chi=max(4, int(p * rng.uniform(0.3, 0.8))),
                    cutoff=rng.choice([0.0, 1e-14, 1e-10]), efolds=round(rng.uniform(6.0, 20.0), 2),
                    mult=rng.choice([1, 1, 2, 3]), right=rng.random() < 0.5,
                    tc=rng.random() < 0.7)
    return dict(op=op, n=rng.randint(8, 14), chi=_log_int(rng, 16, 64),
                prec=rng.choice(["fp64", "fp64_tc"]), scheme=rng.choice(["be", "tr"]),
                dtau=round(rng.uniform(0.02, 0.1), 4), seed_kappa=round(rng.uniform(8.0, 24.0), 2))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _randn(g, *shape):
    z = torch.randn(*shape, 2, generator=g, device=DEV, dtype=torch.float64)
    return torch.view_as_complex(z) / math.sqrt(2.0)


def _orth(g, rows, cols):
    """rows x cols with orthonormal columns (rows >= cols) or rows."""
    if rows >= cols:
        return torch.linalg.qr(_randn(g, rows, cols))[0].contiguous()
    return torch.linalg.qr(_randn(g, cols, rows))[0].mH.contiguous()


def heisenberg_w():
    """Bulk MPO tensor W[w, s', s, w'] of sum S.S (channels: nothing yet, S+, S-, Sz, done)."""
    sp = np.array([[0.0, 1.0], [0.0, 0.0]])
    sz = np.diag([0.5, -0.5])
    W = np.zeros((5, 2, 2, 5))
    W[0, :, :, 0] = W[4, :, :, 4] = np.eye(2)
    W[0, :, :, 1], W[0, :, :, 2], W[0, :, :, 3] = sp, sp.T, sz
    W[1, :, :, 4], W[2, :, :, 4], W[3, :, :, 4] = 0.5 * sp.T, 0.5 * sp, sz
    return W.astype(complex)


def anderson_w(eps=0.3, v=0.2):
    """MPO tensor of a bath site in the star geometry (d = 4, six channels: start, the four
    operators of the impurity carried along with the sign string, done)."""
    F1, a = np.diag([1.0, -1.0]), np.array([[0.0, 1.0], [0.0, 0.0]])
    up, dn = np.kron(np.eye(2), a), np.kron(a, F1)
    F, n = np.kron(F1, F1), up.T @ up + dn.T @ dn
    W = np.zeros((6, 4, 4, 6))
    W[0, :, :, 0] = W[5, :, :, 5] = np.eye(4)
    W[0, :, :, 5] = eps * n
    for k, o in enumerate((up, dn, up.T, dn.T)):
        W[1 + k, :, :, 1 + k] = F
        W[1 + k, :, :, 5] = v * o
    return W.astype(complex)


def bulk_w(model):
    return heisenberg_w() if model == "heisenberg" else anderson_w()


def chain_ws(model, n):
    W = bulk_w(model)
    return [W[:1]] + [W] * (n - 2) + [W[..., -1:]]


def _environment(g, W, chi, left):
    """Environment of a chain of random isometric tensors that ends in bond chi: as the
    left (w, bra, ket) or the right (w, ket, bra) block of the library's layout."""
    d = W.shape[1]
    Wt = torch.from_numpy(W).to(DEV)
    first = Wt[:1] if left else Wt[..., -1:]
    E = torch.ones(1, 1, 1, dtype=C128, device=DEV)
    a, site = 1, 0
    while a < chi or site < 3:
        b = min(chi, a * d)
        Wi = first if site == 0 else Wt
        if left:
            A = _orth(g, a * d, b).reshape(a, d, b)
            T = torch.tensordot(E, A, dims=([2], [0]))                  # w a s b'
            T = torch.tensordot(T, Wi, dims=([0, 2], [0, 2]))           # a b' s' w'
            E = torch.tensordot(A.conj(), T, dims=([0, 1], [0, 2])).permute(2, 0, 1).contiguous()
        else:
            A = _orth(g, b, d * a).reshape(b, d, a)
            T = torch.tensordot(E, A, dims=([1], [2]))                  # w bra a' s
            T = torch.tensordot(T, Wi, dims=([0, 3], [3, 2]))           # bra a' w' s'
            E = torch.tensordot(T, A.conj(), dims=([0, 3], [2, 1])).permute(1, 0, 2).contiguous()
        a, site = b, site + 1
    return E


def _two_site_block(g, chl, d, chr_):
    """A normalised two-site tensor with a decaying Schmidt spectrum."""
    p = min(chl * d, d * chr_)
    U, V = _orth(g, chl * d, p), _orth(g, p, d * chr_)
    s = torch.exp(-torch.arange(p, device=DEV, dtype=torch.float64) * (10.0 / p))
    X = (U * (s / s.norm()).to(C128)) @ V
    return X.reshape(chl, d, d, chr_).contiguous()


def _heff(W, L, R, X):
    """Plain two-site effective Hamiltonian in 64 bits."""
    Wt = torch.from_numpy(W).to(X.device)
    T = torch.tensordot(L, X, dims=([2], [0]))                          # w a s t b'
    T = torch.tensordot(T, Wt, dims=([0, 2], [0, 2]))                   # a t b' s' v
    T = torch.tensordot(T, Wt, dims=([4, 1], [0, 2]))                   # a b' s' t' u
    return torch.tensordot(T, R, dims=([4, 1], [0, 1]))                 # a s' t' b


def _split_matrix(case, seed):
    g = _gen(seed)
    m, n, mult = case["m"], case["n"], case["mult"]
    p = min(m, n)
    k = torch.arange(p, device=DEV) // mult * mult
    s = torch.exp(-k.to(torch.float64) * (case["efolds"] / p))
    return ((_orth(g, m, p) * (s / s.norm()).to(C128)) @ _orth(g, p, n)).contiguous()


def _bonds(n, chi):
    return [min(2 ** min(b, n - b), chi) for b in range(n + 1)]


def _chain_state(case, seed):
    """Site tensors of a chain at its bond cap: random isometries with decaying weights."""
    g = _gen(seed)
    chi = _bonds(case["n"], case["chi"])
    out = []
    for i in range(case["n"]):
        a, b = chi[i], chi[i + 1]
        w = torch.exp(-torch.arange(b, device=DEV, dtype=torch.float64) / case["seed_kappa"])
        out.append((_orth(g, 2 * a, b) * (w / w.norm()).to(C128)).reshape(a, 2, b))
    out[0] = out[0] / _amplitudes(out).norm()
    return out


def _amplitudes(tensors):
    """The state vector of an MPS: its two halves contracted, then joined."""
    T = [t if isinstance(t, torch.Tensor) else torch.from_numpy(t).to(DEV) for t in tensors]
    h = len(T) // 2
    left = T[0].reshape(2, -1)
    for t in T[1:h]:
        left = torch.tensordot(left, t, dims=([1], [0])).reshape(-1, t.shape[2])
    right = T[-1].reshape(-1, 2)
    for t in reversed(T[h:-1]):
        right = torch.tensordot(t, right, dims=([2], [0])).reshape(t.shape[0], -1)
    return (left @ right).reshape(-1)


def _apply_chain(v, n):
    """H v of the open Heisenberg chain on a state vector."""
    out = torch.zeros_like(v)
    for i in range(n - 1):
        x = v.reshape(2 ** i, 4, 2 ** (n - 2 - i))
        y = 0.25 * x
        y[:, 1] = 0.5 * x[:, 2] - 0.25 * x[:, 1]
        y[:, 2] = 0.5 * x[:, 1] - 0.25 * x[:, 2]
        out += y.reshape(-1)
    return out


# ------------------------------------------------------------------ a program's state
def _local_inputs(case, seed):
    W = bulk_w(case["model"])
    g = _gen(seed)
    d = W.shape[1]
    if case["op"] == "solve":
        L = _environment(g, W, case["chl"], True)
        R = _environment(g, W, case["chr"], False)
        X0 = _two_site_block(g, case["chl"], d, case["chr"])
        B = X0 + 0.05 * _two_site_block(g, case["chl"], d, case["chr"])
        shift = float(torch.sum(X0.conj() * _heff(W, L, R, X0)).real)
        return W, dict(L=L, R=R, X0=X0, B=B, alpha=1.0 - case["dtau"] * shift, c=case["dtau"])
    D, la, lb, rb, ra = W.shape[0], case["la"], case["lb"], case["rb"], case["ra"]
    if case["op"] == "heff":
        v = dict(L=_randn(g, D, la, lb), R=_randn(g, D, rb, ra), X=_randn(g, lb, d, d, rb))
        if case["z"]:
            v["Z"] = _randn(g, la, d, d, ra)
        return W, v
    return W, dict(Lin=_randn(g, D, la, lb), Rin=_randn(g, D, rb, ra), bra=_randn(g, la, d, ra),
                   ket=_randn(g, lb, d, rb))


def prepare(case, seed):
    ctx = api.ctx_create(0)
    st = dict(case=case, ctx=ctx)
    if case["op"] == "split":
        X = _split_matrix(case, seed)
        p = min(X.shape)
        st.update(X=X, left=torch.empty(X.shape[0] * p, dtype=C128, device=DEV),
                  right=torch.empty(p * X.shape[1], dtype=C128, device=DEV),
                  sigma=torch.empty(p, dtype=torch.float64, device=DEV),
                  out=torch.empty_like(X))
        return st
    if case["op"] == "step":
        T = [t.cpu().numpy() for t in _chain_state(case, seed)]
        st["H"] = api.mpo_create_heisenberg(ctx, case["n"])
        st["psi0"] = api.mps_create(ctx, T, case["chi"])
        st["psi"] = api.mps_create(ctx, T, case["chi"])
        st["shift"] = api.energy(ctx, st["H"], st["psi0"])
        return st
    W, v = _local_inputs(case, seed)
    st["H"] = api.mpo_create(ctx, chain_ws(case["model"], 6))
    st.update(v)
    if case["op"] == "heff":
        st["Y"] = torch.empty(case["la"], W.shape[1], W.shape[1], case["ra"], dtype=C128, device=DEV)
    elif case["op"] == "env":
        st["Lout"] = torch.empty(W.shape[3], case["ra"], case["rb"], dtype=C128, device=DEV)
        st["Rout"] = torch.empty(W.shape[0], case["lb"], case["la"], dtype=C128, device=DEV)
    else:
        st["X"] = torch.empty_like(v["X0"])
    api.set_kernel_precision(ctx, case["prec"])
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    if case["op"] == "heff":
        api.k_heff(ctx, st["H"], 2, st["L"], st["R"], st["X"], st["Y"], alpha=0.4,
                   Z=st.get("Z"), gamma=1.1 if case["z"] else 0.0)
        return st["Y"]
    if case["op"] == "env":
        api.k_env_left(ctx, st["H"], 2, st["Lin"], st["bra"], st["ket"], st["Lout"])
        api.k_env_right(ctx, st["H"], 2, st["Rin"], st["bra"], st["ket"], st["Rout"])
        return st["Lout"], st["Rout"]
    if case["op"] == "solve":
        st["X"].copy_(st["X0"])
        steps, res = api.k_local_solve(ctx, st["H"], 2, st["L"], st["R"], st["B"], st["X"],
                                       st["alpha"], st["c"], case["m"])
        if case["prec"].startswith("mixed"):
            return {"X": st["X"]}          # converged: the residual left over is rounding
        return {"X": st["X"], "residual": res, "steps": steps}
    if case["op"] == "split":
        m, n = case["m"], case["n"]
        r, disc = api.k_split(ctx, st["X"], m, n, case["chi"], case["cutoff"], case["right"],
                              st["left"], st["right"], st["sigma"], tc=case["tc"])
        left, right = st["left"][:m * r].view(m, r), st["right"][:r * n].view(r, n)
        api.k_zgemm(ctx, left, right, st["out"], mode=1 if case["tc"] else 0)
        return {"product": st["out"], "sigma": st["sigma"][:r], "rank": r, "discarded": disc}
    api.mps_copy(ctx, st["psi0"], st["psi"])
    info = api.implicit_step(ctx, st["H"], st["psi"], case["dtau"], case["scheme"], st["shift"],
                             case["chi"], 1e-10, api.solver_opts(precision=case["prec"]))
    return {"energy": info["energy"], "norm": info["norm_before"],
            "discarded": info["max_discarded_weight"], "chi": info["max_chi"],
            "state": _amplitudes(st["psi"].tensors())}


# ------------------------------------------------------------------ the same in 64 bits
def _krylov(A, B, X0, m):
    """The m-step Krylov least-squares solution (Arnoldi with reorthogonalisation)."""
    r0 = B - A(X0)
    beta = float(r0.norm())
    V, H = [r0 / beta], torch.zeros(m + 1, m, dtype=C128)
    for j in range(m):
        w = A(V[j])
        for _ in range(2):
            for i in range(j + 1):
                h = torch.sum(V[i].conj() * w)
                H[i, j] += h.cpu()
                w = w - h * V[i]
        H[j + 1, j] = float(w.norm())
        V.append(w / H[j + 1, j].real.item())
    e = torch.zeros(m + 1, 1, dtype=C128)
    e[0] = beta
    y = torch.linalg.lstsq(H, e).solution
    X = X0 + sum(complex(y[i, 0]) * V[i] for i in range(m))
    return X, float((e - H @ y).norm()) / float(B.norm())


def _rank(s2, chi, cutoff):
    """The truncation rule: the smallest rank whose discarded weight is within the cutoff,
    at most chi, and no group of equal singular values cut in two."""
    total = s2.sum()
    tail = np.concatenate([np.cumsum(s2[::-1])[::-1], [0.0]])
    r = next(k for k in range(1, len(s2) + 1) if tail[k] <= max(cutoff, 1e-24) * total)
    r = min(r, chi)
    s = np.sqrt(s2)
    if r < len(s) and s[r] >= s[r - 1] * (1 - 1e-10):
        g = r - 1
        while g > 0 and s[g] >= s[g - 1] * (1 - 1e-10):
            g -= 1
        r = g if g >= 1 else r
    return r, tail[r] / total


def exact(case, seed):
    if case["op"] == "split":
        X = _split_matrix(case, seed)
        U, S, Vh = torch.linalg.svd(X.cpu(), full_matrices=False)
        r, disc = _rank(S.numpy() ** 2, case["chi"], case["cutoff"])
        return {"product": (U[:, :r] * S[:r]) @ Vh[:r], "sigma": S[:r], "rank": r,
                "discarded": float(disc)}
    if case["op"] == "step":
        n = case["n"]
        if case["chi"] < 2 ** (n // 2):
            return None                    # the truncated step is defined by its own sweep
        v = _amplitudes(_chain_state(case, seed))
        shift = float((torch.sum(v.conj() * _apply_chain(v, n)) / torch.sum(v.conj() * v)).real)

        def Hs(x):
            return _apply_chain(x, n) - shift * x
        c = case["dtau"] if case["scheme"] == "be" else 0.5 * case["dtau"]
        b = v if case["scheme"] == "be" else v - c * Hs(v)
        x = v
        for _ in range(4):
            x, _res = _krylov(lambda u: u + c * Hs(u), b, x, 10)
        nrm = float(x.norm())
        x = x / nrm
        e = float(torch.sum(x.conj() * _apply_chain(x, n)).real)
        return {"energy": e, "norm": nrm, "discarded": None, "chi": None, "state": x}
    W, v = _local_inputs(case, seed)
    Wt = torch.from_numpy(W).to(DEV)
    if case["op"] == "heff":
        Y = 0.4 * _heff(W, v["L"], v["R"], v["X"])
        return Y + 1.1 * v["Z"] if case["z"] else Y
    if case["op"] == "env":
        T = torch.tensordot(v["Lin"], v["ket"], dims=([2], [0]))        # w a s b'
        T = torch.tensordot(T, Wt, dims=([0, 2], [0, 2]))               # a b' s' w'
        Lo = torch.tensordot(v["bra"].conj(), T, dims=([0, 1], [0, 2])).permute(2, 0, 1)
        T = torch.tensordot(v["Rin"], v["ket"], dims=([1], [2]))        # w b a' s
        T = torch.tensordot(T, Wt, dims=([0, 3], [3, 2]))               # b a' w' s'
        Ro = torch.tensordot(T, v["bra"].conj(), dims=([0, 3], [2, 1])).permute(1, 0, 2)
        return Lo.contiguous(), Ro.contiguous()

    def A(x):
        return v["alpha"] * x + v["c"] * _heff(W, v["L"], v["R"], x)
    if not case["prec"].startswith("mixed"):
        X, res = _krylov(A, v["B"], v["X0"], case["m"])
        return {"X": X, "residual": res, "steps": case["m"]}
    X, res = v["X0"], 1.0
    for _ in range(8):
        if res > 1e-14:
            X, res = _krylov(A, v["B"], X, 10)
    return {"X": X}


# ------------------------------------------------------------------ what a pass cannot do without
def _heff_flops(d, D, la, lb, rb, ra):
    return 8.0 * (D * d * d * la * lb * rb + D * d * d * la * rb * ra +
                  2.0 * D * D * d ** 3 * la * rb)


def work(case):
    if case["op"] == "split":
        m, n, p = case["m"], case["n"], min(case["m"], case["n"])
        return {"bytes": 16.0 * (2 * m * n + case["chi"] * (m + n)),
                "flops": SVD_FLOPS * m * n * p + 16.0 * m * n * min(case["chi"], p)}
    if case["op"] == "step":
        chi = _bonds(case["n"], case["chi"])
        fl = sites = 0.0
        for i in range(case["n"] - 1):
            l, r = chi[i], chi[i + 2]
            fl += 2 * (11 * _heff_flops(2, 5, l, l, r, r) +
                       SVD_FLOPS * (2 * l) * (2 * r) * min(2 * l, 2 * r))
            sites += 2.0 * l * chi[i + 1]
        return {"bytes": 32.0 * sites, "flops": fl * (1.0 if case["scheme"] == "be" else 1.5)}
    W = bulk_w(case["model"])
    D, d = W.shape[0], W.shape[1]
    if case["op"] == "solve":
        l, r = case["chl"], case["chr"]
        return {"bytes": 16.0 * (D * (l * l + r * r) + 3 * d * d * l * r),
                "flops": (case["m"] + 1) * _heff_flops(d, D, l, l, r, r) +
                16.0 * case["m"] * (case["m"] + 3) * d * d * l * r}
    la, lb, rb, ra = case["la"], case["lb"], case["rb"], case["ra"]
    if case["op"] == "heff":
        return {"bytes": 16.0 * (D * (la * lb + rb * ra) +
                                 d * d * (lb * rb + la * ra * (2 if case["z"] else 1))),
                "flops": _heff_flops(d, D, la, lb, rb, ra)}
    return {"bytes": 16.0 * (2 * D * (la * lb + rb * ra) + d * (la * ra + lb * rb)),
            "flops": 16.0 * (D * d * la * lb * rb + D * d * rb * la * ra + D * D * d * d * la * rb)}
