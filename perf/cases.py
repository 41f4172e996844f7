"""The work that is timed: whole calls of the package's public entry points.

Each case names a kind of call, its order (or orders) and its options; ``prepare`` makes the
inputs from the seed with the recipes of ``paper_1405_7537_gb300.workloads`` and the workspace
(or batch object) that a program keeps between calls; ``run`` is one call.
"""
import math

import numpy as np
import torch

from paper_1405_7537_gb300 import binding as B
from paper_1405_7537_gb300 import workloads as W

DEV = "cuda"


def listed():
    return [
        # one small problem solved for its own sake: launches and latency are all there is
        {"name": "eig_uniform_96", "kind": "eig", "spectrum": "uniform", "n": 96, "finder": 0, "vectors": True},
        # the smallest of the benchmark's workloads
        {"name": "eig_uniform_512", "kind": "eig", "spectrum": "uniform", "n": 512, "finder": 0, "vectors": True},
        # an odd order with the accelerated zero finder on the hard spectrum
        {"name": "eig_hard_3001_accel", "kind": "eig", "spectrum": "hard", "n": 3001, "finder": 1, "vectors": True},
        # eigenvalues alone (a secular-equation solve), poles with tight pairs
        {"name": "eigvals_large_6000", "kind": "eig", "spectrum": "large", "n": 6000, "finder": 0, "vectors": False},
        # the headline: lambda and the full V of the hard spectrum
        {"name": "eig_hard_16384", "kind": "eig", "spectrum": "hard", "n": 16384, "finder": 0, "vectors": True},
        # a differentiated eigen-decomposition inside a training step
        {"name": "grad_diff_4096", "kind": "grad", "spectrum": "diff", "n": 4096},
        # the largest differentiated problem (V recomputed in the backward)
        {"name": "grad_large_32768", "kind": "grad", "spectrum": "large", "n": 32768},
        # the lower levels of a divide-and-conquer tree: many tiny problems at once
        {"name": "batch_2000_of_16_128", "kind": "batch", "problems": 2000, "nmin": 16, "nmax": 128},
        # merges of every level in one launch
        {"name": "batch_4096_of_16_2048", "kind": "batch", "problems": 4096, "nmin": 16, "nmax": 2048},
        # a complex Hermitian problem of an odd order
        {"name": "hermitian_hard_2501", "kind": "hermitian", "spectrum": "hard", "n": 2501},
        # divide and conquer on a random tridiagonal matrix, eigenvalues and vectors
        {"name": "tridiag_random_4096", "kind": "tridiag", "spectrum": "random", "n": 4096, "vectors": True},
        # the companion arrowhead problem
        {"name": "arrow_uniform_16384", "kind": "arrow", "n": 16384, "finder": 0},
    ]


def _between(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eig", "eig", "grad", "batch", "hermitian", "tridiag", "arrow"])
    if kind == "eig":
        return {"kind": kind, "spectrum": rng.choice(["uniform", "hard", "large"]), "n": _between(rng, 64, 16384),
                "finder": rng.choice([0, 0, 1]), "vectors": rng.random() < 0.75}
    if kind == "grad":
        return {"kind": kind, "spectrum": rng.choice(["diff", "large"]), "n": _between(rng, 256, 16384)}
    if kind == "batch":
        nmax = _between(rng, 64, 2048)
        # at most the work of the largest listed batch
        most = min(4096.0, 4096.0 * (1024.0 / nmax) ** 2)
        return {"kind": kind, "problems": _between(rng, 16, max(17.0, most)), "nmin": min(16, nmax), "nmax": nmax}
    if kind == "hermitian":
        return {"kind": kind, "spectrum": rng.choice(["uniform", "hard"]), "n": _between(rng, 128, 8192)}
    if kind == "tridiag":
        return {"kind": kind, "spectrum": rng.choice(["random", "schroedinger"]), "n": _between(rng, 200, 4096),
                "vectors": rng.random() < 0.75}
    return {"kind": kind, "n": _between(rng, 128, 16384), "finder": rng.choice([0, 0, 1])}


# -----------------------------------------------------------------------------------------
# inputs
# -----------------------------------------------------------------------------------------
def _problem(spectrum, n, seed):
    """(d, z, rho) of one D + rho z z^T as numpy arrays."""
    if spectrum == "uniform":
        return W.uniform(n, seed)
    if spectrum == "hard":
        return W.hard(n, seed)
    if spectrum == "large":
        return W.large(n, seed, with_W=False)[:3]
    rng = np.random.default_rng(seed)                       # the differentiated workload without W
    return np.sort(rng.uniform(-1.0, 1.0, n))[::-1].copy(), rng.uniform(-1.0, 1.0, n), 0.5


def _tridiagonal(spectrum, n, seed):
    if spectrum == "random":
        return W.tridiagonal(n, seed)
    # -u'' + V u on a uniform grid with a smooth random potential (hardly anything deflates)
    rng = np.random.default_rng(seed)
    x = np.linspace(0.0, 1.0, n)
    v = sum(rng.normal() / (1 + k) * np.cos(math.pi * k * x + rng.uniform(0, 2 * math.pi)) for k in range(8))
    return 2.0 + v / n, np.full(n - 1, -1.0)


def _batch(case, seed):
    """(sizes, offs, d, z, rho): the problems of a batch, with the orders fixed by the case."""
    sizes, _ = W.batch_sizes(case["problems"], 3, case["nmin"], case["nmax"])
    offs = np.concatenate([[0], np.cumsum(sizes)])
    rng = np.random.default_rng(seed)
    d, z = rng.uniform(-1.0, 1.0, offs[-1]), rng.uniform(-1.0, 1.0, offs[-1])
    for p in range(sizes.size):
        d[offs[p]:offs[p + 1]] = np.sort(d[offs[p]:offs[p + 1]])[::-1]
    return sizes, offs, d, z, rng.uniform(0.1, 10.0, sizes.size)


def _dev(x):
    return torch.tensor(np.ascontiguousarray(x), device=DEV)


def _randn(shape, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, dtype=torch.float64, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("eig", "grad"):
        n = case["n"]
        d, z, rho = _problem(case["spectrum"], n, seed)
        s.update(d=_dev(d), z=_dev(z), rho=float(rho))
        if kind == "eig":
            s["ws"] = B.workspace(n, DEV)
            s["options"] = B.default_options(zero_finder=case["finder"])
        else:
            s["d"].requires_grad_(True)
            s["z"].requires_grad_(True)
            s["rho"] = torch.tensor(float(rho), dtype=torch.float64, device=DEV, requires_grad=True)
            # the cotangents of lambda and V; dL/dV in V's own layout, as a loss of V's entries gives it
            s["w"] = _randn((n,), seed + 1)
            s["W"] = _randn((n, n), seed + 2).t()
    elif kind == "batch":
        sizes, _, d, z, rho = _batch(case, seed)
        s["batch"] = B.Batch(sizes, device=DEV)
        s.update(d=_dev(d), z=_dev(z), rho=_dev(rho))
    elif kind == "hermitian":
        d, z, rho = W.hermitian(case["n"], seed, "hard" if case["spectrum"] == "hard" else "uniform")
        s.update(d=_dev(d), z=_dev(z), rho=float(rho), ws=B.hermitian_workspace(case["n"], DEV))
    elif kind == "tridiag":
        a, b = _tridiagonal(case["spectrum"], case["n"], seed)
        s.update(a=_dev(a), b=_dev(b), ws=B.tridiag_workspace(case["n"], DEV))
    else:
        d, z, alpha = W.arrowhead(case["n"], seed)
        s.update(d=_dev(d), z=_dev(z), alpha=float(alpha), ws=B.arrow_workspace(case["n"], DEV),
                 options=B.default_options(zero_finder=case["finder"]))
    return s


# -----------------------------------------------------------------------------------------
# one call
# -----------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "eig":
        return B.eig(s["d"], s["z"], s["rho"], want_vectors=case["vectors"], options=s["options"], ws=s["ws"],
                     check=False)
    if kind == "grad":
        lam, V = B.eigh_dpr1(s["d"], s["z"], s["rho"])
        gd, gz, gr = torch.autograd.grad((lam, V), (s["d"], s["z"], s["rho"]), (s["w"], s["W"]))
        return {"lam": lam, "V": V, "grad_d": gd, "grad_z": gz, "grad_rho": gr}
    if kind == "batch":
        b = s["batch"]
        b.solve(s["d"], s["z"], s["rho"])
        return {"lam": b.lam, "Vt": b.Vt, "sigma": b.sigma, "mu": b.mu, "xnorm": b.xnorm}
    if kind == "hermitian":
        return B.eig_hermitian(s["d"], s["z"], s["rho"], ws=s["ws"], check=False)
    if kind == "tridiag":
        lam, Qt = B.eigh_tridiagonal(s["a"], s["b"], want_vectors=case["vectors"], ws=s["ws"], check=False)
        return {"lam": lam, "Qt": Qt}
    return B.eig_arrowhead(s["d"], s["z"], s["alpha"], options=s["options"], ws=s["ws"], check=False)


def _orders(case):
    """The expected sum of n_p and of n_p^2 over the problems of a batch."""
    lo, hi, p = case["nmin"], case["nmax"], case["problems"]
    ln = math.log(hi / lo) if hi > lo else 1.0
    m1 = (hi - lo) / ln if hi > lo else float(lo)
    m2 = (hi * hi - lo * lo) / (2 * ln) if hi > lo else float(lo * lo)
    return p * m1, p * m2


def work(case):
    """Inputs read and outputs written once; binary64 operations of forming the inverse's elements
    (3 per term), one evaluation of the secular function (5) and an eigenvector component (6), of the
    adjoint (15 per component), and of the products of a divide and conquer without deflation."""
    kind = case["kind"]
    if kind == "batch":
        m1, m2 = _orders(case)
        return {"bytes": 8 * (6 * m1 + m2), "flops": 14 * m2}
    n = float(case["n"])
    if kind == "eig":
        v = case["vectors"]
        return {"bytes": 8 * (6 * n + (n * n if v else 0)), "flops": (14 if v else 8) * n * n}
    if kind == "grad":
        return {"bytes": 8 * (10 * n + 2 * n * n), "flops": 29 * n * n}
    if kind == "hermitian":
        return {"bytes": 8 * (7 * n + 2 * n * n), "flops": 16 * n * n}
    if kind == "tridiag":
        v = case["vectors"]
        return {"bytes": 8 * (3 * n + (n * n if v else 0)), "flops": (4.0 / 3.0 if v else 1.0 / 3.0) * n ** 3}
    return {"bytes": 8 * (6 * n + n * n), "flops": 14 * n * n}


# -----------------------------------------------------------------------------------------
# reference values: the secular equation in double-double, vectorised in plain torch
# -----------------------------------------------------------------------------------------
def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _two_prod(a, b):
    def split(x):
        c = x * 134217729.0
        h = c - (c - x)
        return h, x - h
    p = a * b
    ah, al = split(a)
    bh, bl = split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _dd_sum(h, l):
    """Sum of h + l over the last axis in double-double (a pairwise tree)."""
    while h.shape[-1] > 1:
        m = h.shape[-1]
        if m & 1:
            h = torch.nn.functional.pad(h, (0, 1))
            l = torch.nn.functional.pad(l, (0, 1))
            m += 1
        s, e = _two_sum(h[..., :m // 2], h[..., m // 2:])
        l = l[..., :m // 2] + l[..., m // 2:] + e
        h, l = s, l
        h, l = _two_sum(h, l)
    return h[..., 0], l[..., 0]


def _diffs(d, di, mu, lo):
    """d_j - d_i - (mu + lo) in double-double; d [P, 1, n], the others [P, R, 1]."""
    Dh, Dl = _two_sum(d, -di)
    s, e = _two_sum(Dh, -mu)
    return _two_sum(s, e + Dl - lo)


def _secular(d, zz, zl, di, mu, lo, ch, cl, slope):
    """c + slope (mu + lo) + sum_j zeta_j^2 / (d_j - d_i - mu - lo) in double-double."""
    xh, xl = _diffs(d, di, mu, lo)
    q = zz / xh
    p, e = _two_prod(q, xh)
    r = (((zz - p) - e) + (zl - q * xl)) / xh
    q, r = torch.where(zz == 0, torch.zeros_like(q), q), torch.where(zz == 0, torch.zeros_like(r), r)
    h, l = _dd_sum(q, r)
    s, e = _two_sum(h, ch)
    l = l + e + cl
    if slope:
        s, e = _two_sum(s, mu[..., 0])
        l = l + e + lo[..., 0]
    return s + l


def _pairs(d, z, const, slope, rows, top):
    """Eigenvalues as d_i + (mu + lo): d, z [P, n] (poles decreasing, zero weights padded at the end),
    const(i) -> double-double [P, R] constant of the secular function, rows eigenvalues per problem
    and top [P] a bound of their distance beyond the exterior poles.  The function increases between
    the poles.  Yields (k0, k1, i, di, mu, lo) for chunks of rows."""
    P, n = d.shape
    zz, zl = _two_prod(z, z)
    D, ZZ, ZL = d[:, None, :], zz[:, None, :], zl[:, None, :]
    chunk = max(1, int(2 ** 26 // (P * n)))
    for k0 in range(0, rows, chunk):
        k1 = min(rows, k0 + chunk)
        k = torch.arange(k0, k1, device=d.device)
        up, dn = (k - 1).clamp(0, n - 1), k.clamp(0, n - 1)
        dk, du = d[:, dn], d[:, up]
        tau = torch.where((k > 0) & (k < n), 0.5 * (du - dk), top[:, None].expand(P, k1 - k0))
        zero = torch.zeros_like(tau)[..., None]
        # the nearer pole: the sign at the midpoint
        ch, cl = const(dn)
        mid = _secular(D, ZZ, ZL, dk[..., None], tau[..., None], zero, ch, cl, slope)
        low = torch.where((k == 0)[None, :], torch.ones_like(mid, dtype=torch.bool), mid > 0)
        low = torch.where((k >= n)[None, :], torch.zeros_like(low), low)
        i = torch.where(low, dn[None, :], up[None, :])
        di = torch.gather(d, 1, i)
        ch, cl = const(i)
        sgn = torch.where(low, 1.0, -1.0).to(torch.float64)
        hi = (tau.clamp_min(1e-290) * (1 + 2.0 ** -40)).contiguous().view(torch.int64)
        lo = torch.full_like(tau, 1e-300).view(torch.int64)
        for _ in range(64):
            m = lo + (hi - lo) // 2
            t = sgn * m.view(torch.float64)
            F = _secular(D, ZZ, ZL, di[..., None], t[..., None], zero, ch, cl, slope)
            above = torch.where(low, F > 0, F < 0)
            hi, lo = torch.where(above, m, hi), torch.where(above, lo, m)
        mu = sgn * lo.view(torch.float64)
        F = _secular(D, ZZ, ZL, di[..., None], mu[..., None], zero, ch, cl, slope)
        xh, _ = _diffs(D, di[..., None], mu[..., None], zero)
        dF = torch.where(ZZ == 0, torch.zeros_like(xh), ZZ / (xh * xh)).sum(-1) + (1.0 if slope else 0.0)
        yield k0, k1, i, di, mu, -F / dF


def _eig_exact(d, z, const, slope, rows, top, arrow=False, vectors=True):
    """lambda [P, rows], rows of eigenvectors [P, rows, n (+ 1)], ||x|| [P, rows] and the pairs."""
    P, n = d.shape
    m = n + 1 if arrow else n
    lam, xn = (torch.empty(P, rows, dtype=torch.float64, device=d.device) for _ in range(2))
    V = torch.empty(P, rows, m, dtype=torch.float64, device=d.device) if vectors else None
    pairs = []
    for k0, k1, i, di, mu, lo in _pairs(d, z, const, slope, rows, top):
        s, e = _two_sum(di, mu)
        lam[:, k0:k1] = s + (e + lo)
        xh, xl = _diffs(d[:, None, :], di[..., None], mu[..., None], lo[..., None])
        x = z[:, None, :] / (xh + xl)
        x = torch.where(z[:, None, :] == 0, torch.zeros_like(x), x)
        if arrow:
            x = torch.cat([x, torch.full_like(x[..., :1], -1.0)], -1)
        big = x.abs().amax(-1, keepdim=True)
        nrm = (x / big).square().sum(-1, keepdim=True).sqrt() * big
        xn[:, k0:k1] = nrm[..., 0]
        if vectors:
            V[:, k0:k1] = x / nrm
        pairs.append((di, mu, lo))
    return lam, V, xn, pairs


def _dpr1_exact(d, z, rho, vectors=True):
    """d, z [P, n], rho [P]."""
    inv = 1.0 / rho
    p, e = _two_prod(inv, rho)
    inl = ((1.0 - p) - e) / rho

    def const(i):
        shape = (d.shape[0], i.shape[-1])
        return inv[:, None].expand(shape), inl[:, None].expand(shape)

    return _eig_exact(d, z, const, False, d.shape[1], 2.0 * rho * z.square().sum(-1), vectors=vectors)


def _gradients(d, z, rho, pairs, w, Wm):
    """The adjoint of (lambda, V): the sums without the dominant component p of each row."""
    gd, gz, gr = torch.zeros_like(d), torch.zeros_like(z), torch.zeros((), dtype=torch.float64, device=d.device)
    k0 = 0
    for di, mu, lo in pairs:
        k1 = k0 + di.shape[-1]
        xh, xl = _diffs(d[None, None, :], di[..., None], mu[..., None], lo[..., None])
        s = (xh + xl)[0]
        x = z[None, :] / s
        big = x.abs().amax(-1, keepdim=True)
        nrm = (x / big).square().sum(-1, keepdim=True).sqrt() * big
        v = x / nrm
        vb = Wm[:, k0:k1].t()
        p = v.abs().argmax(-1, keepdim=True)
        vp, vbp, sp = v.gather(1, p), vb.gather(1, p), s.gather(1, p)
        v0 = v.scatter(1, p, 0.0)                               # without component p
        S2, Pm = (v0 * v0).sum(-1, keepdim=True), (v0 * vb).sum(-1, keepdim=True)
        c = vp * vbp + Pm
        gp = vbp * S2 - vp * Pm
        g = vb - v * c
        Lam = w[k0:k1, None] + (g * v0 / s).sum(-1, keepdim=True)
        Tp = gp * vp / sp
        lb = Lam + Tp
        db = (lb * v * v - g * v / s).scatter(1, p, Lam * vp * vp - Tp * S2)
        zb = ((g / s - 2 * lb * v) / nrm).scatter(1, p, (gp / sp * (S2 - vp * vp) - 2 * Lam * vp) / nrm)
        gd += db.sum(0)
        gz += zb.sum(0)
        gr = gr + (lb / (rho * nrm).square()).sum()
        k0 = k1
    return gd, gz, gr


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        if case["problems"] * case["nmax"] ** 2 > 3e8:
            return None
        sizes, offs, d, z, rho = _batch(case, seed)
        P, m = sizes.size, int(sizes.max())
        dp = np.empty((P, m))
        zp = np.zeros((P, m))
        for p in range(P):
            n = sizes[p]
            dp[p, :n], zp[p, :n] = d[offs[p]:offs[p + 1]], z[offs[p]:offs[p + 1]]
            dp[p, n:] = -5.0 - np.arange(m - n)                  # zero weights: no term
        lam, V, xn, _ = _dpr1_exact(_dev(dp), _dev(zp), _dev(rho))
        cut = lambda t: torch.cat([t[p, :sizes[p]] for p in range(P)])                          # noqa: E731
        Vt = torch.cat([V[p, :sizes[p], :sizes[p]].reshape(-1) for p in range(P)])
        return {"lam": cut(lam), "Vt": Vt, "sigma": None, "mu": None, "xnorm": cut(xn)}
    n = case["n"]
    if n > 17000:
        return None                                              # minutes in double-double
    if kind == "tridiag":
        a, b = (_dev(x) for x in _tridiagonal(case["spectrum"], n, seed))
        T = torch.diag(a) + torch.diag(b, 1) + torch.diag(b, -1)
        return {"lam": torch.linalg.eigvalsh(T).flip(0), "Qt": None}
    if kind == "arrow":
        d, z, alpha = W.arrowhead(n, seed)
        d, z = _dev(d)[None], _dev(z)[None]

        def const(i):
            di = d[0][i] if i.dim() == 2 else d[:, i]
            return _two_sum(di, torch.full_like(di, -alpha))

        top = (z.square().sum(-1).sqrt() + abs(alpha) + d.abs().amax(-1)) * 2
        lam, V, xn, _ = _eig_exact(d, z, const, True, n + 1, top, arrow=True)
        return {"lam": lam[0], "Vt": V[0], "sigma": None, "mu": None, "xnorm": xn[0]}
    if kind == "hermitian":
        d, z, rho = W.hermitian(n, seed, "hard" if case["spectrum"] == "hard" else "uniform")
        mod = np.abs(z)
        lam, V, xn, _ = _dpr1_exact(_dev(d)[None], _dev(mod)[None], _dev(np.array([rho])))
        return {"lam": lam[0], "Vt": V[0] * _dev(z / mod)[None, :], "sigma": None, "mu": None, "xnorm": xn[0]}
    d, z, rho = _problem(case["spectrum"], n, seed)
    lam, V, xn, pairs = _dpr1_exact(_dev(d)[None], _dev(z)[None], _dev(np.array([rho])),
                                    vectors=kind == "grad" or case["vectors"])
    if kind == "eig":
        return {"lam": lam[0], "Vt": V[0] if V is not None else None, "sigma": None, "mu": None, "xnorm": xn[0]}
    gd, gz, gr = _gradients(_dev(d), _dev(z), float(rho), pairs, _randn((n,), seed + 1), _randn((n, n), seed + 2).t())
    return {"lam": lam[0], "V": V[0].t(), "grad_d": gd, "grad_z": gz, "grad_rho": gr}
