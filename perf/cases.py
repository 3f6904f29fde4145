"""Workloads of the library's public entry points, for timing and for comparing outputs.

Every case is one call (or the call and the one that always follows it) that a pricing
program makes: the transition counts of a quantization tree (Algorithm III and the
path-wise Algorithm II of Pages & Wilbertz, arXiv:1101.3228), the counting step on given
samples, the backward induction, the swing option, the whole price, and the building of
the grids.  Sizes are those of the five workloads of this project, of the paper's own
scenario and of the tests, with fewer layers or samples where a whole step takes
seconds.

A program keeps one context for all of its calls, so the cases share one.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_1101_3228_gb300 import binding as B

_CTX = {}


def _ctx():
    if "ctx" not in _CTX:
        _CTX["ctx"] = B.Context(torch.cuda.current_device())
    return _CTX["ctx"]


# ---------------------------------------------------------------------------- the cases

def listed():
    return [
        # the whole price of the 1-d Black-Scholes put: ten exercise dates, FP64 samples,
        # grids and payoffs still in host memory (a calculator's call)
        dict(name="price_1d", kind="price", d=1, n=10, N=100, uneven=False, M=10**6, f64=True, u32=False,
             host=True),
        # the smallest call: a four-date tree with a few thousand samples, where the fixed
        # cost of a call is what a user waits for (calibration loops, tests)
        dict(name="tree_2d_small", kind="tree", d=2, n=4, N=64, uneven=False, M=3000, f64=False, u32=False),
        # the 2-factor energy model at its full size: 100 daily layers, 10^7 pairs each
        dict(name="tree_2d", kind="tree", d=2, n=100, N=500, uneven=False, M=10**7, f64=False, u32=False),
        # the paper's scenario as one price: a year of daily exercise, 10^5 pairs per day
        dict(name="price_2d_year", kind="price", d=2, n=365, N=500, uneven=False, M=10**5, f64=False, u32=True,
             host=False),
        # the same 2-factor model by paths (Algorithm II)
        dict(name="paths_2d", kind="paths", d=2, n=100, N=500, uneven=False, M=10**6, f64=False, u32=False,
             euler=False),
        # the 4-asset basket: grids growing from 200 to 2000 points over 50 dates
        dict(name="tree_4d", kind="tree", d=4, n=50, N=2000, uneven=True, M=10**6, f64=False, u32=False),
        # the 8-d chain: 4000-point grids, a tenth of a year's dates per call
        dict(name="tree_8d", kind="tree", d=8, n=12, N=4000, uneven=False, M=2 * 10**6, f64=False, u32=False),
        # the 10-d max-call chain: the largest grids, 32-bit counts
        dict(name="tree_10d", kind="tree", d=10, n=6, N=8000, uneven=False, M=10**6, f64=False, u32=True),
        # a user's own samples (any chain, not only AR(1)): one layer pair in FP64, with cells
        dict(name="samples_3d", kind="samples", d=3, NA=777, NB=1001, M=1000003, u32=False, cells=True),
        # a gas contract: volume between 20 and 60 rights on the 2-factor tree
        dict(name="swing_2d", kind="swing", n=100, N=500, Qmin=20, Qmax=60, u32=False),
        # re-pricing another payoff on a stored 8-d tree: only the backward induction
        dict(name="backward_8d", kind="backward", n=8, N=4000, u32=False),
        # building the grids of a new model by sample Lloyd: the first basket dates
        dict(name="grids_4d", kind="grids", d=4, n=6, N=1100, uneven=True, method=B.GRID_KMEANS,
             samples=100000, iters=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kinds = ["tree", "tree", "tree", "tree", "price", "paths", "samples", "swing", "backward", "grids"]
    while True:
        kind = rng.choice(kinds)
        if kind in ("tree", "price", "paths"):
            d = rng.randint(1, 4) if kind == "paths" else rng.randint(1, 10)
            top = {1: 400, 2: 1000, 3: 1500, 4: 2000}.get(d, 8000)
            f64 = d <= 2 and rng.random() < 0.3
            case = dict(kind=kind, d=d, n=_log_int(rng, 1, 365 if d <= 2 else 50), N=_log_int(rng, 16, top),
                        uneven=rng.random() < 0.3, M=_log_int(rng, 1000, 10**7 if d <= 2 else 2 * 10**6), f64=f64,
                        u32=rng.random() < 0.4)
            if kind == "price":
                case["host"] = rng.random() < 0.5
            if kind == "paths":
                case["euler"] = rng.random() < 0.4
            if f64 and case["n"] * case["M"] > 3 * 10**7:
                continue
        elif kind == "samples":
            d = rng.randint(1, 10)
            top = 1000 if d <= 2 else 4000
            case = dict(kind=kind, d=d, NA=_log_int(rng, 16, top), NB=_log_int(rng, 16, top),
                        M=_log_int(rng, 1000, 2 * 10**6), u32=rng.random() < 0.4, cells=rng.random() < 0.5)
        elif kind == "swing":
            n = _log_int(rng, 5, 100)
            qmin = rng.randint(0, n // 2)
            case = dict(kind=kind, n=n, N=_log_int(rng, 20, 500), Qmin=qmin, Qmax=rng.randint(max(1, qmin), n),
                        u32=rng.random() < 0.4)
        elif kind == "backward":
            case = dict(kind=kind, n=_log_int(rng, 1, 365), N=_log_int(rng, 50, 8000), u32=rng.random() < 0.5)
        else:
            d = rng.randint(2, 8)
            case = dict(kind=kind, d=d, n=rng.randint(1, 6), N=_log_int(rng, 50, 2000), uneven=rng.random() < 0.5,
                        method=B.GRID_KMEANS if rng.random() < 0.7 else B.GRID_PRODUCT,
                        samples=_log_int(rng, 20000, 200000), iters=rng.randint(5, 20))
        # no dearer than the largest listed case, in brute-force distances and in memory
        if _distances(case) <= 10**12 * 2 / max(2, case.get("d", 2)) and _count_entries(case) * 8 <= 1.5e9:
            return case


def _sizes(case):
    """Grid sizes N_0 = 1, N_1, ..., N_n."""
    n, N = case["n"], case["N"]
    if case.get("uneven"):
        lo = max(1, N // 10)
        rest = [int(round(lo + (N - lo) * k / max(1, n - 1))) for k in range(n)]
    else:
        rest = [N] * n
    return np.array([1] + rest, dtype=np.int64)


def _count_entries(case):
    if case["kind"] == "samples":
        return case["NA"] * case["NB"]
    if case["kind"] == "grids":
        return 0
    N = _sizes(case)
    return int(np.sum(N[:-1] * N[1:]))


def _distances(case):
    """Distances that brute force would evaluate."""
    kind = case["kind"]
    if kind in ("tree", "price"):
        N = _sizes(case)
        return int(case["M"] * np.sum(N[:-1] + N[1:]))
    if kind == "paths":
        return int(case["M"] * np.sum(_sizes(case)))
    if kind == "samples":
        return case["M"] * (case["NA"] + case["NB"])
    if kind == "swing":
        return _count_entries(case) * (case["Qmax"] + 1)
    if kind == "backward":
        return _count_entries(case)
    if case["method"] == B.GRID_KMEANS:
        return int(sum({int(v) for v in _sizes(case)[1:]}) * case["samples"] * case["iters"])
    return int(np.sum(_sizes(case)))


# ---------------------------------------------------------------------------- models and grids

def _chain(case, rng):
    """AR(1) chain X_{k+1} = A X_k + b + T eps with its marginal means and factors: Black-Scholes
    for d = 1, the 2-factor OU model for d = 2, correlated log-prices for d = 3 and 4, a
    correlated AR(1) chain above.  The seed moves the volatilities by a few percent."""
    d, n = case["d"], case["n"]
    vol = 1.0 + 0.05 * rng.uniform(-1.0, 1.0)
    m0 = np.zeros(d)
    b = np.zeros(d)
    if d == 1:
        dt, sig, r = 1.0 / max(n, 1), 0.2 * vol, 0.05
        A, Q = np.eye(1), np.array([[sig * sig * dt]])
        b[0] = (r - 0.5 * sig * sig) * dt
        m0[0] = math.log(100.0)
    elif d == 2:
        dt, al = 1.0 / 365.0, np.array([0.5, 5.0])
        sg, R = np.array([0.3, 0.6]) * vol, np.array([[1.0, -0.3], [-0.3, 1.0]])
        s = al[:, None] + al[None, :]
        A, Q = np.diag(np.exp(-al * dt)), sg[:, None] * sg[None, :] * R * (1.0 - np.exp(-s * dt)) / s
    elif d <= 4:
        dt, sg = 1.0 / 50.0, np.linspace(0.2, 0.4, d) * vol
        R = np.full((d, d), 0.5) + 0.5 * np.eye(d)
        A, Q = np.eye(d), sg[:, None] * sg[None, :] * R * dt
        b = (0.05 - 0.5 * sg * sg) * dt
        m0[:] = math.log(100.0)
    else:
        Qm, _ = np.linalg.qr(rng.standard_normal((d, d)))
        A, Q = np.diag(np.linspace(0.9, 0.99, d)), Qm @ np.diag(np.logspace(-4.0, -2.0, d)) @ Qm.T * vol
    Q = 0.5 * (Q + Q.T)
    mean, cov = [m0], [np.zeros((d, d))]
    for _ in range(n):
        mean.append(A @ mean[-1] + b)
        cov.append(A @ cov[-1] @ A.T + Q)
    L = [np.zeros((d, d))] + [np.linalg.cholesky(0.5 * (S + S.T)) for S in cov[1:]]
    rep = lambda a: np.repeat(a[None], n, axis=0)  # noqa: E731
    return types.SimpleNamespace(d=d, n=n, N=_sizes(case), A=rep(A), b=rep(b), T=rep(np.linalg.cholesky(Q)),
                                 m=np.stack(mean), L=np.stack(L))


def _quantizer_1d(N):
    """Near-stationary N-point quantizer of N(0, 1): Lloyd from the quantiles, FP64."""
    x = torch.special.ndtri((torch.arange(N, dtype=torch.float64) + 0.5) / N)
    pdf = lambda z: torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)  # noqa: E731
    inf = torch.full((1,), math.inf, dtype=torch.float64)
    for _ in range(60):
        mid = 0.5 * (x[1:] + x[:-1])
        lo, hi = torch.cat([-inf, mid]), torch.cat([mid, inf])
        mass = torch.special.ndtr(hi) - torch.special.ndtr(lo)
        x = (pdf(lo) - pdf(hi)) / mass
        x = 0.5 * (x - x.flip(0))
    return x.numpy()


def _kmeans(N, d, gen, iters=5):
    """Sample Lloyd on N(0, I_d) draws; fixed-point sums, so that the result is the same every time."""
    S = max(10 * N, 20000)
    Z = torch.randn(S, d, generator=gen, device="cuda", dtype=torch.float32)
    C = Z[:N].clone()
    for _ in range(iters):
        idx = torch.empty(S, dtype=torch.int64, device="cuda")
        half = 0.5 * (C * C).sum(1)
        for s in range(0, S, 16384):
            idx[s:s + 16384] = (half[None, :] - Z[s:s + 16384] @ C.T).argmin(1)
        sums = torch.zeros(N, d, dtype=torch.int64, device="cuda").index_add_(
            0, idx, (Z.double() * 2.0**32).round().long())
        cnt = torch.bincount(idx, minlength=N)
        keep = cnt > 0
        C[keep] = (sums[keep].double() / 2.0**32 / cnt[keep, None]).float()
    return C.double().cpu().numpy()


def _base_grid(N, d, gen):
    if N == 1:
        return np.zeros((1, d))
    if d == 1:
        return _quantizer_1d(N)[:, None]
    if d == 2:
        a = next(v for v in range(int(math.isqrt(N)), 0, -1) if N % v == 0)
        if a > 1:
            u, v = np.meshgrid(_quantizer_1d(a), _quantizer_1d(N // a), indexing="ij")
            return np.stack([u.ravel(), v.ravel()], axis=1)
    return _kmeans(N, d, gen)


def _grids(model, gen):
    base, out = {}, []
    for k in range(model.n + 1):
        N = int(model.N[k])
        if N not in base:
            base[N] = _base_grid(N, model.d, gen)
        out.append(model.m[k][None, :] + base[N] @ model.L[k].T)
    return np.ascontiguousarray(np.concatenate(out, axis=0))


def _payoff(d, x):
    """Put on the price (d = 1), on exp(x1 + x2) (d = 2), on the basket mean above; discounting left out."""
    if d == 1:
        return np.maximum(100.0 - np.exp(x[:, 0]), 0.0)
    if d == 2:
        return np.maximum(1.0 - np.exp(x.sum(1)), 0.0)
    s = np.exp(x).mean(1)
    return np.maximum((100.0 if d <= 4 else 1.0) - s, 0.0)


def _tree_counts(n, N, u32, gen):
    """Transition counts of a 2-factor chain of n dates on N-point product grids, from 2 10^5 pairs a date."""
    M = 200000
    a = next(v for v in range(int(math.isqrt(N)), 0, -1) if N % v == 0)
    axes = [torch.from_numpy(_quantizer_1d(v)).cuda() for v in (a, N // a)]
    mids = [0.5 * (x[1:] + x[:-1]) for x in axes]
    cell = lambda z: torch.bucketize(z[:, 0], mids[0]) * (N // a) + torch.bucketize(z[:, 1], mids[1])  # noqa: E731
    out = []
    for k in range(n):
        # whitened states of consecutive dates: correlation grows with the date
        c = math.sqrt(k / (k + 1.0))
        z = torch.randn(M, 2, generator=gen, device="cuda", dtype=torch.float64)
        e = torch.randn(M, 2, generator=gen, device="cuda", dtype=torch.float64)
        j = cell(c * z + math.sqrt(1.0 - c * c) * e)
        i, rows = (torch.zeros_like(j), 1) if k == 0 else (cell(z), N)
        out.append(torch.bincount(i * N + j, minlength=rows * N))
    flat = torch.cat(out)
    return flat.int() if u32 else flat


def _stored_counts(n, N, u32, gen):
    """Counts of a high-dimensional tree: every row spreads 250 pairs over its columns."""
    out = [torch.bincount(torch.randint(0, N, (250 * N,), generator=gen, device="cuda"), minlength=N)]
    for _ in range(1, n):
        i = torch.arange(N, device="cuda").repeat_interleave(250)
        j = torch.randint(0, N, (250 * N,), generator=gen, device="cuda")
        out.append(torch.bincount(i * N + j, minlength=N * N))
    flat = torch.cat(out)
    return flat.int() if u32 else flat


# ---------------------------------------------------------------------------- prepare and run

def prepare(case, seed):
    torch.backends.cuda.matmul.allow_tf32 = False
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    st = dict(kind=kind, ctx=_ctx(), case=case, seed=0xC0FFEE0000 + int(seed))
    if kind in ("tree", "price", "paths"):
        model = _chain(case, rng)
        grids = _grids(model, gen)
        st["model"] = model
        st["opts"] = B.options(prec=B.PREC_F64 if case["f64"] else B.PREC_F32,
                               counts_type=B.COUNTS_U32 if case["u32"] else B.COUNTS_I64)
        if kind == "price":
            phi = _payoff(model.d, grids)
            st["grids"], st["phi"] = ((grids, phi) if case["host"] else
                                      (torch.from_numpy(grids).cuda(), torch.from_numpy(phi).cuda()))
        else:
            st["grids"] = torch.from_numpy(grids).cuda()
        if kind == "paths" and case["euler"]:
            # a square-root diffusion: innovations scaled by sqrt(max(1 + beta x, 0))
            st["euler"] = (np.ones((model.n, model.d)), np.full((model.n, model.d), 0.2 / (1.0 + abs(model.m[0, 0]))))
    elif kind == "samples":
        d, M = case["d"], case["M"]
        S = torch.from_numpy(np.linalg.cholesky(np.full((d, d), 0.5) + 0.5 * np.eye(d))).cuda()
        X = torch.randn(M, d, generator=gen, device="cuda", dtype=torch.float64) @ S.T
        Y = 0.95 * X + 0.3 * torch.randn(M, d, generator=gen, device="cuda", dtype=torch.float64) @ S.T
        for key, N in (("gA", case["NA"]), ("gB", case["NB"])):
            st[key] = (torch.from_numpy(_base_grid(N, d, gen)).cuda() @ S.T).contiguous()
        st["X"], st["Y"] = X.contiguous(), Y.contiguous()
        st["opts"] = B.options(counts_type=B.COUNTS_U32 if case["u32"] else B.COUNTS_I64)
    elif kind in ("swing", "backward"):
        st["N"] = np.array([1] + [case["N"]] * case["n"], dtype=np.int64)
        st["ct"] = B.COUNTS_U32 if case["u32"] else B.COUNTS_I64
        make = _tree_counts if kind == "swing" else _stored_counts
        st["counts"] = make(case["n"], case["N"], case["u32"], gen)
        pts = int(st["N"].sum())
        v = torch.exp(0.3 * torch.randn(pts, generator=gen, device="cuda", dtype=torch.float64))
        st["v"] = v - 1.0 if kind == "swing" else torch.clamp(1.0 - v, min=0.0)
    else:
        st["model"] = _chain(case, rng)
        st["seed"] = int(seed)
    return st


def run(state):
    ctx, kind, case = state["ctx"], state["kind"], state["case"]
    if kind == "tree":
        counts, _, _ = ctx.transitions(state["model"], state["grids"], case["M"], state["seed"], state["opts"],
                                       want_stats=False)
        return counts
    if kind == "paths":
        counts, _, _ = ctx.transitions_pathwise(state["model"], state["grids"], case["M"], state["seed"],
                                                state["opts"], euler=state.get("euler"), want_stats=False)
        return counts
    if kind == "price":
        price, _ = ctx.price(state["model"], state["grids"], case["M"], state["seed"], state["phi"], state["opts"])
        return price
    if kind == "samples":
        counts, _, ii, jj = ctx.counts_from_samples(state["gA"], state["gB"], state["X"], state["Y"], state["opts"],
                                                    want_cells=case["cells"])
        return [counts, ii, jj] if case["cells"] else counts
    if kind == "swing":
        P, price = ctx.swing(state["N"], state["counts"], state["v"], case["Qmin"], case["Qmax"], state["ct"])
        return [P, price]
    if kind == "backward":
        return ctx.backward(state["N"], state["counts"], state["v"], state["ct"])
    return ctx.build_grids(state["model"], case["method"], samples=case["samples"], iters=case["iters"],
                           seed=state["seed"])


# ---------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Bytes: grids, samples, counts and values once each.  Flops: for a drawn pair its normals
    (about 40 operations each: logarithm, square root, sine, cosine), the AR(1) map and one
    distance per search; for a given count a multiply-add per value it meets."""
    kind, d = case["kind"], case.get("d", 0)
    ent = _count_entries(case)
    csize = 4 if case.get("u32") else 8
    if kind in ("tree", "price", "paths"):
        pts = int(_sizes(case).sum())
        searches = 1 if kind == "paths" else 2
        normals = d if kind == "paths" else 2 * d
        per = 40 * normals + 2 * d * d + d * (d + 1) * searches + 3 * d * searches
        flops = case["M"] * case["n"] * per
        if kind == "price":                       # the counts never leave the call
            return {"bytes": 8 * pts * (d + 1), "flops": flops + 2 * ent}
        return {"bytes": 8 * pts * d + csize * ent, "flops": flops}
    if kind == "samples":
        cells = 8 * case["M"] if case["cells"] else 0
        return {"bytes": 16 * case["M"] * d + 8 * d * (case["NA"] + case["NB"]) + csize * ent + cells,
                "flops": 6 * d * case["M"]}
    pts = int(_sizes(case).sum())
    if kind == "swing":
        nq = case["Qmax"] + 1
        return {"bytes": csize * ent + 8 * pts * (nq + 1), "flops": 2 * ent * nq}
    if kind == "backward":
        return {"bytes": csize * ent + 16 * pts, "flops": 2 * ent}
    # sample Lloyd: the draws once, one distance per draw and iteration, the grids written
    km = len({int(v) for v in _sizes(case)[1:]}) * case["samples"] if case["method"] == B.GRID_KMEANS else 0
    return {"bytes": 8 * pts * d, "flops": km * (40 * d + 3 * d * case["iters"]) + 2 * pts * d * d}


# ---------------------------------------------------------------------------- the same in plain 64-bit torch

def _philox(m, k, seed):
    """Philox4x32-10 of counter (m_lo, m_hi, k, 0): four int64 tensors of 32-bit words."""
    mask = 0xFFFFFFFF
    c = [m & mask, m >> 32, torch.full_like(m, k), torch.zeros_like(m)]
    k0, k1 = seed & mask, seed >> 32
    hi = lambda a, x: ((a * (x >> 16)) + ((a * (x & 0xFFFF)) >> 16)) >> 16  # noqa: E731
    for _ in range(10):
        h0, l0 = hi(0xD2511F53, c[0]), (0xD2511F53 * c[0]) & mask
        h1, l1 = hi(0xCD9E8D57, c[2]), (0xCD9E8D57 * c[2]) & mask
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _exact_price_1d(case, seed):
    """The price of a 1-d tree with FP64 samples: the pairs drawn, projected and counted in torch."""
    st = prepare(case, seed)
    mdl, M = st["model"], case["M"]
    grids = torch.as_tensor(st["grids"], device="cuda").reshape(-1)
    phi = torch.as_tensor(st["phi"], device="cuda")
    off = np.concatenate([[0], np.cumsum(mdl.N)])
    layer = lambda a, k: a[int(off[k]):int(off[k + 1])]  # noqa: E731
    m = torch.arange(M, device="cuda")
    counts = []
    for k in range(mdl.n):
        w = _philox(m, k, st["seed"])
        u = [(2 * (((w[2 * q] >> 6) << 26) | (w[2 * q + 1] >> 6)) + 1).double() * 2.0**-53 for q in range(2)]
        rad, ang = torch.sqrt(-2.0 * torch.log(u[0])), 2.0 * math.pi * u[1]
        X = mdl.m[k, 0] + mdl.L[k, 0, 0] * rad * torch.cos(ang)
        Y = mdl.b[k, 0] + mdl.A[k, 0, 0] * X + mdl.T[k, 0, 0] * rad * torch.sin(ang)
        cells = []
        for x, g in ((X, layer(grids, k)), (Y, layer(grids, k + 1))):
            order = torch.argsort(g)
            s = g[order]
            cells.append(order[torch.bucketize(x, 0.5 * (s[1:] + s[:-1]))])
        counts.append(torch.bincount(cells[0] * int(mdl.N[k + 1]) + cells[1],
                                     minlength=int(mdl.N[k] * mdl.N[k + 1])).reshape(int(mdl.N[k]), -1))
    V = layer(phi, mdl.n)
    for k in range(mdl.n - 1, -1, -1):
        V = _continue(counts[k], V, layer(phi, k))
    return float((counts[0].sum(1).double() * V).sum() / M)


def _continue(counts, V, phi):
    tot = counts.sum(1)
    cont = (counts.double() @ V) / tot.clamp(min=1).double()
    return torch.where(tot > 0, torch.maximum(phi, cont), phi)


def exact(case, seed):
    kind = case["kind"]
    if kind == "price" and case["d"] == 1 and case["f64"]:
        return _exact_price_1d(case, seed)
    if kind in ("swing", "backward"):
        st = prepare(case, seed)
        N = st["N"]
        n = len(N) - 1
        off = np.concatenate([[0], np.cumsum(N)])
        coff = np.concatenate([[0], np.cumsum(N[:-1] * N[1:])])
        block = lambda k: st["counts"][int(coff[k]):int(coff[k + 1])].reshape(int(N[k]), int(N[k + 1])).long()  # noqa: E731
        v = lambda k: st["v"][int(off[k]):int(off[k + 1])]  # noqa: E731
        if kind == "backward":
            V = [v(n)]
            for k in range(n - 1, -1, -1):
                V.append(_continue(block(k), V[-1], v(k)))
            return torch.cat(V[::-1])
        qmin, qmax = case["Qmin"], case["Qmax"]
        Q = torch.arange(qmax + 2, device="cuda")
        neg = torch.tensor(-math.inf, dtype=torch.float64, device="cuda")
        ok = lambda k: (Q <= qmax) & (Q + n - k >= qmin)  # noqa: E731
        P = torch.where(ok(n)[:, None], torch.zeros(qmax + 2, int(N[n]), dtype=torch.float64, device="cuda"), neg)
        out = [P[:-1].reshape(-1)]
        for k in range(n - 1, -1, -1):
            cnt = block(k)
            tot = cnt.sum(1).clamp(min=1).double()
            C = (torch.where(torch.isfinite(P), P, torch.zeros_like(P)) @ cnt.double().T) / tot[None, :]
            C = torch.where(ok(k + 1)[:, None], C, neg)
            nxt = torch.cat([C[1:], torch.full_like(C[:1], -math.inf)]) + v(k)[None, :]
            P = torch.maximum(C, nxt)
            out.append(P[:-1].reshape(-1))
        return [torch.cat(out[::-1]), float(P[0, 0])]
    # counts and cells are whole numbers; a price on FP32 samples and sample Lloyd are defined by their
    # FP32 roundings, so they have no 64-bit value
    return None
