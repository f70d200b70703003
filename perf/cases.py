"""What is measured of this library: calls that its users make, over the range of sizes they are made at.

A case is one call (or the few calls that belong together) of the public binding on resident
device arrays, as a program that evaluates log-CDFs makes it:

  kind "unordered"  vecchia_log_cdf_unordered: order, neighbours and log-CDF of raw sites
  kind "log_cdf"    vecchia_log_cdf on ordered sites with their neighbour rows (an optimiser's step)
  kind "terms"      vecchia_log_cdf_terms: the same with every term and per-shift partial
  kind "plan"       Plan.run: a resident batch of problems replayed with new parameters
  kind "order"      vecchia_order, vecchia_apply_order, vecchia_neighbors: the preparation of a large problem
  kind "grouped"    vecchia_group_conditioning and vecchia_grouped_log_cdf: joint groups of sites
  kind "censored"   vecchia_censored_log_cdf: one replicate of the application's likelihood
  kind "full"       vecchia_full_genz: the full D-dimensional estimate

`exact` evaluates the same quantities in 64 bits with torch and numpy alone.
"""
import math

import numpy as np
import torch

import paper_2007_15195_gb300 as V

EXPONENTIAL, MATERN, ANISO = 0, 1, 2
Z90 = 1.2815515655446004  # the standard normal's 0.9 quantile


def listed():
    return [
        # the smallest problem of the simulation study (10 x 10 grid): launches and latency
        dict(name="grid10", kind="unordered", sites="grid", D=100, order="xy", m=10, cov=EXPONENTIAL, range=0.2, nu=0.5,
             u="zero", N=2000, S=10, fp64=False),
        # the benchmark's evaluation: 50 x 50 grid, m = 20
        dict(name="grid50", kind="unordered", sites="grid", D=2500, order="xy", m=20, cov=MATERN, range=0.1, nu=1.5,
             u="normal", N=4096, S=16, fp64=False),
        # the same problem where a caller wants double precision throughout
        dict(name="grid50_fp64", kind="log_cdf", sites="grid", D=2500, order="xy", m=20, cov=MATERN, range=0.1, nu=1.5,
             u="normal", N=4096, S=16, fp64=True),
        # a ragged small problem in double precision with every term (diagnostics, convergence studies)
        dict(name="terms_fp64", kind="terms", sites="uniform", D=333, order="maxmin", m=13, cov=EXPONENTIAL, range=0.3, nu=0.5,
             u="normal", N=1021, S=6, fp64=True),
        # the longest conditioning sets of the study (m = 50)
        dict(name="m50", kind="log_cdf", sites="grid", D=1600, order="xy", m=50, cov=MATERN, range=0.1, nu=1.5,
             u="normal", N=2048, S=8, fp64=False),
        # a batch of problems of 50 to 2,000 sites along an optimiser's trajectory
        dict(name="plan", kind="plan", sites="uniform", D=2000, order="xy", m=20, cov=EXPONENTIAL, range=0.2, nu=0.5,
             u="z90", N=2048, S=8, fp64=False, problems=192),
        # a request with sites in no order: exact maxmin ordering, m = 30
        dict(name="request", kind="unordered", sites="uniform", D=20011, order="maxmin", m=30, cov=MATERN, range=0.1, nu=0.5,
             u="z90", N=2048, S=8, fp64=False),
        # what precedes a large problem's evaluations: ordering, gather, neighbour rows
        dict(name="order100k", kind="order", sites="uniform", D=100000, order="maxmin", m=30),
        # joint groups of five on a 100 x 100 grid
        dict(name="grouped", kind="grouped", sites="grid", D=10000, order="xy", m=5, p=5, cov=EXPONENTIAL, range=0.1, nu=0.5,
             u="normal", N=2048, S=8, fp64=False),
        # one replicate of the censored likelihood: 528 stations, a tenth observed
        dict(name="censored", kind="censored", sites="uniform", D=528, order="maxmin", m=20, cov=ANISO, range=0.2, nu=0.5,
             u="z90", N=2048, S=8, fp64=False, nodes=16),
        # the comparison estimate over all 2,500 variables
        dict(name="full", kind="full", sites="grid", D=2500, order="xy", m=0, cov=MATERN, range=0.1, nu=1.5,
             u="normal", N=4096, S=16, fp64=False),
        # the comparison estimate in double precision, odd sizes
        dict(name="full_fp64", kind="full", sites="uniform", D=1021, order="xy", m=0, cov=EXPONENTIAL, range=0.2, nu=0.5,
             u="normal", N=2000, S=12, fp64=True),
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["unordered", "unordered", "log_cdf", "log_cdf", "terms", "plan", "order", "grouped", "censored", "full"])
    c = dict(kind=kind, sites=rng.choice(["grid", "uniform"]), D=0, order=rng.choice(["xy", "maxmin"]),
             m=rng.randint(2, 34), cov=rng.choice([EXPONENTIAL, MATERN]), range=round(rng.uniform(0.05, 0.4), 3), nu=0.5,
             u=rng.choice(["normal", "z90", "zero"]), N=log_uniform(500, 4096), S=rng.randint(4, 16), fp64=rng.random() < 0.35)
    if c["cov"] == MATERN:
        c["nu"] = rng.choice([0.5, 1.5])
    if kind == "order":
        return dict(kind=kind, sites="uniform", D=log_uniform(300, 100000), order=c["order"], m=c["m"])
    if kind == "full":
        c.update(D=log_uniform(40, 1200 if c["fp64"] else 2500), m=0, order="xy")
        c["N"] = min(c["N"], 2048 if c["fp64"] else 4096)
    elif kind == "plan":
        c.update(problems=rng.randint(3, 64), D=2000, sites="uniform", m=max(5, min(c["m"], 30)), fp64=False)
    elif kind == "grouped":
        p = rng.randint(2, 6)
        c.update(p=p, m=rng.randint(2, 8), D=log_uniform(200, 10000), fp64=False)
    elif kind == "censored":
        c.update(D=rng.randint(100, 600), sites="uniform", cov=ANISO, u="z90", m=max(8, min(c["m"], 24)), nodes=rng.choice([0, 8, 16]), fp64=False)
    else:
        if kind == "terms":  # the partials are asked for where double precision is wanted
            c["fp64"] = True
        c["D"] = log_uniform(60, 2500 if c["fp64"] else 20000)
        if kind == "log_cdf" and not c["fp64"] and rng.random() < 0.3:
            c["m"] = rng.randint(35, 60)
        if c["fp64"]:
            c["N"] = min(c["N"], 2048)
    if c["sites"] == "grid":
        c["D"] = max(2, round(math.sqrt(c["D"]))) ** 2
    return c


# ------------------------------ inputs ---------------------------------------

def _gen(seed, stream):
    return np.random.Generator(np.random.Philox(np.random.SeedSequence([int(seed), int(stream)])))


def _grid(n):
    t = np.arange(n, dtype=np.float64) / (n - 1)
    xx, yy = np.meshgrid(t, t, indexing="ij")
    return np.stack([xx.ravel(), yy.ravel()], axis=1)


def _raw(case, seed):
    """Raw sites and thresholds on the host."""
    D = case["D"]
    if case["sites"] == "grid":
        s = _grid(int(round(math.sqrt(D))))
    else:
        s = _gen(seed, 0).random((D, 2))
    kind = case.get("u", "normal")
    if kind == "normal":
        u = _gen(seed, 1).normal(0.5, 0.25, size=D)
    elif kind == "z90":
        u = np.full(D, Z90)
    else:
        u = np.zeros(D)
    return s, u


def _cov(case):
    if case["cov"] == ANISO:
        return (ANISO, 1.0, case["range"], 0.5, 0.0, 0.5, 1.5)
    return (case["cov"], 1.0, case["range"], case["nu"], 0.0)


def _qmc_seed(seed):
    return int(_gen(seed, 2).integers(1, 2 ** 62))


def _plan_parts(case, seed):
    g = _gen(seed, 3)
    n = case["problems"]
    Ds = np.rint(np.exp(g.uniform(math.log(50.0), math.log(2000.0), size=n))).astype(int)
    covs = [(EXPONENTIAL, 1.0, float(r), 0.5, 0.0) for r in g.uniform(0.05, 0.5, size=n)]
    seeds = g.integers(1, 2 ** 62, size=n).astype(np.uint64)
    raw = [g.random((int(d), 2)) for d in Ds]
    return raw, covs, seeds


def _censored_parts(case, seed):
    """Censored sites, their thresholds, the observed sites and values (a tenth of the sites)."""
    s, _ = _raw(case, seed)
    g = _gen(seed, 4)
    D = case["D"]
    k = max(1, int(round(0.1 * D)))
    obs = np.sort(g.choice(D, size=k, replace=False))
    cen = np.setdiff1d(np.arange(D), obs)
    return s[cen].copy(), np.full(cen.size, Z90), s[obs].copy(), Z90 + 0.5 * g.exponential(size=k)


_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = V.Context(0)
    return _ctx


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _prepared(ctx, s, u, order, m):
    """Ordered device arrays and neighbour rows, as a program that evaluates repeatedly keeps them."""
    s, u = _dev(s), _dev(u)
    perm = V.vecchia_order(ctx, s, order)
    s, u = V.vecchia_apply_order(ctx, perm, s, u)
    return s, u, V.vecchia_neighbors(ctx, s, m)


def prepare(case, seed):
    ctx = _context()
    kind = case["kind"]
    st = dict(case=case, ctx=ctx, seed=_qmc_seed(seed), precision=V.FP64 if case.get("fp64") else V.MIXED)
    if kind == "plan":
        raw, covs, seeds = _plan_parts(case, seed)
        problems = []
        for s, cov, sd in zip(raw, covs, seeds):
            s, u, nbr = _prepared(ctx, s, np.full(len(s), Z90), case["order"], case["m"])
            problems.append(dict(sites=s, u=u, nbr=nbr, m=case["m"], cov=cov, N=case["N"], S=case["S"], seed=int(sd)))
        st.update(plan=V.Plan(ctx, problems, st["precision"]), covs=covs, seeds=seeds)
        return st
    if kind == "censored":
        sc, xc, si, xi = _censored_parts(case, seed)
        sc, xc, nbr = _prepared(ctx, sc, xc, case["order"], case["m"])
        st.update(sites=sc, x=xc, nbr=nbr, sites_i=_dev(si), x_i=_dev(xi), cov=_cov(case))
        return st
    s, u = _raw(case, seed)
    if kind == "order":
        st.update(sites=_dev(s), u=_dev(u))
        return st
    st["cov"] = _cov(case)
    if kind in ("log_cdf", "terms"):
        st["sites"], st["u"], st["nbr"] = _prepared(ctx, s, u, case["order"], case["m"])
    elif kind in ("grouped", "full"):
        s, u = _dev(s), _dev(u)
        perm = V.vecchia_order(ctx, s, case["order"])
        st["sites"], st["u"] = V.vecchia_apply_order(ctx, perm, s, u)
    else:
        st["sites"], st["u"] = _dev(s), _dev(u)
    return st


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "order":
        perm = V.vecchia_order(ctx, state["sites"], c["order"])
        s, u = V.vecchia_apply_order(ctx, perm, state["sites"], state["u"])
        return perm, s, u, V.vecchia_neighbors(ctx, s, c["m"])
    if kind == "plan":
        return state["plan"].run(seeds=state["seeds"], covs=state["covs"])
    args = dict(N=c["N"], S=c["S"], seed=state["seed"], precision=state["precision"])
    if kind == "unordered":
        perm = torch.empty(c["D"], dtype=torch.int32, device="cuda")
        lp, se = V.vecchia_log_cdf_unordered(ctx, state["sites"], state["u"], c["m"], state["cov"], order=c["order"],
                                             perm_out=perm, **args)
        return lp, se, perm
    if kind == "log_cdf":
        return V.vecchia_log_cdf(ctx, state["sites"], state["nbr"], c["m"], state["cov"], state["u"], **args)
    if kind == "terms":
        return V.vecchia_log_cdf_terms(ctx, state["sites"], state["nbr"], c["m"], state["cov"], state["u"], **args)
    if kind == "grouped":
        cond, count = V.vecchia_group_conditioning(ctx, state["sites"], c["p"], c["m"])
        lp, se = V.vecchia_grouped_log_cdf(ctx, state["sites"], c["p"], cond, state["cov"], state["u"], **args)
        return lp, se, cond, count
    if kind == "censored":
        return V.vecchia_censored_log_cdf(ctx, state["sites"], state["nbr"], c["m"], state["sites_i"], state["cov"],
                                          state["x"], state["x_i"], n_nodes=c["nodes"], **args)
    return V.vecchia_full_genz(ctx, state["sites"], state["cov"], state["u"], **args)


# ------------------------------ work -----------------------------------------

def _steps(case):
    """Lattice steps (one coordinate of one point of one term) and conditional-mean products of a pass."""
    NS = float(case["N"] * case["S"])

    def classic(D, m):
        q = np.minimum(np.arange(D, dtype=np.float64), m)
        return NS * q.sum(), NS * (q * (q + 1) / 2).sum()

    kind, D, m = case["kind"], case["D"], case["m"]
    if kind == "full":
        return NS * (D - 1), NS * D * (D - 1) / 2.0
    if kind == "plan":
        # D log-uniform in [50, 2000]: the mean size
        mean = (2000.0 - 50.0) / math.log(2000.0 / 50.0)
        a, b = classic(int(mean), m)
        return a * case["problems"], b * case["problems"]
    if kind == "grouped":
        # a group's conditioning set: the union of its members' neighbours, about half of p m apart from the members
        p = case["p"]
        q = p - 1 + max(m, p * m // 2)
        return NS * (D // p) * q, NS * (D // p) * q * (q + 1) / 2.0
    if kind == "censored":
        a, b = classic(int(0.9 * D), m)
        return a * max(1, case["nodes"]), b * max(1, case["nodes"])
    return classic(D, m)


def work(case):
    D, m = case["D"], case["m"]
    if case["kind"] == "order":  # sites and thresholds in and out, the permutation and the rows out
        return {"bytes": 48.0 * D + 4.0 * D + 4.0 * D * m, "flops": 10.0 * D * m}
    n = case.get("problems", 1) * (D if case["kind"] != "plan" else 530)
    by = 24.0 * n + 4.0 * n * m * (0 if case["kind"] in ("full", "unordered", "grouped") else 1)
    if case["kind"] == "terms":
        by += 16.0 * n * case["S"] + 8.0 * n
    if case["kind"] == "unordered":
        by += 4.0 * n
    steps, fma = _steps(case)
    fl = 31.0 * steps + 2.0 * fma  # quantile, distribution function and lattice coordinate a step, one product a coefficient
    if case["kind"] == "full":
        fl += D ** 3 / 3.0
    return {"bytes": by, "flops": fl}


# ------------------------------ 64-bit values ---------------------------------

def _philox(c0, c1, c2, c3, seed):
    """Words 0 and 1 of Philox4x32-10 (Salmon et al., SC'11) for arrays of counters."""
    M = 0xFFFFFFFF
    c = [np.broadcast_to(np.asarray(v, dtype=np.uint64), np.broadcast(c0, c1).shape).copy() for v in (c0, c1, c2, c3)]
    k0, k1 = seed & M, (seed >> 32) & M
    for r in range(10):
        p0 = c[0] * np.uint64(0xD2511F53)
        p1 = c[2] * np.uint64(0xCD9E8D57)
        lo, hi = np.uint64(M), np.uint64(32)
        c = [(p1 >> hi) ^ c[1] ^ np.uint64(k0), p1 & lo, (p0 >> hi) ^ c[3] ^ np.uint64(k1), p0 & lo]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c[0], c[1]


def _shifts(seed, S, dim):
    s, j = np.meshgrid(np.arange(S), np.arange(dim), indexing="ij")
    a, b = _philox(s, j, 0x51A7, 0, int(seed))
    return (((a >> np.uint64(5)) << np.uint64(26)) | (b >> np.uint64(6))).astype(np.float64) * 2.0 ** -53


def _lattice(N, dim):
    """Powers of the Korobov multiplier that minimises the weighted P2 criterion (weights 1/j^2, 30 dimensions)."""
    cand = np.array([a for a in range(2, N // 2 + 1) if math.gcd(a, N) == 1], dtype=np.int64)
    best = 1
    if N >= 4 and cand.size:
        x = torch.arange(N, dtype=torch.float64, device="cuda") / N
        b2 = (x * x - x) + 1.0 / 6.0
        k = torch.arange(N, device="cuda")
        crit = []
        for ch in torch.from_numpy(cand).cuda().split(max(1, (1 << 24) // N)):
            g = torch.ones_like(ch) % N
            prod = torch.ones(len(ch), N, dtype=torch.float64, device="cuda")
            for j in range(30):
                prod *= 1.0 + (2.0 * math.pi ** 2 / (j + 1) ** 2) * b2[(k[None, :] * g[:, None]) % N]
                g = (g * ch) % N
            crit.append(prod.mean(1))
        crit = torch.cat(crit)
        lo = crit.min()
        best = int(cand[int(torch.nonzero(crit <= lo + 1e-12 * (1.0 + abs(lo)))[0])])
    g, out = 1 % N, []
    for _ in range(dim):
        out.append(g)
        g = g * best % N
    return out


def _covariance(case, h_of, r2=1.0):
    h = h_of / case["range"]
    if case["cov"] == MATERN and case["nu"] == 1.5:
        a = math.sqrt(3.0) * h
        return r2 * (1.0 + a) * torch.exp(-a)
    return r2 * torch.exp(-h)


def _distance(case, a, b):
    dx, dy = a[..., 0] - b[..., 0], a[..., 1] - b[..., 1]
    if case["cov"] == ANISO:
        c, s = math.cos(0.5), math.sin(0.5)
        return torch.sqrt((dx * c - dy * s) ** 2 + (1.5 * (dx * s + dy * c)) ** 2)
    return torch.sqrt(dx * dx + dy * dy)


def _phi_pair(z):
    t = 0.5 * torch.special.erfc(z.abs() * math.sqrt(0.5))
    return torch.where(z < 0, t, 1.0 - t), torch.where(z < 0, 1.0 - t, t)


def _quantile(p, q):
    s = torch.minimum(p, q).clamp_min(2.0 ** -1000)
    y = torch.special.ndtri(s)
    return torch.where(p <= q, y, -y)


def _points(g, delta, t, N):
    """Tent-mapped lattice coordinate t of all shifts: (w, 1 - w), each S x N."""
    k = torch.arange(N, device="cuda")
    x = ((k * g[t]) % N).double() / N
    x = x[None, :] + delta[:, t, None]
    x = torch.where(x >= 1.0, x - 1.0, x)
    a = (2.0 * x - 1.0).abs()
    return (1.0 - a).reshape(-1), a.reshape(-1)


def _genz(sigma, u, c, g, delta, N, S):
    """Per-shift means (num, den), n x S, of n terms of d variables whose first c condition."""
    n, d = u.shape
    num = torch.empty(n, S, dtype=torch.float64, device="cuda")
    den = torch.ones_like(num)
    L = torch.linalg.cholesky(sigma)
    pts = [_points(g, delta, t, N) for t in range(d - 1)]
    step = max(1, 6_000_000 // (N * S))
    for i in range(0, n, step):
        Lc, uc = L[i:i + step], u[i:i + step]
        b = uc.shape[0]
        e, ec = _phi_pair((uc[:, 0] / Lc[:, 0, 0])[:, None].expand(b, N * S))
        f = torch.ones(b, N * S, dtype=torch.float64, device="cuda")
        ys, fc = [], None
        for t in range(d - 1):
            f = f * e
            if t + 1 == c:
                fc = f
            w, a = pts[t]
            ys.append(_quantile(w * e, a + w * ec))
            acc = uc[:, t + 1, None].expand(b, N * S).clone()
            for j, y in enumerate(ys):
                acc.addcmul_(y, Lc[:, t + 1, j, None], value=-1.0)
            e, ec = _phi_pair(acc / Lc[:, t + 1, t + 1, None])
        num[i:i + step] = (f * e).reshape(b, S, N).mean(2)
        if c > 0:
            den[i:i + step] = (f * e if c == d else fc).reshape(b, S, N).mean(2)
    return num, den


def _reduce(num, den):
    S = num.shape[1]
    a, b = num.mean(1, keepdim=True), den.mean(1, keepdim=True)
    terms = (torch.log(a) - torch.log(b))[:, 0]
    ell = (num / a - den / b).sum(0)
    return terms.sum().item(), math.sqrt((ell * ell).sum().item() / (S * (S - 1))), terms


def _vecchia(case, blocks, sigma_of, u, seed):
    """blocks: list of (indices, c) with the indices of a term in block order."""
    N, S = case["N"], case["S"]
    dim = max(1, max(len(b) for b, _ in blocks) - 1)
    g = _lattice(N, dim)
    delta = torch.from_numpy(_shifts(seed, S, dim)).cuda()
    num = torch.empty(len(blocks), S, dtype=torch.float64, device="cuda")
    den = torch.empty_like(num)
    same = {}
    for i, (b, c) in enumerate(blocks):
        same.setdefault((len(b), c), []).append(i)
    for (d, c), at in same.items():
        idx = torch.tensor(np.array([blocks[i][0] for i in at]), device="cuda")
        num[at], den[at] = _genz(sigma_of(idx), u[idx], c, g, delta, N, S)
    return num, den


def _quantised(s):
    lo = s.min(0)
    ext = float((s.max(0) - lo).max())
    return np.floor((s - lo) * (2.0 ** 30 / ext)).astype(np.int64) if ext > 0 else np.zeros(s.shape, np.int64)


def _order(s, kind):
    D = len(s)
    if kind == "xy":
        return np.lexsort((np.arange(D), s[:, 1], s[:, 0]))
    q = torch.from_numpy(_quantised(s)).cuda()
    mid = ((2 * q - q.max(0).values) ** 2).sum(1)
    first = torch.nonzero(mid == mid.min())[0, 0]  # nearest to the box's centre
    mind = torch.full((D,), 2 ** 62, dtype=torch.int64, device="cuda")
    perm = torch.empty(D, dtype=torch.int64, device="cuda")
    pick = first.reshape(1)
    at = torch.arange(D, device="cuda")
    for i in range(D):
        perm[i] = pick[0]
        mind = torch.minimum(mind, ((q - q[pick]) ** 2).sum(1))
        mind[pick] = -1
        top = mind.max()
        pick = torch.where(mind == top, at, D).min().reshape(1)  # ties to the smaller index
    return perm.cpu().numpy()


def _rows(s, m, limit=None):
    """The min(m, i) nearest earlier sites of every ordered site (limit[i]: only sites before it), ascending."""
    D = len(s)
    q = torch.from_numpy(_quantised(s)).cuda()
    limit = np.arange(D) if limit is None else limit
    lim = torch.from_numpy(limit).cuda()
    j = torch.arange(D, device="cuda")
    rows = []
    for i in range(0, D, 2048):
        d2 = ((q[i:i + 2048, None, :] - q[None, :, :]) ** 2).sum(2)
        d2 = torch.where(j[None, :] < lim[i:i + 2048, None], d2, 2 ** 62)
        rows.append(torch.sort(d2, dim=1, stable=True).indices[:, :m].cpu().numpy())
    rows = np.concatenate(rows)
    return [np.sort(r[:min(m, int(n))]) for r, n in zip(rows, limit)]


def _nodes(n):
    """Quadrature over the mixing law (beta = 0.5, gamma = 1): (r, weight) pairs."""
    if n == 0:
        return [(1.0, 1.0)]
    t, w = np.polynomial.legendre.leggauss(n)
    t = 0.5 * (t + 1.0)
    w = 2.0 * w * (1.0 - t) ** 3
    r = (1.0 - 0.5 * np.log((1.0 - t) ** 4)) ** 2
    return list(zip(r.tolist(), w.tolist()))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("order", "plan"):
        return None  # whole numbers; and a batch of a hundred problems and more takes too long here
    if _steps(case)[0] > 4.5e9:
        return None
    qs = _qmc_seed(seed)
    if kind == "censored":
        sc, xc, si, xi = _censored_parts(case, seed)
        perm = _order(sc, case["order"])
        sc, xc = sc[perm], torch.from_numpy(xc[perm]).cuda()
        rows = _rows(sc, case["m"])
        a, b, xi = torch.from_numpy(sc).cuda(), torch.from_numpy(si).cuda(), torch.from_numpy(xi).cuda()
        Lo = torch.linalg.cholesky(_covariance(case, _distance(case, b[:, None], b[None, :])))
        Vc = torch.linalg.solve_triangular(Lo, _covariance(case, _distance(case, b[:, None], a[None, :])), upper=False)
        wv = torch.linalg.solve_triangular(Lo, xi[:, None], upper=False)
        cond = _covariance(case, _distance(case, a[:, None], a[None, :])) - Vc.T @ Vc
        u = xc - (Vc.T @ wv)[:, 0]
        quad, k = float((wv * wv).sum()), len(xi)
        logdet = 2.0 * float(torch.log(torch.diagonal(Lo)).sum())
        blocks = [(list(r) + [i], len(r)) for i, r in enumerate(rows)]
        terms, ses = [], []
        for r, w in _nodes(case["nodes"]):
            num, den = _vecchia(case, blocks, lambda idx: r * r * cond[idx[:, :, None], idx[:, None, :]], u, qs)
            lp, se, _ = _reduce(num, den)
            terms.append(math.log(w) + lp - 0.5 * k * math.log(2 * math.pi) - 0.5 * logdet - quad / (2 * r * r) - k * math.log(r))
        top = max(terms)
        return top + math.log(sum(math.exp(t - top) for t in terms)), None
    s, u = _raw(case, seed)
    perm = _order(s, case["order"])
    s, u = s[perm], torch.from_numpy(u[perm]).cuda()
    sd = torch.from_numpy(s).cuda()

    def sigma_of(idx):
        p = sd[idx]
        return _covariance(case, _distance(case, p[:, :, None], p[:, None, :]))

    if kind == "full":
        N, S, D = case["N"], case["S"], case["D"]
        L = torch.linalg.cholesky(sigma_of(torch.arange(D, device="cuda")[None])[0])
        g = _lattice(N, max(1, D - 1))
        delta = torch.from_numpy(_shifts(qs, S, max(1, D - 1))).cuda()
        y = torch.empty(max(1, D - 1), N * S, dtype=torch.float64, device="cuda")
        e, ec = _phi_pair((u[0] / L[0, 0]).expand(N * S))
        f = e
        for t in range(D - 1):
            w, a = _points(g, delta, t, N)
            y[t] = _quantile(w * e, a + w * ec)
            e, ec = _phi_pair((u[t + 1] - L[t + 1, :t + 1] @ y[:t + 1]) / L[t + 1, t + 1])
            f = f * e
        mean = f.reshape(S, N).mean(1)
        p = mean.mean()
        return math.log(p.item()), math.sqrt((((mean - p) ** 2).sum() / (S * (S - 1))).item()) / p.item()
    if kind == "grouped":
        p = case["p"]
        lim = (np.arange(len(s)) // p) * p
        rows = _rows(s, case["m"], lim)
        blocks = []
        for i0 in range(0, len(s), p):
            i1 = min(i0 + p, len(s))
            c = sorted(set(int(v) for i in range(i0, i1) for v in rows[i]))
            blocks.append((c + list(range(i0, i1)), len(c)))
    else:
        blocks = [(list(r) + [i], len(r)) for i, r in enumerate(_rows(s, case["m"]))]
    num, den = _vecchia(case, blocks, sigma_of, u, qs)
    lp, se, terms = _reduce(num, den)
    if kind == "terms":
        return lp, se, terms, num, den
    return (lp, se, None) if kind == "unordered" else (lp, se, None, None) if kind == "grouped" else (lp, se)
