"""The work that is measured: block-Vecchia likelihood evaluations over the range of
problem shapes that the library's users have (single and many datasets, 2D and 3D, block
and classic Vecchia, closed-form and general smoothness, FP64 and mixed precision),
prediction with conditional simulation, the exact likelihood, and the one-time set-up.

Every case goes through the public binding (``paper_2410_04477_gb300.bv``).  Locations are
uniform points (2D) or jittered profiles (3D); the observations are a Gaussian field of the
case's own Matern covariance, summed from random spectral frequencies, plus the nugget.
Blocks are nearest-centre cells refined by Lloyd steps, in a random order, made here and
handed to the library (``set_blocks``), so that ``exact`` can evaluate the same model.
"""
import math

import numpy as np
import torch

from paper_2410_04477_gb300 import bv

Z95 = 1.959963984540054


# ---- the cases ---------------------------------------------------------------------

def listed():
    return [
        # the smallest study: one evaluation is mostly latency (n = 2,000, m = 30)
        dict(name="fp64_2k_m30", kind="fp64", n=2000, bc=200, m=30, d=2, nu=0.5, beta=0.1, nugget=1e-6, block_terms=True),
        # the ordinary 2D fit: one evaluation of a maximum-likelihood search, N about 70
        dict(name="fp64_200k_m60", kind="fp64", n=200_000, bc=20_000, m=60, d=2, nu=1.5, beta=0.05, nugget=1e-4,
             block_terms=False),
        # odd sizes, larger conditioning sets, smooth field
        dict(name="fp64_37k_m113", kind="fp64", n=36_931, bc=3_517, m=113, d=2, nu=2.5, beta=0.03, nugget=1e-3,
             block_terms=False),
        # the 3D profile data with anisotropic ranges, N about 210 (the headline shape, fewer sites)
        dict(name="fp64_3d_100k_m200", kind="fp64", n=100_000, bc=10_000, m=200, d=3, nu=0.5, beta=0.1, nugget=1e-3,
             block_terms=False),
        # classic Vecchia: blocks of one point, m = 30 (the method's own baseline)
        dict(name="fp64_classic_50k_m30", kind="fp64", n=50_000, bc=50_000, m=30, d=2, nu=1.5, beta=0.05, nugget=1e-4,
             block_terms=False),
        # a free smoothness: the covariance through K_nu
        dict(name="fp64_100k_m60_nu12", kind="fp64", n=100_000, bc=10_000, m=60, d=2, nu=1.2, beta=0.05, nugget=1e-4,
             block_terms=False),
        # many datasets in one evaluation (a simulation study), ragged sizes, own parameters
        dict(name="fp64_multi16_m60", kind="multi", ndata=16, nlo=5_000, nhi=40_000, m=60),
        # mixed precision as it is called by default (its FP64 check on)
        dict(name="mixed_150k_m100", kind="mixed", n=150_000, bc=15_000, m=100, d=2, nu=1.5, beta=0.05, nugget=5e-3,
             tol=1e-6),
        # mixed precision without the check (the search stage of a mixed fit), 3D
        dict(name="mixed32_3d_100k_m200", kind="mixed", n=100_000, bc=10_000, m=200, d=3, nu=0.5, beta=0.1, nugget=1e-3,
             tol=0.0),
        # prediction at held-out sites and 1,000 rounds of conditional simulation
        dict(name="predict_180k_m120", kind="predict", n=180_000, nstar=20_000, bc=2_000, m=120, rounds=1000, nu=1.5,
             beta=0.05, nugget=1e-2),
        # the exact likelihood of the KL study (dense)
        dict(name="exact_8k", kind="exact", n=8_000, nu=1.5, beta=0.052537, nugget=1e-4),
        # what comes before the first evaluation of new data: load, K-means blocks, neighbours
        dict(name="setup_20k_m60", kind="setup", n=20_000, bc=2_000, m=60, iters=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "fp64", "fp64", "classic", "3d", "gen", "multi", "mixed", "predict", "exact", "setup"])
    nu = rng.choice([0.5, 1.5, 2.5])
    beta = round(math.exp(rng.uniform(math.log(0.03), math.log(0.15))), 5)
    nugget = round(math.exp(rng.uniform(math.log(1e-4), math.log(1e-2))), 7)
    if kind == "exact":
        return dict(kind="exact", n=_log(rng, 500, 8000), nu=nu, beta=beta, nugget=nugget)
    if kind == "setup":
        n = _log(rng, 2000, 20_000)
        return dict(kind="setup", n=n, bc=n // rng.randint(5, 20), m=rng.randint(10, 120), iters=20)
    if kind == "multi":
        return dict(kind="multi", ndata=rng.randint(2, 16), nlo=1000, nhi=_log(rng, 2000, 40_000), m=rng.randint(20, 90))
    if kind == "predict":
        n = _log(rng, 5000, 180_000)
        ns = max(200, n // rng.randint(8, 12))
        return dict(kind="predict", n=n, nstar=ns, bc=max(4, ns // rng.randint(7, 13)), m=rng.randint(30, 150), rounds=1000,
                    nu=nu, beta=beta, nugget=max(nugget, 1e-3))
    if kind == "classic":
        n = _log(rng, 2000, 50_000)
        return dict(kind="fp64", n=n, bc=n, m=rng.randint(10, 60), d=2, nu=nu, beta=beta, nugget=nugget, block_terms=False)
    if kind == "3d":
        n = 50 * _log(rng, 100, 1500)
        return dict(kind="fp64", n=n, bc=n // rng.randint(8, 14), m=rng.randint(60, 200), d=3, nu=nu, beta=beta,
                    nugget=max(nugget, 1e-3), block_terms=False)
    n = _log(rng, 2000, 150_000)
    c = dict(n=n, bc=n // rng.randint(5, 18), m=rng.randint(10, 130), d=2, beta=beta, nugget=nugget)
    if kind == "mixed":
        return dict(c, kind="mixed", nu=nu, tol=rng.choice([0.0, 1e-6]))
    if kind == "gen":
        return dict(c, kind="fp64", nu=round(rng.uniform(0.3, 3.2), 3), block_terms=False)
    return dict(c, kind="fp64", nu=nu, block_terms=rng.random() < 0.5)


# ---- inputs ------------------------------------------------------------------------

def _dev():
    return torch.device("cuda")


def _ranges(d, beta):
    return (beta, beta, 3.0 * beta)[:d] if d == 3 else None


def _locations(rng, n, d):
    if d == 3:  # profiles: sites x 50 jittered levels, in the unit cube
        sites, levels = n // 50, 50
        xy = rng.random((sites, 2))
        z = (np.arange(levels)[None, :] + 0.5 + 0.2 * (2.0 * rng.random((sites, levels)) - 1.0)) / levels
        return np.column_stack([np.repeat(xy, levels, axis=0), z.reshape(-1)])
    return rng.random((n, d))


def _field(rng, locs, nu, beta, nugget, ranges=None, sigma2=1.0):
    """A Matern field by 400 random frequencies (its spectral law is a multivariate t with
    2 nu degrees of freedom) plus independent noise of variance `nugget`."""
    k, d = 400, locs.shape[1]
    om = rng.standard_normal((k, d)) / np.sqrt(2.0 * rng.gamma(nu, 1.0, (k, 1)))
    om = om / np.asarray(ranges if ranges is not None else [beta] * d)
    ph = torch.from_numpy(rng.uniform(0.0, 2.0 * math.pi, k)).to(_dev())
    amp = torch.from_numpy(rng.standard_normal(k)).to(_dev())
    x, w = torch.from_numpy(np.ascontiguousarray(locs)).to(_dev()), torch.from_numpy(om).to(_dev())
    f = torch.cat([torch.cos(c @ w.T + ph) @ amp for c in x.split(65536)])
    return (math.sqrt(2.0 * sigma2 / k) * f).cpu().numpy() + math.sqrt(nugget) * rng.standard_normal(len(locs))


def _cells(rng, locs, bc):
    """Cells of `bc` centres after two Lloyd steps, in a random order: (block_ptr,
    point_idx, centroids).  Integer sums: the same on every run."""
    n = len(locs)
    if bc >= n:
        idx = rng.permutation(n).astype(np.int32)
        return np.arange(n + 1, dtype=np.int64), idx, locs[idx]
    x = torch.from_numpy(locs).to(_dev())
    q = torch.round(x * 2.0 ** 40).to(torch.int64)
    cen = x[torch.from_numpy(np.sort(rng.permutation(n)[:bc])).to(_dev())]
    for step in range(3):
        c32 = cen.float()
        c2 = (c32 * c32).sum(1)
        lab = torch.cat([torch.addmm(c2, p, c32.T, alpha=-2.0).argmin(1) for p in x.float().split(max(1, (1 << 28) // bc))])
        cnt = torch.zeros(bc, dtype=torch.int64, device=_dev()).index_add_(0, lab, torch.ones_like(lab))
        s = torch.zeros(bc, x.shape[1], dtype=torch.int64, device=_dev()).index_add_(0, lab, q)
        cen = torch.where(cnt[:, None] > 0, s.double() / cnt.clamp(min=1)[:, None].double() * 2.0 ** -40, cen)
    lab, cnt, cen = lab.cpu().numpy(), cnt.cpu().numpy(), cen.cpu().numpy()
    used = np.flatnonzero(cnt)
    order = used[rng.permutation(len(used))]
    pos = np.full(bc, -1, np.int64)
    pos[order] = np.arange(len(order))
    idx = np.argsort(pos[lab], kind="stable").astype(np.int32)
    return np.concatenate([[0], np.cumsum(cnt[order])]).astype(np.int64), idx, np.ascontiguousarray(cen[order])


def _inputs(case, seed):
    rng = np.random.default_rng([seed, case["n"], case["m"]])
    locs = _locations(rng, case["n"], case["d"])
    ra = _ranges(case["d"], case["beta"])
    y = _field(rng, locs, case["nu"], case["beta"], case["nugget"], ra)
    return locs, y, _cells(rng, locs, case["bc"]), ra


def _study(case, seed):
    """The datasets of a simulation study: sizes log-uniform, own parameters."""
    rng = np.random.default_rng([seed, case["ndata"], case["m"]])
    out = []
    for _ in range(case["ndata"]):
        n = int(np.exp(rng.uniform(np.log(case["nlo"]), np.log(case["nhi"]))))
        th = dict(sigma2=float(np.exp(rng.uniform(np.log(0.5), np.log(2.0)))), beta=float(np.exp(rng.uniform(np.log(0.02), np.log(0.3)))),
                  nu=float(rng.choice([0.5, 1.5, 2.5])), nugget=float(np.exp(rng.uniform(np.log(1e-3), np.log(1e-1)))))
        locs = rng.random((n, 2))
        out.append((locs, _field(rng, locs, th["nu"], th["beta"], th["nugget"], sigma2=th["sigma2"]), th))
    return out


def _pred_inputs(case, seed):
    rng = np.random.default_rng([seed, case["n"], case["nstar"], 3])
    locs = rng.random((case["n"] + case["nstar"], 2))
    y = _field(rng, locs, case["nu"], case["beta"], case["nugget"])
    n = case["n"]
    return locs[:n], y[:n], locs[n:], y[n:]


# ---- prepare, run ------------------------------------------------------------------

def prepare(case, seed):
    ctx = bv.Context()
    kind = case["kind"]
    if kind == "setup":  # host arrays of new data
        rng = np.random.default_rng([seed, case["n"]])
        locs = rng.random((case["n"], 2))
        return dict(case=case, ctx=ctx, locs=locs, y=_field(rng, locs, 1.5, 0.05, 1e-4), seed=seed)
    if kind == "exact":
        rng = np.random.default_rng([seed, case["n"], 2])
        locs = rng.random((case["n"], 2))
        ctx.set_data(locs, _field(rng, locs, case["nu"], case["beta"], case["nugget"]))
        return dict(case=case, ctx=ctx, theta=bv.theta(1.0, case["beta"], case["nu"], case["nugget"]))
    if kind == "predict":
        locs, y, star, truth = _pred_inputs(case, seed)
        ctx.set_data(locs, y)
        ctx.set_pred_locations(star, truth)
        ctx.build_pred_blocks(case["bc"], seed=seed)
        ctx.select_pred_neighbors(case["m"])
        return dict(case=case, ctx=ctx, theta=bv.theta(1.0, case["beta"], case["nu"], case["nugget"]), seed=seed)
    if kind == "multi":
        sets = _study(case, seed)
        ctx.set_datasets([s[0] for s in sets], [s[1] for s in sets])
        ctx.build_blocks_multi([max(1, len(s[0]) // 10) for s in sets], seed=seed)
        ctx.select_neighbors(case["m"])
        th = [bv.theta(s[2]["sigma2"], s[2]["beta"], s[2]["nu"], s[2]["nugget"]) for s in sets]
        ctx.loglik_multi([bv.theta(t.sigma2, 0.9 * t.range[0], t.nu, 1.1 * t.nugget) for t in th])
        return dict(case=case, ctx=ctx, theta=th)
    locs, y, (bp, pi, cen), ra = _inputs(case, seed)
    ctx.set_data(locs, y)
    ctx.set_blocks(bp, pi, cen)
    ctx.select_neighbors(case["m"])
    prec = bv.BV_MIXED if kind == "mixed" else bv.BV_FP64
    if kind == "mixed":
        ctx.set_mixed_tolerance(case["tol"])
    # the first evaluation of the search that the timed one belongs to: it builds the plan
    ctx.loglik(bv.theta(1.1, 0.9 * case["beta"], case["nu"], 1.1 * case["nugget"],
                        ranges=None if ra is None else [0.9 * r for r in ra]), prec)
    return dict(case=case, ctx=ctx, prec=prec, theta=bv.theta(1.0, case["beta"], case["nu"], case["nugget"], ranges=ra))


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "setup":
        ctx.set_data(state["locs"], state["y"])
        bp, pi = ctx.build_blocks(case["bc"], seed=state["seed"], iters=case["iters"])
        nnp, nni = ctx.select_neighbors(case["m"])
        # one shape whatever the number of non-empty cells
        full = np.full(case["bc"] * case["m"], -1, np.int32)
        full[:len(nni)] = nni
        ptrs = np.full((2, case["bc"] + 1), -1, np.int64)
        ptrs[0, :len(bp)], ptrs[1, :len(nnp)] = bp, nnp
        return dict(block_ptr=ptrs[0], point_idx=pi, nn_ptr=ptrs[1], nn_idx=full)
    if kind == "exact":
        ell, quad, logdet = ctx.exact_loglik(state["theta"])
        return dict(terms=np.array([ell, quad, logdet]))
    if kind == "predict":
        mean, var, _ = ctx.predict(state["theta"])
        lo, up, covered = ctx.cond_sim(rounds=case["rounds"], seed=state["seed"], z_crit=Z95)
        return dict(mean=mean, var=var, lower=lo, upper=up, covered=covered)
    if kind == "multi":
        return dict(loglik=ctx.loglik_multi(state["theta"]))
    if kind == "mixed":
        return dict(loglik=ctx.loglik(state["theta"], bv.BV_MIXED))
    if case["block_terms"]:
        ell, per, _ = ctx.loglik(state["theta"], bv.BV_FP64, per_block=True)
        return dict(loglik=np.array([ell]), per_block=per)
    return dict(terms=np.array(ctx.loglik_terms(state["theta"])))


# ---- what a pass cannot do without -------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "setup":  # one distance per point and centre in each assignment; neighbour distances
        n, bc, d = case["n"], case["bc"], 2
        return dict(bytes=8.0 * n * (d + 1) + 4.0 * n + 4.0 * bc * case["m"] + 16.0 * bc,
                    flops=3.0 * d * n * bc * (case["iters"] + 2))
    if kind == "exact":
        n = case["n"]
        return dict(bytes=8.0 * n * 3 + 24, flops=n ** 3 / 3.0 + 2.0 * n * n)
    if kind == "predict":
        b = case["nstar"] / case["bc"]
        n1 = case["m"] + b
        f = sum((n1 - k) * (n1 - k + 2) for k in range(case["m"]))
        return dict(bytes=8.0 * 3 * (case["n"] + case["nstar"]) + 4.0 * case["bc"] * case["m"] + 32.0 * case["nstar"],
                    flops=case["bc"] * f + 4.0 * case["nstar"] * case["rounds"])
    if kind == "multi":
        n = case["ndata"] * (case["nhi"] - case["nlo"]) / math.log(case["nhi"] / case["nlo"]) if case["nhi"] > case["nlo"] else case["ndata"] * case["nlo"]
        bc, d = n / 10.0, 2
    else:
        n, bc, d = case["n"], case["bc"], case["d"]
    size = case["m"] + n / bc
    return dict(bytes=8.0 * n * (d + 1) + 4.0 * (n + bc * case["m"]) + 24.0, flops=bc * (size ** 3 / 3.0 + size ** 2))


# ---- the same in plain 64-bit torch ------------------------------------------------

def _corr(x, nu):
    if nu == 0.5:
        return torch.exp(-x)
    if nu == 1.5:
        return (1.0 + x) * torch.exp(-x)
    return (1.0 + x + x * x / 3.0) * torch.exp(-x)


def _cov(a, b, th):
    acc = 0.0
    for k in range(a.shape[-1]):
        t = (a[..., :, None, k] - b[..., None, :, k]) / (th["ranges"][k] if th["ranges"] is not None else th["beta"])
        acc = acc + t * t
    return th["sigma2"] * _corr(torch.sqrt(acc), th["nu"])


def _nearest(x, pos, cen, before, m):
    """The `m` points nearest to each centre among those with pos < before, by (squared
    distance, index); pos None: all points."""
    d2 = 0.0
    for k in range(x.shape[1]):
        t = x[None, :, k] - cen[:, None, k]
        d2 = d2 + t * t
    if pos is not None:
        d2 = torch.where(pos[None, :] < before[:, None], d2, torch.full_like(d2, math.inf))
    return torch.topk(d2, min(m, x.shape[0]), dim=1, largest=False, sorted=True).indices


def _exact_terms(locs, y, cells, m, th):
    """Per-block conditional log-density, quadratic form and log-determinant."""
    bp, pi, cen = cells
    x, yd = torch.from_numpy(locs).to(_dev()), torch.from_numpy(y).to(_dev())
    bpt, pit, cent = (torch.from_numpy(np.ascontiguousarray(v)).to(_dev()) for v in (bp, pi, cen))
    nb = len(bp) - 1
    size = bpt[1:] - bpt[:-1]
    pos = torch.empty(len(locs), dtype=torch.int64, device=_dev())
    pos[pit.long()] = torch.repeat_interleave(torch.arange(nb, device=_dev()), size)
    nn = torch.empty(nb, min(m, len(locs)), dtype=torch.int32, device=_dev())
    step = max(1, (1 << 28) // len(locs))
    for s in range(0, nb, step):
        e = min(nb, s + step)
        nn[s:e] = _nearest(x, pos, cent[s:e], torch.arange(s, e, device=_dev()), m).to(torch.int32)
    mi = torch.minimum(bpt[:-1], torch.tensor(m, device=_dev()))
    u, ld = (torch.empty(nb, dtype=torch.float64, device=_dev()) for _ in range(2))
    key = mi * (1 << 32) + size
    for kv in torch.unique(key).tolist():
        ks, b = kv >> 32, kv & 0xFFFFFFFF
        for blk in torch.nonzero(key == kv).reshape(-1).split(max(1, (1 << 26) // (ks + b) ** 2)):
            own = pit[(bpt[blk][:, None] + torch.arange(b, device=_dev()))].long()
            g = torch.cat([nn[blk, :ks].long(), own], 1)
            c = _cov(x[g], x[g], th) + th["nugget"] * torch.eye(ks + b, device=_dev(), dtype=torch.float64)
            chol = torch.linalg.cholesky(c)
            z = torch.linalg.solve_triangular(chol, yd[g][:, :, None], upper=False)[:, ks:, 0]
            u[blk] = (z * z).sum(1)
            ld[blk] = 2.0 * torch.log(torch.diagonal(chol, dim1=1, dim2=2)[:, ks:]).sum(1)
    return -0.5 * (u + ld + size.double() * math.log(2.0 * math.pi)), u, ld


def exact(case, seed):
    kind = case["kind"]
    if kind in ("setup", "multi") or case["nu"] not in (0.5, 1.5, 2.5):
        return None  # whole numbers; blocks that only the library makes; K_nu that torch has not
    th = dict(sigma2=1.0, beta=case["beta"], nu=case["nu"], nugget=case["nugget"], ranges=None)
    if kind == "exact":
        rng = np.random.default_rng([seed, case["n"], 2])
        locs = rng.random((case["n"], 2))
        y = _field(rng, locs, case["nu"], case["beta"], case["nugget"])
        x = torch.from_numpy(locs).to(_dev())
        chol = torch.linalg.cholesky(_cov(x, x, th) + th["nugget"] * torch.eye(len(x), device=_dev(), dtype=torch.float64))
        z = torch.linalg.solve_triangular(chol, torch.from_numpy(y).to(_dev())[:, None], upper=False)[:, 0]
        quad, logdet = float((z * z).sum()), float(2.0 * torch.log(torch.diagonal(chol)).sum())
        return dict(terms=np.array([-0.5 * (quad + logdet + len(y) * math.log(2.0 * math.pi)), quad, logdet]))
    if kind == "predict":
        return None  # the prediction blocks come from the library's K-means
    locs, y, cells, ra = _inputs(case, seed)
    per, u, ld = _exact_terms(locs, y, cells, case["m"], dict(th, ranges=ra))
    if kind == "mixed":
        return dict(loglik=float(per.sum()))
    if case["block_terms"]:
        return dict(loglik=np.array([float(per.sum())]), per_block=per.cpu().numpy())
    return dict(terms=np.array([float(per.sum()), float(u.sum()), float(ld.sum())]))
