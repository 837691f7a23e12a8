"""The work that users of this framework have it do, as cases that can be timed.

Every case is one pass through the public entry points of
``paper_1508_02766_gb300``: density estimates (bin, kernel grid, FFT
evaluation) in one to three dimensions and both precisions, densities for many
bandwidths, bandwidth selection by LSCV, ragged batches of datasets, and the
learned selection with its network's training gradient.  Samples are
correlated Gaussian mixtures drawn on the GPU from the seed; a grid covers the
data plus four kernel widths, as in the framework's own workloads.
"""
import itertools
import math
import random

import numpy as np
import torch

from paper_1508_02766_gb300 import kde, learned

MEANS2 = [(0.0, 0.0), (2.0, 1.0), (-1.0, 2.0)]
RHOS2 = [0.8, -0.5, 0.0]


def listed():
    return [
        # the smallest call: one interactive plot of ten thousand samples, double precision
        dict(name="eval2d_128_f64", kind="eval", d=2, M0=128, M1=128, n=10_000, precision="f64",
             samples="f64", scale=1.0, major=0.16, minor=0.02),
        # the ordinary large plane: a million samples, a strongly correlated bandwidth
        dict(name="eval2d_1024_f32", kind="eval", d=2, M0=1024, M1=1024, n=1_000_000,
             precision="f32", samples="f32", scale=3.0, major=0.2, minor=0.005),
        # the largest estimate: ten million samples on a volume
        dict(name="eval3d_256_f32", kind="eval", d=3, M0=256, M1=256, M2=256, n=10_000_000,
             precision="f32", samples="f32"),
        # one axis, odd length, double precision (an income or a waiting-time density)
        dict(name="eval1d_2001_f64", kind="eval", d=1, M0=2001, n=200_000, precision="f64",
             samples="f64"),
        # a ragged volume of odd sides, samples kept in double
        dict(name="eval3d_ragged_f32", kind="eval", d=3, M0=75, M1=91, M2=110, n=1_000_000,
             precision="f32", samples="f64"),
        # a map: odd sides whose padded lines exceed 2048 points, samples kept in double
        dict(name="eval2d_map_f32", kind="eval", d=2, M0=2017, M1=3001, n=4_000_000,
             precision="f32", samples="f64", scale=3.0, major=0.02, minor=0.004),
        # one binned grid shown under many bandwidths
        dict(name="densities2d_512", kind="densities", M0=512, M1=512, n=2_000_000, nH=1024),
        # bandwidth selection on one dataset: binning, autocorrelation, every candidate's LSCV
        dict(name="lscv2d_512", kind="lscv", M0=512, M1=512, n=2_000_000, nH=1024),
        # many independent datasets with grids of their own sizes, in one call
        dict(name="ragged64_f32", kind="ragged", count=64, n_lo=1_000, n_hi=1_000_000,
             M_lo=64, M_hi=1024, shapes=5),
        # labelling: the plain search over the whole candidate grid for a batch of datasets
        dict(name="label256", kind="label", count=256, n=10_000),
        # the learned selection of a batch of datasets: features, network, scored neighbourhoods
        dict(name="select256", kind="select", count=256, n=10_000),
        # one training step's forward and backward pass of the proposal network
        dict(name="mlp_grad256", kind="mlp", count=256),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval"] * 7 + ["densities", "lscv", "ragged", "label", "select", "mlp"])
    if kind == "eval":
        d = rng.choice([1, 2, 2, 2, 3, 3])
        p = "f32" if d == 3 else rng.choice(["f32", "f32", "f64"])
        c = dict(kind=kind, d=d, precision=p, samples=rng.choice([p, p, "f32" if p == "f64" else "f64"]))
        top = {1: 3500, 2: 1400 if p == "f32" else 700, 3: 256}[d]
        for k in range(d):
            c["M%d" % k] = _between(rng, {1: 200, 2: 64, 3: 32}[d], top)
        c["n"] = _between(rng, 1_000, 5_000_000 if p == "f32" else 500_000)
        if d == 2:
            c.update(scale=round(rng.uniform(1.0, 3.0), 3), major=round(rng.uniform(0.05, 0.25), 4),
                     minor=round(rng.uniform(0.004, 0.05), 4))
        return c
    if kind == "densities":
        return dict(kind=kind, M0=_between(rng, 64, 512), M1=_between(rng, 64, 512),
                    n=_between(rng, 10_000, 2_000_000), nH=_between(rng, 16, 512))
    if kind == "lscv":
        return dict(kind=kind, M0=_between(rng, 64, 512), M1=_between(rng, 64, 512),
                    n=_between(rng, 10_000, 2_000_000), nH=_between(rng, 32, 1024))
    if kind == "ragged":
        return dict(kind=kind, count=rng.randint(4, 64), n_lo=1_000, n_hi=_between(rng, 10_000, 1_000_000),
                    M_lo=64, M_hi=rng.choice([256, 512, 1024]), shapes=rng.randint(0, 10**6))
    if kind == "mlp":
        return dict(kind=kind, count=_between(rng, 16, 256))
    return dict(kind=kind, count=_between(rng, 8, 256), n=_between(rng, 1_000, 10_000))


# ---------------------------------------------------------------------------
# Inputs, the same for run() and exact().
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _dtype(name):
    return torch.float32 if name == "f32" else torch.float64


def _mixture(g, n, means, factors, dtype):
    """n samples of the equal-weight mixture of means[k] + factors[k] z."""
    means = torch.tensor(np.asarray(means), dtype=torch.float64, device="cuda")
    factors = torch.tensor(np.asarray(factors), dtype=torch.float64, device="cuda")
    k, d = means.shape
    c = torch.randint(k, (n,), generator=g, device="cuda")
    z = torch.randn(n, d, generator=g, device="cuda", dtype=torch.float64)
    x = means[c]
    for a in range(d):
        for b in range(a + 1):
            x[:, a] += factors[c, a, b] * z[:, b]
    return x.to(dtype).contiguous()


def _plane(g, n, scale, dtype):
    f = [np.linalg.cholesky(np.array([[1.0, r], [r, 1.0]])) * scale for r in RHOS2]
    return _mixture(g, n, np.array(MEANS2) * scale, f, dtype)


def _rotated(major, minor, angle=math.pi / 4):
    c, s = math.cos(angle), math.sin(angle)
    Q = np.array([[c, -s], [s, c]])
    return Q @ np.diag([major, minor]) @ Q.T


def _normal_reference(X):
    n, d = X.shape
    S = np.atleast_2d(torch.cov(X.double().T).cpu().numpy())
    return (4.0 / (d + 2)) ** (2.0 / (d + 4)) * n ** (-2.0 / (d + 4)) * S


def _range(X, lam):
    pad = 4.0 * math.sqrt(lam)
    lo, hi = (v.double().cpu().numpy() for v in (X.amin(0), X.amax(0)))
    return lo - pad, hi + pad


def _grid(case):
    return tuple(case["M%d" % k] for k in range(case.get("d", 2)))


def _eval_inputs(case, seed):
    g, d, n = _gen(seed), case["d"], case["n"]
    dt = _dtype(case["samples"])
    if d == 2:
        X = _plane(g, n, case["scale"], dt)
        H = _rotated(case["major"], case["minor"])
    else:
        r = np.random.default_rng(seed)
        means = r.uniform(-3.0, 3.0, size=(4, d))
        covs = []
        for _ in range(4):
            Q, _R = np.linalg.qr(r.standard_normal((d, d)))
            covs.append((Q * r.uniform(1.0, 50.0) ** (-np.linspace(0.0, 1.0, d))) @ Q.T)
        X = _mixture(g, n, means, [np.linalg.cholesky(c) for c in covs], dt)
        H = _normal_reference(X)
    lo, hi = _range(X, np.linalg.eigvalsh(H).max())
    return X, H, lo, hi


def _candidates(seed, count):
    """H = R R^T, R lower triangular, diagonal exp(U[-4, 0]), off-diagonal U[-1, 1]."""
    r = np.random.default_rng(seed)
    R = np.zeros((count, 2, 2))
    R[:, 0, 0], R[:, 1, 1] = np.exp(r.uniform(-4.0, 0.0, size=(2, count)))
    R[:, 1, 0] = r.uniform(-1.0, 1.0, size=count)
    return R @ R.transpose(0, 2, 1)


# the widest candidate: a search over many datasets keeps one grid and one padding
WIDEST = np.array([[1.0, 1.0], [1.0, 2.0]])
SEARCH_LO, SEARCH_HI = [-13.0, -13.0], [14.0, 14.0]


def _search_inputs(case, seed):
    return _plane(_gen(seed), case["n"], 1.0, torch.float32), _candidates(seed, case["nH"])


def _search_padding(case):
    return kde.kde_plan_info_compute(_grid(case), SEARCH_LO, SEARCH_HI,
                                     (2.0 if case["kind"] == "lscv" else 1.0) * WIDEST).P


def _ragged_inputs(case, seed):
    r, g, out = random.Random(case["shapes"]), _gen(seed), []
    sides = [m for m in (64, 128, 256, 512, 1024) if case["M_lo"] <= m <= case["M_hi"]]
    for _ in range(case["count"]):
        n, m = _between(r, case["n_lo"], case["n_hi"]), r.choice(sides)
        s = n ** (-1.0 / 3.0)
        H = _rotated(s * r.uniform(0.5, 2.0), s * r.uniform(0.02, 0.3), r.uniform(0.0, math.pi))
        X = _plane(g, n, 1.0, torch.float32)
        out.append((X, H, (m, m), *_range(X, np.linalg.eigvalsh(H).max())))
    return out


def _datasets(case, seed):
    """count datasets of 2-5 components each, one after another."""
    B, n, g = case["count"], case["n"], _gen(seed)
    u = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    k = torch.randint(2, 6, (B, 1), generator=g, device="cuda")
    w = torch.where(torch.arange(5, device="cuda") < k, -torch.log(u(B, 5)) - torch.log(u(B, 5)), 0.0)
    c = torch.multinomial(w, n, replacement=True, generator=g)
    means, ang = 6.0 * u(B, 5, 2) - 3.0, math.pi * u(B, 5)
    sd = torch.sqrt(torch.exp(math.log(0.05) + (math.log(1.5) - math.log(0.05)) * u(B, 5, 2)))
    z = torch.randn(B, n, 2, generator=g, device="cuda") * torch.gather(sd, 1, c[..., None].expand(-1, -1, 2))
    a = torch.gather(ang, 1, c)
    x = torch.gather(means, 1, c[..., None].expand(-1, -1, 2))
    x = x + torch.stack([torch.cos(a) * z[..., 0] - torch.sin(a) * z[..., 1],
                         torch.sin(a) * z[..., 0] + torch.cos(a) * z[..., 1]], dim=-1)
    return x.reshape(B * n, 2).contiguous(), np.arange(B + 1, dtype=np.int64) * n


def _network(seed, hidden=256):
    """He-normal parameters, flat: W1, b1, W2, b2, W3, b3."""
    r, shapes = np.random.default_rng(seed), [(hidden, kde.FEAT_DIM), (hidden, hidden), (3, hidden)]
    return [(math.sqrt(2.0 / b) * r.standard_normal((a, b)), 0.1 * r.standard_normal(a)) for a, b in shapes]


def _mlp_inputs(case, seed):
    """Rows as kde_features2 makes them: block roots of unit mass, then the moments."""
    g, B = _gen(seed), case["count"]
    F = torch.zeros(B, kde.FEAT_DIM, device="cuda")
    m = torch.relu(torch.randn(B, 1024, generator=g, device="cuda"))
    F[:, :1024] = 8.0 * m / m.norm(dim=1, keepdim=True)
    F[:, 1024:1029] = torch.randn(B, 5, generator=g, device="cuda")
    F[:, 1029] = 1.0
    T = torch.rand(B, 3, generator=g, device="cuda") * 2.2 - 2.8
    return F, T


# ---------------------------------------------------------------------------
# What a program has in hand, and one pass.
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind, s = case["kind"], {"kind": case["kind"]}
    if kind == "eval":
        X, H, lo, hi = _eval_inputs(case, seed)
        plan = kde.Plan(_grid(case), lo, hi, H, precision=case["precision"])
        counts = torch.empty(plan.M, dtype=torch.int64, device="cuda")
        K = torch.empty(plan.info.kspec_elems, dtype=plan.real_dtype(), device="cuda")
        dens = torch.empty(plan.M, dtype=plan.real_dtype(), device="cuda")
        s.update(counts=counts, dens=dens,
                 path=kde.PreparedPath(plan, X, counts, K, dens, plan.workspace()))
    elif kind in ("densities", "lscv"):
        X, H = _search_inputs(case, seed)
        plan = kde.Plan(_grid(case), SEARCH_LO, SEARCH_HI, H[0], P_min=_search_padding(case))
        s.update(X=X, H=H, plan=plan, counts=torch.empty(plan.M, dtype=torch.int64, device="cuda"))
        if kind == "densities":
            s.update(dens=torch.empty((len(H),) + plan.M, device="cuda"),
                     ws=torch.empty(kde.kde_fft_eval_multi_workspace_bytes(plan), dtype=torch.uint8, device="cuda"))
        else:
            s.update(cands=kde.LscvCands(plan, H), R=torch.empty(plan.info.P[0], plan.info.P[1], device="cuda"),
                     scores=torch.empty(len(H), dtype=torch.float64, device="cuda"),
                     ws=torch.empty(kde.kde_lscv_autocorr_workspace_bytes(plan), dtype=torch.uint8, device="cuda"))
    elif kind == "ragged":
        sets = _ragged_inputs(case, seed)
        plan = kde.BatchPlan([(M, lo, hi, H, X.shape[0]) for X, H, M, lo, hi in sets])
        # the tuner's usual choice, set by hand so that every pass is the same work
        plan.set_mode("staged")
        plan.set_shape(64, 64)
        s.update(plan=plan, X=torch.cat([x[0] for x in sets]), ws=plan.workspace(),
                 dens=torch.empty(plan.density_elems, device="cuda"))
    elif kind == "mlp":
        net = kde.MLP(max_batch=256)
        net.set_params(np.concatenate([v.ravel() for wb in _network(seed) for v in wb]))
        F, T = _mlp_inputs(case, seed)
        s.update(net=net, F=F, T=T, loss=torch.empty(1, device="cuda"),
                 grads=torch.empty(net.nparam, device="cuda"))
    else:
        X, off = _datasets(case, seed)
        sc, B = learned.LscvScorer(case["n"]), case["count"]
        P = sc.plan.info.P
        sc.bprep = kde.BatchPrep(sc.plan, B, X.shape[0])
        s.update(X=X, off=off, sc=sc, F=torch.empty(B, kde.FEAT_DIM, device="cuda"),
                 R=torch.empty(B, P[0], P[1], device="cuda"), ns=np.diff(off))
        if kind == "label":
            s.update(scores=torch.empty(B, sc.cand_set.nH, dtype=torch.float64, device="cuda"),
                     ws=torch.empty(max(256, sc.cand_set.batch_workspace_bytes(B)), dtype=torch.uint8, device="cuda"))
        else:
            net = kde.MLP(max_batch=256)
            net.set_params(np.concatenate([v.ravel() for wb in _network(7) for v in wb]))
            offs = 0.5 * learned.NEIGHBOUR_OFFSETS * learned.STEP
            ends = [np.array([g[i] for g in (learned.A_GRID, learned.BETA_GRID, learned.C_GRID)]) for i in (0, -1)]
            s.update(net=net, TH=torch.empty(B, 3, device="cuda"), offs=offs, box_lo=ends[0] - 0.5 * learned.STEP,
                     box_hi=ends[1] + 0.5 * learned.STEP, ref=learned.normal_reference_thetas(s["ns"]),
                     scores=torch.empty(B, len(offs) + 1, dtype=torch.float64, device="cuda"),
                     out=torch.empty(B, 6, dtype=torch.float64, device="cuda"),
                     ws=torch.empty(max(256, kde.lscv_theta_select_workspace_bytes(sc.plan, B, len(offs))),
                                    dtype=torch.uint8, device="cuda"))
    return s


def run(s):
    """One pass.  LSCV scores are computed from an FP32 autocorrelation and
    FP32 terms, so they are returned as the FP32 numbers that they are."""
    kind = s["kind"]
    if kind == "eval":
        s["path"]()
        return {"counts": s["counts"], "density": s["dens"]}
    if kind == "densities":
        kde.kde_bin(s["X"], SEARCH_LO, SEARCH_HI, s["plan"].M, counts=s["counts"])
        kde.kde_fft_eval_multi(s["plan"], s["X"].shape[0], s["H"], s["counts"], density=s["dens"], workspace=s["ws"])
        return {"counts": s["counts"], "density": s["dens"]}
    if kind == "lscv":
        kde.kde_bin(s["X"], SEARCH_LO, SEARCH_HI, s["plan"].M, counts=s["counts"])
        kde.kde_autocorrelation(s["plan"], s["counts"], R=s["R"], workspace=s["ws"])
        s["cands"].score(s["X"].shape[0], s["R"], lscv=s["scores"], workspace=s["ws"])
        return {"counts": s["counts"], "R": s["R"], "lscv": s["scores"].float()}
    if kind == "ragged":
        return {"density": s["plan"].eval(s["X"], density=s["dens"], workspace=s["ws"])}
    if kind == "mlp":
        s["net"].loss_grad(s["F"], s["T"], loss=s["loss"], grads=s["grads"])
        return {"loss": s["loss"], "grads": s["grads"]}
    sc = s["sc"]
    sc.prepare_batch(s["X"], s["off"], F=s["F"], Rs=s["R"])
    if kind == "label":
        sc.cand_set.score_batch(s["ns"], s["R"], lscv=s["scores"], workspace=s["ws"])
        return {"features": s["F"], "R": s["R"], "lscv": s["scores"].float()}
    s["net"].forward(s["F"], Y=s["TH"])
    kde.kde_lscv_theta_select(sc.plan, s["ns"], s["TH"], s["box_lo"], s["box_hi"], s["offs"], s["ref"], s["R"],
                              lscv=s["scores"], out=s["out"], workspace=s["ws"])
    return {"features": s["F"], "R": s["R"], "theta": s["TH"], "lscv": s["scores"].float()}


def work(case):
    """Inputs read once, outputs written once; transforms at 2.5 N log2 N flops of the unpadded grid."""
    kind = case["kind"]
    fft = lambda N: 2.5 * N * math.log2(max(N, 2))  # noqa: E731
    if kind in ("eval", "densities", "lscv"):
        d, N, n = case.get("d", 2), math.prod(_grid(case)), case["n"]
        bin_b = n * d * (8 if case.get("samples") == "f64" else 4) + 8 * N
        bin_f = n * (3 * d + 2 * 2 ** d)
        if kind == "eval":
            return {"bytes": bin_b + N * (8 if case["precision"] == "f64" else 4), "flops": bin_f + 3 * fft(N)}
        if kind == "densities":
            return {"bytes": bin_b + 4 * N * case["nH"], "flops": bin_f + fft(N) * (1 + 2 * case["nH"])}
        return {"bytes": bin_b + 4 * N + 8 * case["nH"], "flops": bin_f + 2 * fft(N) + 8 * 2 * case["nH"] * N / 64}
    if kind == "ragged":
        r, b, f = random.Random(case["shapes"]), 0, 0.0
        sides = [m for m in (64, 128, 256, 512, 1024) if case["M_lo"] <= m <= case["M_hi"]]
        for _ in range(case["count"]):
            n, m = _between(r, case["n_lo"], case["n_hi"]), r.choice(sides)
            r.uniform(0, 1), r.uniform(0, 1), r.uniform(0, 1)
            b, f = b + 8 * n + 4 * m * m, f + 14 * n + 3 * fft(m * m)
        return {"bytes": b, "flops": f}
    params = 1088 * 256 + 256 * 256 + 3 * 256 + 515
    if kind == "mlp":
        return {"bytes": 4 * (case["count"] * 1091 + 2 * params), "flops": 2 * case["count"] * (1088 * 256 * 2 + 256 * 256 * 3)}
    B, n, lags = case["count"], case["n"], 5000
    cand = 2 * (1008 if kind == "label" else 28)
    return {"bytes": B * (8 * n + 4 * 1088 + 4 * 256 * 256 + 8 * cand // 2),
            "flops": B * (20 * n + 2 * fft(256 * 256) + 8 * cand * lags)}


# ---------------------------------------------------------------------------
# The same results in 64 bits.
# ---------------------------------------------------------------------------
def _counts(X, lo, hi, M):
    """Linear binning in units of 2^-32 with the entry point's rounding rules, as float64 samples."""
    d, dt = len(M), X.dtype
    keep, base, Q = torch.ones(X.shape[0], dtype=torch.bool, device="cuda"), [], []
    for k in range(d):
        t = (X[:, k] - torch.tensor(lo[k], dtype=dt, device="cuda")) * \
            torch.tensor((M[k] - 1) / (hi[k] - lo[k]), dtype=dt, device="cuda")
        keep &= (t >= 0) & (t <= M[k] - 1)
        i = torch.clamp(torch.floor(t), 0, M[k] - 2)
        base.append(i.long())
        Q.append(torch.round((t - i).double() * 2.0 ** 32))
    out = torch.zeros(math.prod(M), dtype=torch.int64, device="cuda")
    for corner in itertools.product((0, 1), repeat=d):
        w, at = torch.full((X.shape[0],), 2.0 ** 32, dtype=torch.float64, device="cuda"), 0
        for k in range(d):
            up = torch.floor(w * Q[k] / 2.0 ** 32 + 0.5)
            w = up if corner[k] else w - up
            at = at * M[k] + base[k] + corner[k]
        out.index_add_(0, torch.where(keep, at, 0), torch.where(keep, w, 0.0).long())
    return out.double().reshape(M) * 2.0 ** -32


def _support(H, delta, M):
    r = 3.7 * math.sqrt(np.linalg.eigvalsh(H).max())
    return [min(m - 1, math.ceil(r / x)) for m, x in zip(M, delta)]


def _kernel(H, delta, L):
    """K_H on the lags -L .. L of every axis."""
    d, A = len(L), np.linalg.inv(H)
    u = torch.meshgrid(*[torch.arange(-v, v + 1, dtype=torch.float64, device="cuda") * x for v, x in zip(L, delta)],
                       indexing="ij")
    q = sum(A[a, b] * u[a] * u[b] for a in range(d) for b in range(d))
    return torch.exp(-0.5 * q) / math.sqrt((2 * math.pi) ** d * np.linalg.det(H))


def _density(c, n, H, lo, hi, C=None, P=None):
    M, d = tuple(c.shape), c.dim()
    delta = [(hi[k] - lo[k]) / (M[k] - 1) for k in range(d)]
    L = _support(H, delta, M)
    if P is None:
        P = [2 * ((m + v + 2) // 2) for m, v in zip(M, L)]
        C = torch.fft.rfftn(c, s=P)
    k = torch.zeros(P, dtype=torch.float64, device="cuda")
    k[tuple(slice(0, 2 * v + 1) for v in L)] = _kernel(H, delta, L)
    k = torch.roll(k, [-v for v in L], dims=list(range(d)))
    return torch.fft.irfftn(C * torch.fft.rfftn(k), s=P)[tuple(slice(0, m) for m in M)] / n


def _autocorrelation(c, P):
    """Cyclic autocorrelation on the padded lengths P, over the last two axes."""
    return torch.fft.irfft2(torch.fft.rfft2(c, s=P).abs().square(), s=P)


def _lscv(H, R, ns, lo, hi, M):
    """LSCV of H for every autocorrelation in R (B x P_0 x P_1)."""
    delta, n = [(hi[k] - lo[k]) / (M[k] - 1) for k in range(2)], ns.double()
    sums = []
    for A in (H, 2.0 * H):
        L = _support(A, delta, M)
        i, j = (torch.arange(-v, v + 1, device="cuda") % p for v, p in zip(L, R.shape[1:]))
        sums.append((R[:, i][:, :, j] * _kernel(A, delta, L)).sum(dim=(1, 2)))
    k0 = 1.0 / (2 * math.pi * math.sqrt(np.linalg.det(H)))
    return sums[1] / n**2 - 2.0 * (sums[0] - n * k0) / (n * (n - 1))


def _learned_inputs(case, seed):
    """Features and autocorrelations of the standardised datasets."""
    X, off = _datasets(case, seed)
    B, n, M = case["count"], case["n"], (learned.GRID_M,) * 2
    x = X.double().reshape(B, n, 2)
    mean, sd = x.mean(1, keepdim=True), x.std(1, correction=0, keepdim=True)
    z = (x - mean) / sd
    ends = [learned.GRID_LO] * 2, [learned.GRID_HI] * 2
    F = torch.zeros(B, kde.FEAT_DIM, dtype=torch.float64, device="cuda")
    c = torch.stack([_counts(z[b].float(), *ends, M) for b in range(B)])
    w = M[0] // 32
    F[:, :1024] = 8.0 * torch.sqrt(c.reshape(B, 32, w, 32, w).sum(dim=(2, 4)) / n).reshape(B, 1024)
    F[:, 1024] = (z[..., 0] * z[..., 1]).mean(1)
    F[:, 1025:1027] = (z ** 3).mean(1)
    F[:, 1027] = (z ** 4).mean(dim=(1, 2)) - 3.0
    F[:, 1028], F[:, 1029] = math.log10(n) / 4.0, 1.0
    return F, c, torch.full((B,), n, device="cuda"), ends


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        X, H, lo, hi = _eval_inputs(case, seed)
        return {"counts": None, "density": _density(_counts(X, lo, hi, _grid(case)), case["n"], H, lo, hi)}
    if kind == "densities":
        X, H = _search_inputs(case, seed)
        lo, hi, M = SEARCH_LO, SEARCH_HI, _grid(case)
        c = _counts(X, lo, hi, M)
        P = [2 * m for m in M]
        C, out = torch.fft.rfftn(c, s=P), torch.empty((len(H),) + M, dtype=torch.float64, device="cuda")
        for k, h in enumerate(H):
            out[k] = _density(c, case["n"], h, lo, hi, C, P)
        return {"counts": None, "density": out}
    if kind == "lscv":
        X, H = _search_inputs(case, seed)
        lo, hi, M = SEARCH_LO, SEARCH_HI, _grid(case)
        R = _autocorrelation(_counts(X, lo, hi, M), _search_padding(case))
        n = torch.tensor([case["n"]], device="cuda")
        return {"counts": None, "R": R, "lscv": torch.cat([_lscv(h, R[None], n, lo, hi, M) for h in H])}
    if kind == "ragged":
        return {"density": torch.cat([_density(_counts(X, lo, hi, M), X.shape[0], H, lo, hi).reshape(-1)
                                      for X, H, M, lo, hi in _ragged_inputs(case, seed)])}
    if kind == "mlp":
        F, T = _mlp_inputs(case, seed)
        ps = [torch.tensor(v, device="cuda").float().double().requires_grad_() for wb in _network(seed) for v in wb]
        h = F.double()
        for i in range(3):
            h = h @ ps[2 * i].T + ps[2 * i + 1]
            h = torch.relu(h) if i < 2 else h
        loss = (h - T.double()).square().sum() / case["count"]
        loss.backward()
        return {"loss": loss.detach().reshape(1), "grads": torch.cat([p.grad.reshape(-1) for p in ps])}
    F, c, n, ends = _learned_inputs(case, seed)
    R = _autocorrelation(c, learned.LscvScorer(case["n"]).plan.info.P)
    if kind == "select":  # theta follows the network's 16-bit operands, and the scores follow theta
        return {"features": F, "R": R, "theta": None, "lscv": None}
    M = (learned.GRID_M,) * 2
    s = [_lscv(h, R, n, *ends, M) for h in learned.thetas_to_H(learned.candidate_thetas())]
    return {"features": F, "R": R, "lscv": torch.stack(s, dim=1)}
