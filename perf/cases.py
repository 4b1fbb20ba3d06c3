"""The work that is timed: what a planner has this library do, through its
public entry points, from the smallest operator call to whole solves of the
realistic plan.

Every plan is a synthetic head-and-neck case: an ellipsoidal body on a 2.5 mm
grid, an ellipsoidal target, three organs at risk, spots from three beams on a
5 mm lateral grid with several energy layers each, Gaussian lateral falloff and
a Bragg-like depth curve, and setup-shift and range scenarios.  Entries are
truncated to a given number per spot.  The seed sets the layers' ranges (and so
the matrices), the weights' scatter and the vectors.  Sizes: the realistic
workload (299k voxels, 5000 spots, 13 scenarios, 127M entries), the small
batched plans, the tiny plan and odd sizes between.
"""
import math

import numpy as np
import torch

from paper_2304_14568_gb300 import rpt

DEV = "cuda"
H = 2.5                     # voxel edge, mm
SPACING = 5.0               # lateral spot grid, mm
SIGMA = 3.0                 # lateral falloff, mm
RCUT = 4.0 * SIGMA
FORMATS = {"f32": (rpt.F32, 4), "bf16": (rpt.BF16, 2), "fp8": (rpt.FP8E4M3, 1)}
SMALL_PLANS = ((12_000, 250), (18_000, 350), (24_000, 450), (30_000, 550))


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _op(name, what, voxels, spots, scenarios, per_spot, fmt="f32", index=32, exact_sums=False, **more):
    return dict(name=name, what=what, voxels=voxels, spots=spots, scenarios=scenarios, per_spot=per_spot,
                fmt=fmt, index=index, exact_sums=exact_sums, **more)


def listed():
    return [
        # one application of every scenario's normal operator on a plan that a
        # test or an interactive check uses: latency, launches, copies
        _op("normal_tiny", "normal", 8_000, 200, 13, 960),
        # the same on the realistic plan: the row pass every solver repeats
        _op("normal_realistic", "normal", 299_088, 5000, 13, 2000),
        # a quantised plan of odd width (BF16 values, 16-bit indices)
        _op("normal_bf16", "normal", 170_000, 3001, 13, 1700, fmt="bf16", index=16),
        # gradient and objective at a plan, in the bitwise reproducible sums, ragged sizes
        _op("gradient_exact", "gradient", 61_000, 1777, 7, 1500, index=16, exact_sums=True),
        # dose report of a small plan: objective and the doses of every scenario
        _op("dose_report", "dose", 54_000, 950, 13, 1700),
        # the allocation-free operator on one scenario held by the caller on the device
        _op("noalloc_realistic", "noalloc", 299_088, 5000, 1, 2000),
        # first iterations of a whole ADMM-BB solve, small plan: launch-bound control flow
        _op("admm_small", "admm", 12_000, 250, 13, 1700, iterations=30),
        # the headline solve (CG x-updates, realistic plan, autotuned), its first iterations
        _op("admm_realistic", "admm", 299_088, 5000, 13, 2000, iterations=12),
        # the projected-gradient baseline
        _op("pgd", "pgd", 100_000, 2000, 13, 1700, iterations=10),
        # weight sweep (training targets of the learned warm start): new weights, then
        # the paper's cached-factor solve, which forms and inverts B_s again
        _op("sweep_factor", "sweep", 48_000, 1250, 13, 1700, iterations=20),
        # several small plans solved side by side
        _op("batched_small", "batched", 0, 0, 13, 1700, plans=4, iterations=12),
        # learned warm start: loss and gradient of one minibatch (9 -> 512 x 3 -> spots)
        dict(name="learned_grad", what="mlp", hidden=512, layers=3, spots=200, rows=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["normal", "normal", "gradient", "dose", "noalloc", "admm", "admm", "pgd", "sweep",
                       "batched", "mlp"])
    if what == "mlp":
        return dict(what="mlp", hidden=rng.choice([512, 256, 384]), layers=rng.choice([1, 2, 3]),
                    spots=_log(rng, 200, 5000), rows=_log(rng, 32, 512))
    if what == "batched":
        return dict(what="batched", voxels=0, spots=0, scenarios=rng.choice([5, 7, 13]),
                    per_spot=_log(rng, 900, 1700), fmt="f32", index=rng.choice([32, 16]), exact_sums=False,
                    plans=rng.choice([2, 3, 4]), iterations=rng.randint(6, 12))
    voxels = _log(rng, 8_000, 299_088)
    sc = (voxels / 299_088.0) ** (1.0 / 3.0)
    # a spot count in proportion to the target's cross-section, as planners place
    # them, wider or narrower by up to 1.5; every lateral position has a spot
    spots = int(round(5000 * sc * sc * math.exp(rng.uniform(-0.4, 0.0))))
    spots = max(spots, int(3 * 1.5 * math.pi * (32.0 * sc + 5.0) ** 2 / SPACING ** 2) + 5)
    c = dict(what=what, voxels=voxels, spots=spots, scenarios=rng.choice([1, 3, 7, 9, 13]),
             per_spot=_log(rng, 800, 2000), fmt="f32", index=rng.choice([32, 32, 16]), exact_sums=False)
    if what in ("normal", "gradient"):
        c["fmt"] = rng.choice(["f32", "f32", "bf16", "fp8"])
        c["exact_sums"] = rng.random() < 0.2
    if what == "noalloc":
        c["scenarios"] = 1
        c["index"] = 32
    if what == "sweep":          # n^3 work per scenario: up to the listed size
        c["spots"] = min(c["spots"], 1300)
        c["voxels"] = min(c["voxels"], 50_000)
    if what in ("admm", "pgd", "sweep"):
        c["iterations"] = rng.randint(5, 12)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _scenarios(count):
    """(dx, dy, dz, range factor): nominal, axis shifts, range errors, then lattice shifts."""
    s, k = 3.0, 0.035
    out = [(0.0, 0.0, 0.0, 0.0)]
    for ax in range(3):
        for sg in (s, -s):
            d = [0.0, 0.0, 0.0]
            d[ax] = sg
            out.append((d[0], d[1], d[2], 0.0))
    for dz in (0.0, s, -s):
        out += [(0.0, 0.0, dz, k), (0.0, 0.0, dz, -k)]
    return out[:count]


def _inside(P, center, semi):
    c = torch.tensor(center, dtype=torch.float64, device=DEV)
    r = torch.tensor(semi, dtype=torch.float64, device=DEV)
    return (((P - c) / r) ** 2).sum(1) <= 1.0


def _depth(Q, semi, d):
    """Distance from Q back along -d to the body's surface (nan outside)."""
    s = torch.tensor(semi, dtype=torch.float64, device=Q.device)
    D = torch.tensor(d, dtype=torch.float64, device=Q.device) / s
    X = Q / s
    a, b, c = float((D * D).sum()), X @ D, (X * X).sum(1) - 1.0
    t = (b + torch.sqrt(b * b - a * c)) / a
    return torch.where(c <= 0, t, torch.full_like(t, math.nan))


def _beam(angle, sc, body, count, rng):
    """Spots of one beam: lateral positions whose ray crosses the target, energy
    layers in proportion to the depth span crossed, ranges jittered by the seed."""
    th = math.radians(angle)
    d, e1, e2 = (math.cos(th), math.sin(th), 0.0), (-math.sin(th), math.cos(th), 0.0), (0.0, 0.0, 1.0)
    iso = np.array([10.0, 5.0, 0.0]) * sc
    semi = np.array([30.0, 28.0, 32.0]) * sc + 1.0
    hc = int(math.ceil(semi.max() / SPACING)) + 1
    ij = np.stack(np.meshgrid(np.arange(-hc, hc + 1), np.arange(-hc, hc + 1), indexing="ij"), -1).reshape(-1, 2)
    o = iso + SPACING * (ij[:, :1] * np.array(e1) + ij[:, 1:] * np.array(e2))
    X, D = (o - iso) / semi, np.array(d) / semi
    a, b, c = (D * D).sum(), X @ D, (X * X).sum(1) - 1.0
    disc = b * b - a * c
    hit = disc > 0
    ij, o, b, disc = ij[hit], o[hit], b[hit], disc[hit]
    root = np.sqrt(disc)
    p_in = o + ((-b - root) / a)[:, None] * np.array(d)
    p_out = o + ((-b + root) / a)[:, None] * np.array(d)
    d_in = _depth(torch.from_numpy(p_in), body, d).numpy()
    d_out = _depth(torch.from_numpy(p_out), body, d).numpy()
    L = len(ij)
    span = d_out - d_in + 2.0
    quota = span / span.sum() * (count - L)
    cnt = 1 + np.floor(quota).astype(np.int64)
    cnt[np.argsort(-(quota - np.floor(quota)), kind="stable")[:count - int(cnt.sum())]] += 1
    lay = np.arange(int(cnt.max()))
    R = d_in[:, None] + (lay[None, :] + 0.5) / cnt[:, None] * (d_out - d_in)[:, None]
    R = R + rng.uniform(-1.0, 1.0, size=R.shape)
    live = lay[None, :] < cnt[:, None]
    Rmax = np.where(live, R, 0.0).max(1)
    lo = ij.min(0) - 6
    table = np.full(tuple(ij.max(0) + 7 - lo), -1, dtype=np.int64)
    table[ij[:, 0] - lo[0], ij[:, 1] - lo[1]] = np.arange(L)
    g = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(DEV)  # noqa: E731
    return dict(d=d, e1=e1, e2=e2, iso=g(iso), lo=lo, shape=table.shape, table=g(table), R=g(R), live=g(live),
                reach=g(Rmax + 4.0 * (0.012 * Rmax + 1.0)), start=g(np.cumsum(cnt) - cnt), count=count)


def _entries(geo, shift, kappa):
    """(row, spot, dose) of every entry of one scenario, before truncation."""
    rows, spots, vals = [], [], []
    K = int(math.ceil(RCUT / SPACING)) + 1
    off = torch.arange(-K, K + 1, device=DEV)
    du, dv = off.repeat_interleave(2 * K + 1), off.repeat(2 * K + 1)
    base = 0
    for B in geo["beams"]:
        Q = geo["P"] + torch.tensor(shift, dtype=torch.float64, device=DEV)
        X = Q - B["iso"]
        u = X @ torch.tensor(B["e1"], dtype=torch.float64, device=DEV)
        v = X @ torch.tensor(B["e2"], dtype=torch.float64, device=DEV)
        dep = _depth(Q, geo["body"], B["d"]) * (1.0 + kappa)
        near = torch.isfinite(dep) & (u.abs() <= SPACING * B["shape"][0]) & (v.abs() <= SPACING * B["shape"][1])
        vox = near.nonzero()[:, 0]
        u, v, dep = u[vox], v[vox], dep[vox]
        iu = torch.round(u / SPACING).long()[:, None] + du
        iv = torch.round(v / SPACING).long()[:, None] + dv
        a, b = iu - int(B["lo"][0]), iv - int(B["lo"][1])
        ok = (a >= 0) & (a < B["shape"][0]) & (b >= 0) & (b < B["shape"][1])
        lat = torch.where(ok, B["table"][a.clamp(0, B["shape"][0] - 1), b.clamp(0, B["shape"][1] - 1)], -1)
        r2 = (u[:, None] - iu * SPACING) ** 2 + (v[:, None] - iv * SPACING) ** 2
        at = ((lat >= 0) & (r2 <= RCUT * RCUT) & (dep[:, None] <= B["reach"][lat.clamp(min=0)])).nonzero()
        lat, r2, who = lat[at[:, 0], at[:, 1]], r2[at[:, 0], at[:, 1]], at[:, 0]
        R, dep = B["R"][lat], dep[who]
        sR = 0.012 * R + 1.0
        x = dep[:, None] - R
        keep = (B["live"][lat] & (x <= 4.0 * sR)).nonzero()
        p, l = keep[:, 0], keep[:, 1]
        x, sR = x[p, l], sR[p, l]
        g = torch.exp(-(x * x) / (2.0 * sR * sR))
        bragg = torch.where(x <= 0, 0.25 + 0.75 * g, g)
        rows.append(vox[who[p]])
        spots.append(B["start"][lat[p]] + l + base)
        vals.append((torch.exp(-r2 / (2.0 * SIGMA * SIGMA))[p] * bragg).float())
        base += B["count"]
    return torch.cat(rows), torch.cat(spots), torch.cat(vals)


def _problem(voxels, spots, scenarios, per_spot, seed):
    """A plan's data on the device: per scenario CSR (row_ptr, col, val), weights, prescription."""
    rng = np.random.default_rng(seed)
    sc = (voxels / 299_088.0) ** (1.0 / 3.0)
    nx, ny, nz = (max(8, int(round(k * sc))) for k in (128, 128, 96))
    ax = [(torch.arange(k, dtype=torch.float64, device=DEV) + 0.5 - k / 2.0) * H for k in (nx, ny, nz)]
    Z, Y, X = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    P = torch.stack([X.reshape(-1), Y.reshape(-1), Z.reshape(-1)], 1)
    body = [90.0 * sc, 105.0 * sc, 118.0 * sc]
    P = P[_inside(P, [0.0, 0.0, 0.0], body)]
    m = P.shape[0]
    target = _inside(P, [10.0 * sc, 5.0 * sc, 0.0], [30.0 * sc, 28.0 * sc, 32.0 * sc])
    organ = torch.zeros(m, dtype=torch.bool, device=DEV)
    for c, r in (((-42, 0, 10), (12, 15, 20)), ((35, 45, -10), (10, 12, 15)), ((0, -55, 0), (8, 8, 60))):
        organ |= _inside(P, [t * sc for t in c], [t * sc for t in r])
    w = torch.ones(m, dtype=torch.float64, device=DEV)
    w[organ] = 10.0 * math.exp(rng.uniform(-0.5, 0.5))
    w[target] = 100.0 * math.exp(rng.uniform(-0.5, 0.5))
    p = torch.where(target, 70.0, 0.0).double()
    per = [spots // 3 + (1 if k < spots % 3 else 0) for k in range(3)]
    geo = dict(P=P, body=body, beams=[_beam(a, sc, body, c, rng) for a, c in zip((0.0, 120.0, 240.0), per)])
    tau, csr, scale = None, [], None
    for dx, dy, dz, kappa in _scenarios(scenarios):
        r, c, v = _entries(geo, (dx, dy, dz), kappa)
        if tau is None:
            want = min(per_spot * spots, v.numel())
            tau = float(torch.sort(v, descending=True).values[want - 1] / v.max())
        keep = v >= tau * v.max()
        r, c, v = r[keep], c[keep], v[keep]
        order = torch.argsort(r * spots + c)
        r, c, v = r[order], c[order], v[order]
        rp = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
        rp[1:] = torch.cumsum(torch.bincount(r, minlength=m), 0)
        if scale is None:   # x = 1 gives a third of the prescription in the target
            dose = torch.zeros(m, dtype=torch.float64, device=DEV).index_add_(0, r, v.double())
            scale = 70.0 / 3.0 / float(dose[target].mean())
        csr.append((rp.int(), c.int(), (v * scale).float()))
    return dict(m=m, n=spots, N=scenarios, csr=csr, w=w, p=p, target=target)


def _plan(prob, case):
    return rpt.Plan(prob["m"], prob["n"], prob["N"], *_host(prob)[:5], lb=np.zeros(prob["n"]),
                    ub=np.full(prob["n"], 10.0), value_format=FORMATS[case["fmt"]][0], index_width=case["index"],
                    accumulate=1 if case["exact_sums"] else 0,
                    autotune=1 if case["what"] == "admm" and case["voxels"] > 100_000 else 0)


def _host(prob):
    rp, ci, va = ([t[k].cpu().numpy() for t in prob["csr"]] for k in range(3))
    return rp, ci, va, prob["w"].cpu().numpy(), prob["p"].cpu().numpy()


class _Fields:
    """One problem of a batched plan."""

    def __init__(self, prob):
        self.m, self.n, self.N = prob["m"], prob["n"], prob["N"]
        self.row_ptr, self.col_idx, self.val, self.voxel_w, self.presc = _host(prob)
        self.scen_weight, self.lb, self.ub = None, np.zeros(self.n), np.full(self.n, 10.0)


def _vector(case, prob, seed):
    """The spot vector an operator is applied to: search directions of mixed sign
    for the normal operator, plans (non-negative) for the others."""
    rng = np.random.default_rng(seed + 1_000_003)
    if case["what"] in ("normal", "noalloc"):
        return rng.standard_normal(prob["N"] * prob["n"])
    return rng.uniform(0.0, 6.0, size=prob["n"])


def _network(case, seed):
    """Parameters (Glorot-uniform weights, small biases), features and targets of a minibatch."""
    rng = np.random.default_rng(seed)
    dims = [9] + [case["hidden"]] * case["layers"] + [case["spots"]]
    par = []
    for i, o in zip(dims[:-1], dims[1:]):
        a = math.sqrt(6.0 / (i + o))
        par += [rng.uniform(-a, a, size=i * o), rng.uniform(-0.05, 0.05, size=o)]
    X = rng.uniform(-1.0, 1.0, size=(case["rows"], 9)).astype(np.float32)
    Y = np.clip(rng.normal(0.1, 0.1, size=(case["rows"], case["spots"])), 0.0, 1.0).astype(np.float32)
    return dims, np.concatenate(par).astype(np.float32), X, Y


def _new_weights(prob, seed):
    """Weights of the next point of a weight sweep."""
    rng = np.random.default_rng(seed + 7)
    w = prob["w"].cpu().numpy() * math.exp(rng.uniform(-0.3, 0.3))
    p = prob["p"].cpu().numpy() * rng.uniform(0.9, 1.05)
    return w, p


def prepare(case, seed):
    what = case["what"]
    if what == "mlp":
        dims, par, X, Y = _network(case, seed)
        net = rpt.Mlp(9, case["hidden"], case["layers"], case["spots"], seed=1)
        net.set_params(par)
        return dict(case=case, net=net, X=X, Y=Y)
    if what == "batched":
        probs = [_Fields(_problem(v, s, case["scenarios"], case["per_spot"], seed + 101 * k))
                 for k, (v, s) in enumerate(SMALL_PLANS[:case["plans"]])]
        return dict(case=case, plan=rpt.Plan.batched(probs, index_width=case["index"]))
    prob = _problem(case["voxels"], case["spots"], case["scenarios"], case["per_spot"], seed)
    if what == "noalloc":
        rp, ci, va = prob["csr"][0]
        v = torch.from_numpy(_vector(case, prob, seed)).float().to(DEV)
        return dict(case=case, m=prob["m"], n=prob["n"], rp=rp, ci=ci, va=va, w=prob["w"].float(), v=v,
                    u=torch.empty_like(v), stream=torch.cuda.current_stream().cuda_stream)
    state = dict(case=case, plan=_plan(prob, case), rho=50.0)
    if what in ("normal", "gradient", "dose"):
        state["x"] = _vector(case, prob, seed)
    if what == "sweep":
        state["w"], state["p"] = _new_weights(prob, seed)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    what = case["what"]
    if what == "normal":
        return state["plan"].apply_normal(state["x"], rho=state["rho"])
    if what == "gradient":
        g, f = state["plan"].gradient(state["x"])
        return dict(g=g, f=f)
    if what == "dose":
        f, dose = state["plan"].objective(state["x"], dose=True)
        return dict(f=f, dose=dose)
    if what == "noalloc":
        rpt.normal_apply_noalloc(state["m"], state["n"], state["rp"].data_ptr(), state["ci"].data_ptr(),
                                 state["va"].data_ptr(), state["w"].data_ptr(), state["v"].data_ptr(), 50.0,
                                 state["u"].data_ptr(), state["stream"])
        return state["u"]
    if what == "admm":
        z, info = state["plan"].admm_bb_solve(max_iter=case["iterations"])
        return dict(z=z, f=info["f"])
    if what == "pgd":
        x, info = state["plan"].pgd_solve(max_iter=case["iterations"])
        return dict(x=x, f=info["f"])
    if what == "sweep":
        state["plan"].set_weights(state["w"], state["p"])
        z, info = state["plan"].admm_bb_solve(subproblem=rpt.SUB_CHOL, max_iter=case["iterations"])
        return dict(z=z, f=info["f"])
    if what == "batched":
        xs, info, _ = state["plan"].admm_bb_solve_batched(max_iter=case["iterations"])
        return dict(x=xs, f=info["f"])
    loss, grad = state["net"].loss_grad(state["X"], state["Y"])
    return dict(loss=loss, grad=grad)


# What one ADMM-BB iteration needs of the matrix: the residual pass and the CG
# steps that its stopping rule asks for (about ten over the first iterations),
# one pass for the final objective of the solve.
CG_PASSES = 11


def work(case):
    what = case["what"]
    if what == "mlp":
        dims = [9] + [case["hidden"]] * case["layers"] + [case["spots"]]
        prods = [i * o for i, o in zip(dims[:-1], dims[1:])]
        par = sum(prods) + sum(dims[1:])
        return dict(bytes=float(8 * par + 4 * case["rows"] * (9 + case["spots"])),
                    flops=float(2 * case["rows"] * (3 * sum(prods) - prods[0])))
    if what == "batched":
        sizes = SMALL_PLANS[:case["plans"]]
    else:
        sizes = [(case["voxels"], case["spots"])]
    N = case["scenarios"]
    nnz = sum(s for _, s in sizes) * case["per_spot"] * N
    n = sum(s for _, s in sizes)
    matrix = nnz * (FORMATS[case["fmt"]][1] + case["index"] // 8)
    it = case.get("iterations", 0)
    if what == "normal":
        return dict(bytes=float(matrix + 16 * N * n), flops=float(4 * nnz))
    if what == "noalloc":
        return dict(bytes=float(matrix + 8 * case["voxels"] + 8 * n), flops=float(4 * nnz))
    if what == "gradient":
        return dict(bytes=float(matrix + 16 * n), flops=float(4 * nnz))
    if what == "dose":
        return dict(bytes=float(matrix + 8 * n + 8 * N * case["voxels"]), flops=float(2 * nnz))
    if what in ("admm", "batched"):
        return dict(bytes=float(matrix * (CG_PASSES * it + 1)), flops=float(4 * nnz * CG_PASSES * it))
    if what == "pgd":       # gradient and one trial an iteration
        return dict(bytes=float(matrix * 2 * it), flops=float(6 * nnz * it))
    # forming, factoring and inverting B_s (n^3 multiply-adds), then one read of the
    # inverse's half (it is symmetric) per iteration
    return dict(bytes=float(matrix * 2 + 2 * n * n * N * it), flops=float(2.0 * N * n ** 3 + 2.0 * n * n * N * it))


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _stored(prob, case):
    """Each scenario's (row, column, value) in 64 bits, the values as the format
    stores them: code times the column's scale, code = round(value / scale)."""
    out = []
    for rp, ci, va in prob["csr"]:
        r = torch.repeat_interleave(torch.arange(prob["m"], device=DEV), (rp[1:] - rp[:-1]).long())
        c, v = ci.long(), va.double()
        if case["fmt"] != "f32":
            top = 1.0 if case["fmt"] == "bf16" else 448.0
            s = torch.zeros(prob["n"], device=DEV).scatter_reduce_(0, c, va, "amax") / top
            s = torch.where(s > 0, s, torch.ones_like(s))
            q = (va / s[c]).to(torch.bfloat16 if case["fmt"] == "bf16" else torch.float8_e4m3fn)
            v = q.double() * s.double()[c]
        out.append((r, c, v))
    return out


def _dot(prob, e, x):
    return torch.zeros(prob["m"], dtype=torch.float64, device=DEV).index_add_(0, e[0], e[2] * x[e[1]])


def _scatter(prob, e, t):
    return torch.zeros(prob["n"], dtype=torch.float64, device=DEV).index_add_(0, e[1], e[2] * t[e[0]])


def _objective(prob, E, w, p, x):
    return sum(float((w * (_dot(prob, e, x) - p) ** 2).sum()) for e in E)


def exact(case, seed):
    what = case["what"]
    if what in ("admm", "batched"):
        return None         # the x-updates stop CG early: no value that is the iterate's own
    if what == "mlp":
        return _exact_network(case, seed)
    prob = _problem(case["voxels"], case["spots"], case["scenarios"], case["per_spot"], seed)
    E, w, p = _stored(prob, case), prob["w"], prob["p"]
    if what in ("normal", "noalloc"):
        v = torch.from_numpy(_vector(case, prob, seed)).to(DEV)
        if what == "noalloc":
            v, w = v.float().double(), w.float().double()
        V = v.reshape(prob["N"], prob["n"])
        U = torch.stack([_scatter(prob, e, w * _dot(prob, e, V[s])) + 25.0 * V[s] for s, e in enumerate(E)])
        return U[0] if what == "noalloc" else U.cpu().numpy()
    if what in ("gradient", "dose"):
        x = torch.from_numpy(_vector(case, prob, seed)).to(DEV)
        D = [_dot(prob, e, x) for e in E]
        f = sum(float((w * (d - p) ** 2).sum()) for d in D)
        if what == "dose":
            return dict(f=f, dose=torch.stack(D).cpu().numpy())
        g = sum(_scatter(prob, e, 2.0 * w * (d - p)) for e, d in zip(E, D))
        return dict(g=g.cpu().numpy(), f=f)
    if what == "pgd":
        return _exact_pgd(case, prob, E, w, p)
    w, p = (torch.from_numpy(a).to(DEV) for a in _new_weights(prob, seed))
    return _exact_factor(case, prob, E, w, p)


def _exact_pgd(case, prob, E, w, p):
    n = prob["n"]
    v = torch.full((n,), 1.0 / math.sqrt(n), dtype=torch.float64, device=DEV)
    for _ in range(30):
        u = sum(_scatter(prob, e, w * _dot(prob, e, v)) for e in E)
        lam = float(u.norm())
        v = u / lam
    alpha = 4.0 / (2.0 * lam)
    x = torch.zeros(n, dtype=torch.float64, device=DEV)
    fx = _objective(prob, E, w, p, x)
    for _ in range(case["iterations"]):
        g = sum(_scatter(prob, e, 2.0 * w * (_dot(prob, e, x) - p)) for e in E)
        t = alpha
        for _ in range(30):
            xt = (x - t * g).clamp(0.0, 10.0)
            ft = _objective(prob, E, w, p, xt)
            if ft <= fx + 1e-4 * float(g @ (xt - x)):
                break
            t *= 0.5
        rel, x, fx = abs(fx - ft) / abs(fx), xt, ft
        if rel <= 1e-5:
            break
    return dict(x=x.cpu().numpy(), f=fx)


def _exact_factor(case, prob, E, w, p):
    """ADMM-BB with exact x-updates from a cold start: B_s x_s = c_s by Cholesky."""
    n, N = prob["n"], prob["N"]
    G, b = [], []
    for e in E:
        B = torch.zeros(n, n, dtype=torch.float64, device=DEV)
        rows = torch.unique(e[0])
        place = torch.zeros(prob["m"], dtype=torch.long, device=DEV)
        place[rows] = torch.arange(rows.numel(), device=DEV)
        for k in range(0, rows.numel(), 8192):
            lo, hi = k, min(k + 8192, rows.numel())
            at = (place[e[0]] >= lo) & (place[e[0]] < hi)
            A = torch.zeros(hi - lo, n, dtype=torch.float64, device=DEV)
            A[place[e[0][at]] - lo, e[1][at]] = e[2][at] * torch.sqrt(w[e[0][at]])
            B += A.T @ A
        G.append(B)
        b.append(_scatter(prob, e, w * p))
    rho = 2.0 * sum(float(torch.diagonal(B).sum()) for B in G) / N / n
    eye = torch.eye(n, dtype=torch.float64, device=DEV)
    Lc = [torch.linalg.cholesky(B + 0.5 * rho * eye) for B in G]
    z = torch.zeros(n, dtype=torch.float64, device=DEV)
    y = torch.zeros(N, n, dtype=torch.float64, device=DEV)
    dprev, step = torch.zeros_like(y), rho
    for k in range(case["iterations"]):
        x = torch.stack([torch.cholesky_solve((b[s] + 0.5 * rho * z - 0.5 * y[s])[:, None], Lc[s])[:, 0]
                         for s in range(N)])
        zn = (x + y / rho).mean(0).clamp(0.0, 10.0)
        d = x - zn
        if k > 0:
            dd = d - dprev
            bb = -step * float((dd * dprev).sum()) / max(float((dd * dd).sum()), 1e-300)
            step = bb if math.isfinite(bb) and bb > 0 else rho
        else:
            step = rho
        y = y + step * d
        rp, rd = float(d.norm()), math.sqrt(N) * rho * float((zn - z).norm())
        ep = 1e-4 * math.sqrt(N * n) + 1e-4 * max(float(x.norm()), math.sqrt(N) * float(zn.norm()))
        ed = 1e-4 * math.sqrt(N * n) + 1e-4 * float(y.norm())
        z, dprev = zn, d
        if rp <= ep and rd <= ed:
            break
    return dict(z=z.cpu().numpy(), f=_objective(prob, E, w, p, z))


def _exact_network(case, seed):
    """Loss and gradient of the network in 64 bits (no rounding of operands)."""
    dims, par, X, Y = _network(case, seed)
    q = torch.from_numpy(par).double().to(DEV).requires_grad_(True)
    a, at = torch.from_numpy(X).double().to(DEV), 0
    for l, (i, o) in enumerate(zip(dims[:-1], dims[1:])):
        W, c = q[at:at + i * o].reshape(o, i), q[at + i * o:at + i * o + o]
        at += i * o + o
        a = a @ W.T + c
        if l + 2 < len(dims):
            a = torch.relu(a)
    loss = ((a - torch.from_numpy(Y).double().to(DEV)) ** 2).mean()
    loss.backward()
    return dict(loss=float(loss.detach()), grad=q.grad.cpu().numpy())
