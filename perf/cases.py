"""Workloads of the Vecchia likelihood library as its users run them, through the Python binding.

Each case is one call (or the short sequence of calls that belong together) of
``paper_2403_07412_gb300.vecchia`` on synthetic geospatial data: the likelihood of one field, its
gradient, an optimiser's step through autograd, many (field, theta) pairs at once, kriging, and a new
data set from its locations to its likelihood.  Sizes, smoothness values, orderings and conditioning
sizes are those of the paper's studies as this repository's benchmark and tests run them.

A case is a dict of plain values.  Keys: ``op`` (see ``run``), ``n`` locations, ``m`` conditioning
points, ``nu`` (smoothness, or the exponent of the power exponential), ``beta``, ``sigma2``,
``tau2``, ``order`` ("random", "maxmin" or "morton"), ``layout`` ("uniform", "clustered" or
"sphere"), ``kernel`` ("matern" or "powexp").  The batched call has ``fields`` and ``thetas``, the
prediction ``n_new``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2403_07412_gb300 import datagen
from paper_2403_07412_gb300 import vecchia as V

ORDERS = {"random": V.ORDER_RANDOM, "maxmin": V.ORDER_MAXMIN, "morton": V.ORDER_MORTON}
KERNELS = {"matern": V.KERNEL_MATERN, "powexp": V.KERNEL_POWEXP}
RADIUS = 6371.0  # km: distances, and beta, on the sphere
DEVICE = "cuda"
FEATURES = 1024  # random Fourier features of a synthetic field
BATCH_NUS = (0.5, 1.0, 1.5)


def _case(name, op, n, m, nu, beta, sigma2=1.0, tau2=0.01, order="random", layout="uniform", kernel="matern", **more):
    return dict(name=name, op=op, n=n, m=m, nu=nu, beta=beta, sigma2=sigma2, tau2=tau2, order=order, layout=layout,
                kernel=kernel, **more)


def listed():
    return [
        # A small study: one likelihood of 2,000 locations without nugget; latency and launches count.
        _case("loglik_2k_m10", "loglik", 2000, 10, 0.5, 0.1, tau2=0.0),
        # An optimiser's step on a small data set: value and gradient.
        _case("grad_6k_m30", "grad", 6000, 30, 1.5, 0.05),
        # The many-candidates end of an optimiser: a mid-sized field's likelihood.
        _case("loglik_100k_m30", "loglik", 100_000, 30, 1.5, 0.05),
        # Small conditioning sets over a large field, with the gradient.
        _case("grad_250k_m10", "grad", 250_000, 10, 1.0, 0.03, tau2=0.02),
        # The smooth end of the paper's study (nu = 5/2), value and gradient, at m = 60.
        _case("grad_250k_m60", "grad", 250_000, 60, 2.5, 0.03, sigma2=1.5, tau2=0.05),
        # The headline workload: a million clustered locations, maxmin ordering, general nu.
        _case("grad_1m_m60", "grad", 1_000_000, 60, 1.0, 0.02, order="maxmin", layout="clustered"),
        # Per-location likelihood terms (diagnostics of a fit), an odd size, Morton ordering.
        _case("terms_77777_m45", "terms", 77_777, 45, 0.5, 0.05, tau2=0.05, order="morton"),
        # The large conditioning sets of the paper's performance study.
        _case("grad_50k_m120", "grad", 50_000, 120, 1.5, 0.05),
        # Longitude/latitude data with the paper's real-data model (power exponential), value and gradient.
        _case("sphere_100k_m60", "grad", 100_000, 60, 1.0, 50.0, layout="sphere", kernel="powexp"),
        # Kriging: 250,000 observed, 25,000 new locations, mean and variance.
        _case("predict_25k_m30", "predict", 250_000, 30, 1.5, 0.01, n_new=25_000),
        # Model selection over many fields and parameter vectors in one launch.
        _case("batched_12x8", "batched", 60_000, 60, 1.0, 0.05, fields=12, thetas=8),
        # A new data set, from its locations to its first likelihood and gradient.
        _case("new_data_100k_m30", "dataset", 100_000, 30, 0.5, 0.05),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _flops(m):
    """FP64 operations of one location's block: factorisation and the two triangular solves."""
    k = m + 1
    return k**3 / 3 + k**2 / 2 + k / 6 + k**2


def draw(rng):
    op = rng.choice(["loglik", "loglik", "grad", "grad", "grad", "terms", "autograd", "predict", "batched", "dataset"])
    if op in ("predict", "batched"):
        m = round(_log_uniform(rng, 5, 63))
    else:
        m = rng.choice([round(_log_uniform(rng, 5, 63)), round(_log_uniform(rng, 5, 63)), rng.randint(64, 150)])
    most = min(250_000.0, 3e10 / _flops(m))
    n = int(_log_uniform(rng, 500, most))
    nu = rng.choice([0.5, 1.0, 1.5, 2.5, round(rng.uniform(0.4, 2.4), 3)])
    case = dict(op=op, n=n, m=min(m, n - 1), nu=nu, beta=round(_log_uniform(rng, 0.01, 0.2), 5),
                sigma2=round(rng.uniform(0.5, 2.0), 3), tau2=round(rng.uniform(0.005, 0.1), 4),
                order=rng.choice(["random", "random", "morton", "maxmin"]), layout=rng.choice(["uniform", "uniform", "clustered"]),
                kernel="matern")
    if op in ("loglik", "grad", "predict") and rng.random() < 0.3:
        case.update(layout="sphere", order="random", kernel="powexp", n=min(n, 100_000), nu=round(rng.uniform(0.5, 1.0), 3),
                    beta=round(_log_uniform(rng, 20.0, 200.0), 3))
    if op == "predict":
        case["n_new"] = rng.randint(100, 30_000)
    if op == "batched":
        case.update(fields=rng.randint(2, 12), thetas=rng.randint(1, 8), n=min(n, 60_000), order="random", layout="uniform",
                    nu=1.0, m=max(8, case["m"]))
    if op in ("dataset", "autograd"):
        case["order"] = "random"
    return case


# ------------------------------------------------------------------ inputs
def _locations(case, n, seed):
    if case["layout"] == "sphere":
        return datagen.sphere_locations(n, seed)
    if case["layout"] == "clustered":
        return datagen.gmm_locations(n, seed)
    return datagen.uniform_locations(n, seed)


def _field(case, xy, theta, seed):
    """A field at the locations: a Matérn draw (on the sphere in chordal distance, of the same range)."""
    p, th = xy, list(theta)
    if case["layout"] == "sphere":
        p = datagen.sphere_coords(xy, RADIUS)
    if case["kernel"] == "powexp":
        th[1], th[2] = th[1] ** (1.0 / th[2]), 0.5
    return datagen.field_rff(p, th, seed, features=FEATURES, device=DEVICE)


def _seeds(case, seed):
    return datagen.BASE_SEED + 1009 * int(seed)


def _theta(case, seed):
    """The parameters of one evaluation: the case's, moved a little by the seed as an optimiser moves them."""
    g = datagen.rng(_seeds(case, seed) + 7)
    nu = case["nu"] if case["op"] != "autograd" else case["nu"] * math.exp(g.uniform(-0.05, 0.05))
    return (case["sigma2"] * math.exp(g.uniform(-0.05, 0.05)), case["beta"] * math.exp(g.uniform(-0.05, 0.05)), nu,
            case["tau2"] * math.exp(g.uniform(-0.05, 0.05)))


def _plan(case, xy, seed):
    radius = RADIUS if case["layout"] == "sphere" else None
    plan = V.Plan(xy, case["m"], order=ORDERS[case["order"]], seed=seed, radius=radius)
    plan.set_kernel(KERNELS[case["kernel"]])
    return plan


def _batch_shape(case):
    """Sizes and conditioning sizes of a batch's fields: spread over a factor of six in n and over three m."""
    f = np.arange(case["fields"])
    ns = np.floor(case["n"] * 6.0 ** (-f / max(1, case["fields"] - 1))).astype(int)
    ms = np.array([case["m"], max(4, case["m"] // 2), max(4, case["m"] // 6)])[f % 3]
    return ns, ms


def _batch_inputs(case, seed):
    s = _seeds(case, seed)
    ns, ms = _batch_shape(case)
    fields = []
    for f, (n, m) in enumerate(zip(ns, ms)):
        c = dict(case, n=int(n), m=int(m), op="loglik")
        xy = _locations(c, int(n), s + 31 * f)
        fields.append((c, xy, _field(c, xy, _theta(c, seed + f), s + 31 * f + 1), s + 31 * f + 2))
    return fields, datagen.theta_candidates(case["fields"], case["thetas"], s + 5)


def prepare(case, seed):
    s = _seeds(case, seed)
    if case["op"] == "batched":
        fields, thetas = _batch_inputs(case, seed)
        plans = [_plan(c, xy, ps) for c, xy, _, ps in fields]
        ys = [torch.as_tensor(y, device=DEVICE) for _, _, y, _ in fields]
        V.vecchia_batched_prepare(list(BATCH_NUS))
        batch = V.Batch(plans, ys, case["thetas"], want_grad=True)
        return {"op": "batched", "batch": batch, "thetas": torch.as_tensor(thetas, device=DEVICE).contiguous()}
    theta = _theta(case, seed)
    xy = _locations(case, case["n"], s)
    state = {"op": case["op"], "case": case, "theta": theta, "seed": s + 2,
             "y": torch.as_tensor(_field(case, xy, theta, s + 1), device=DEVICE)}
    if case["op"] == "dataset":
        state["xy"] = xy
        return state
    state["plan"] = _plan(case, xy, s + 2)
    if case["op"] == "predict":
        state["new"] = _locations(case, case["n_new"], s + 3)
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    op = state["op"]
    if op == "batched":  # every (field, theta): value and gradient
        return {"out": state["batch"].run(state["thetas"])}
    theta, y = state["theta"], state["y"]
    if op == "loglik":
        return {"loglik": V.vecchia_loglik(state["plan"], y, theta)}
    if op == "grad":
        g = V.vecchia_loglik_grad(state["plan"], y, theta)
        return {"loglik": g[0:1], "grad": g[1:4]}
    if op == "terms":
        return {"terms": V.vecchia_loglik_terms(state["plan"], y, theta)}
    if op == "autograd":  # an optimiser's step that estimates the smoothness too
        th = torch.tensor(theta, dtype=torch.float64, requires_grad=True)
        ll = V.VecchiaLogLik.apply(th, state["plan"], y)
        ll.backward()
        return {"loglik": ll.detach(), "grad": th.grad}
    if op == "predict":
        mean, var = V.vecchia_predict(state["plan"], state["new"], y, theta)
        return {"mean": mean, "var": var}
    if op == "dataset":
        plan = _plan(state["case"], state["xy"], state["seed"])
        g = V.vecchia_loglik_grad(plan, y, theta)
        terms = V.vecchia_loglik_terms(plan, y, theta)
        plan.close()
        return {"loglik": g[0:1], "grad": g[1:4], "terms": terms}
    raise ValueError(op)


def work(case):
    """Coordinates, data and conditioning sets read once, results written once; the blocks' FP64 operations."""
    def of(n, m, thetas=1):
        return n * (16.0 + 8.0 + 4.0 * m), float(n) * _flops(m) * thetas

    if case["op"] == "batched":
        parts = [of(int(n), int(m), case["thetas"]) for n, m in zip(*_batch_shape(case))]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n, m = case["n"], case["m"]
    if case["op"] == "predict":  # observed points read once, new points and their results
        return {"bytes": n * 24.0 + case["n_new"] * (32.0 + 4.0 * m), "flops": case["n_new"] * _flops(m)}
    b, f = of(n, m)
    if case["op"] == "terms":
        return {"bytes": b + 8.0 * n, "flops": f}
    if case["op"] == "autograd":  # value and gradient, and two likelihoods for the smoothness
        return {"bytes": b, "flops": 3 * f}
    if case["op"] == "dataset":  # the terms are the summands of the value
        return {"bytes": b + 8.0 * n, "flops": f}
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in 64 bits, plain torch and numpy
def _random_order(n, seed):
    """Fisher–Yates from the end, driven by splitmix64."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.uint64(0x9E3779B97F4A7C15) * np.arange(1, n, dtype=np.uint64)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    at = np.arange(n - 1, 0, -1, dtype=np.uint64)
    js = (z % (at + np.uint64(1))).tolist()
    p = list(range(n))
    for i, j in zip(range(n - 1, 0, -1), js):
        p[i], p[j] = p[j], p[i]
    return np.array(p)


def _morton_order(xy):
    lo, hi = xy.min(0), xy.max(0)
    q = np.clip(np.floor((xy - lo) / (hi - lo) * 65536.0), 0, 65535).astype(np.uint64)
    code = np.zeros(len(xy), dtype=np.uint64)
    for b in range(16):
        code |= ((q[:, 0] >> np.uint64(b)) & np.uint64(1)) << np.uint64(2 * b)
        code |= ((q[:, 1] >> np.uint64(b)) & np.uint64(1)) << np.uint64(2 * b + 1)
    return np.lexsort((np.arange(len(xy)), code))


def _points(case, xy):
    return datagen.sphere_coords(xy, 1.0) if case["layout"] == "sphere" else xy


def _nearest(points, queries, m, previous):
    """Rows of the m nearest points of each query (with `previous`, of the points before it), -1 where there are fewer."""
    n, out = points.shape[0], []
    rows = max(1, int(2e8 // n))
    for a in range(0, queries.shape[0], rows):
        q = queries[a:a + rows]
        cols = min(n, a + q.shape[0]) if previous else n
        d = torch.zeros(q.shape[0], cols, dtype=torch.float64, device=DEVICE)
        for k in range(points.shape[1]):
            t = q[:, k, None] - points[None, :cols, k]
            d += t * t
        if previous:
            d.masked_fill_(torch.arange(cols, device=DEVICE)[None, :] >= torch.arange(a, a + q.shape[0], device=DEVICE)[:, None], math.inf)
        v, j = torch.topk(d, min(m, cols), dim=1, largest=False)
        j = torch.where(torch.isinf(v), -1, j)
        out.append(torch.nn.functional.pad(j, (0, m - j.shape[1]), value=-1))
    return torch.cat(out)


def _bessel_k(nu, x):
    """K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt by the trapezoidal rule (geometric convergence), x > 0."""
    h, acc = 0.1, 0.5 * torch.exp(-x)
    for k in range(1, 240):
        acc += torch.exp(-x * math.cosh(k * h)) * math.cosh(nu * k * h)
    return acc * h


def _correlation(kernel, d, beta, nu):
    """rho(d) and d rho / d beta."""
    if kernel == "powexp":
        w = d.pow(nu) / beta
        return torch.exp(-w), torch.exp(-w) * w / beta
    x = d / beta
    e = torch.exp(-x)
    if nu == 0.5:
        return e, x * e / beta
    if nu == 1.5:
        return (1 + x) * e, x * x * e / beta
    if nu == 2.5:
        return (1 + x + x * x / 3) * e, x * x * (1 + x) / 3 * e / beta
    z = torch.clamp(x, min=1e-150)
    c = 2.0 ** (1.0 - nu) / math.gamma(nu) * z.pow(nu)
    rho, db = c * _bessel_k(nu, z), c * z * _bessel_k(abs(nu - 1.0), z) / beta
    return torch.where(x == 0, torch.ones_like(rho), rho), torch.where(x == 0, torch.zeros_like(db), db)


def _blocks(case, points, y, sets, own_points, own_y, theta, want_grad):
    """Conditional residual and variance of each row's location given its set, and the term's gradient."""
    sigma2, beta, nu, tau2 = theta
    m, res, var, grads = sets.shape[1], [], [], []
    rows = max(1, int(4e7 // (m + 1) ** 2))
    for a in range(0, sets.shape[0], rows):
        J = sets[a:a + rows]
        ok = J >= 0
        pts = torch.cat([points[J.clamp(min=0)], own_points[a:a + rows, None, :]], 1)
        d2 = torch.zeros(J.shape[0], m + 1, m + 1, dtype=torch.float64, device=DEVICE)
        for k in range(pts.shape[2]):
            t = pts[:, :, None, k] - pts[:, None, :, k]
            d2 += t * t
        d = torch.sqrt(d2)
        if case["layout"] == "sphere":
            d = 2.0 * RADIUS * torch.asin(torch.clamp(0.5 * d, max=1.0))
        live = torch.nn.functional.pad(ok, (0, 1), value=True)
        mask = live[:, :, None] & live[:, None, :]
        rho, db = _correlation(case["kernel"], d, beta, nu)
        rho, db = rho * mask, db * mask
        eye = torch.eye(m + 1, dtype=torch.float64, device=DEVICE)
        C = sigma2 * rho + tau2 * eye * live[:, None, :]
        C = C + eye * (~live)[:, None, :]
        yJ = torch.where(ok, y[J.clamp(min=0)], 0.0)
        L = torch.linalg.cholesky(C[:, :m, :m])
        wa = torch.cholesky_solve(torch.stack([C[:, :m, m], yJ], 2), L)
        w, al = wa[:, :, 0], wa[:, :, 1]
        s = sigma2 + tau2 - (C[:, :m, m] * w).sum(1)
        r = own_y[a:a + rows] - (w * yJ).sum(1)
        res.append(r)
        var.append(s)
        if want_grad:
            wh = torch.cat([-w, torch.ones_like(r)[:, None]], 1)
            g = (r / s)[:, None] * torch.nn.functional.pad(al, (0, 1)) + (0.5 * (r * r / (s * s) - 1 / s))[:, None] * wh
            t2 = (wh * g * live).sum(1)
            s2 = (wh * torch.bmm(rho, g[:, :, None])[:, :, 0]).sum(1)
            b = sigma2 * (wh * torch.bmm(db, g[:, :, None])[:, :, 0]).sum(1)
            grads.append(torch.stack([s2, b, t2], 1))
    return torch.cat(res), torch.cat(var), torch.cat(grads) if want_grad else None


def _exact_terms(case, xy, y, order_seed, theta, want_grad, sets=None):
    """(terms, gradient terms, conditioning sets) in the plan's order."""
    pts = _points(case, xy)
    perm = _random_order(len(pts), order_seed) if case["order"] == "random" else _morton_order(xy)
    p = torch.as_tensor(pts[perm], device=DEVICE)
    yo = torch.as_tensor(y, device=DEVICE)[torch.as_tensor(perm, device=DEVICE)]
    if sets is None:
        sets = _nearest(p, p, case["m"], True)
    r, s, g = _blocks(case, p, yo, sets, p, yo, theta, want_grad)
    return -0.5 * r * r / s - 0.5 * torch.log(s) - 0.5 * math.log(2 * math.pi), g, sets


def exact(case, seed):
    general = case["kernel"] == "matern" and case["nu"] not in (0.5, 1.5, 2.5)
    s = _seeds(case, seed)
    if case["op"] == "batched":
        ns, ms = _batch_shape(case)
        if sum(float(n) * m * m for n, m in zip(ns, ms)) * case["thetas"] > 3e9:
            return None
        fields, thetas = _batch_inputs(case, seed)
        out = torch.empty(case["fields"], case["thetas"], 4, dtype=torch.float64)
        for f, (c, xy, y, ps) in enumerate(fields):
            sets = None
            for t in range(case["thetas"]):
                l, g, sets = _exact_terms(c, xy, y, ps, tuple(thetas[f, t]), True, sets)
                out[f, t, 0], out[f, t, 1:] = l.sum().cpu(), g.sum(0).cpu()
        return {"out": out}
    if case["order"] == "maxmin" or case["n"] * float(case["m"]) ** 2 > (3e8 if general else 1.2e9):
        return None
    theta = _theta(case, seed)
    xy = _locations(case, case["n"], s)
    y = _field(case, xy, theta, s + 1)
    if case["op"] == "predict":
        new = _locations(case, case["n_new"], s + 3)
        p, q = (torch.as_tensor(_points(case, v), device=DEVICE) for v in (xy, new))
        zero = torch.zeros(len(new), dtype=torch.float64, device=DEVICE)
        r, v, _ = _blocks(case, p, torch.as_tensor(y, device=DEVICE), _nearest(p, q, case["m"], False), q, zero, theta, False)
        return {"mean": -r, "var": v}
    op = case["op"]
    l, g, _ = _exact_terms(case, xy, y, s + 2, theta, op in ("grad", "dataset"))
    if op == "loglik":
        return {"loglik": l.sum()[None]}
    if op == "grad":
        return {"loglik": l.sum()[None], "grad": g.sum(0)}
    if op == "terms":
        return {"terms": l}
    if op == "autograd":  # the derivative in nu is a finite difference by definition
        return {"loglik": l.sum(), "grad": None}
    return {"loglik": l.sum()[None], "grad": g.sum(0), "terms": l}
