"""What a user of this library has it do, as cases that can be timed and checked.

Each case is one call (or one training step, or one run of the search) through
the Python entry points of paper_2602_05179_gb300.api on seeded inputs: the
scenario-batched Split (hard, soft and fleet-limited capacity, its gradient,
batched plans, the candidate search) and the order-up-to reinsertion (two
actions, route options).  Sizes and distributions are those of the repository's
workloads, tests and benchmark, with odd and ragged ones between them.
"""
import math

import numpy as np
import torch

from paper_2602_05179_gb300 import api

SEARCH_MOVES = ("2opt", "relocate", "swap")


def listed():
    return [
        # one short tour, a few scenarios: the call's latency and launches
        {"name": "split_small", "op": "split", "n": 50, "Q": 100, "S": 1000, "demand": "poisson", "lam": 10.0,
         "tour": "random", "preds": "u16"},
        # the large evaluation of one tour: every scenario's cost and predecessors
        {"name": "split_large", "op": "split", "n": 500, "Q": 200, "S": 1_000_000, "demand": "uniform", "hi": 30,
         "tour": "random", "preds": "u16"},
        # an ordinary evaluation with odd sizes: rows that are no multiple of 16 bytes, a last tile of 17, int32 predecessors
        {"name": "split_ragged", "op": "split", "n": 333, "Q": 120, "S": 50_001, "demand": "poisson", "lam": 10.0,
         "tour": "sweep", "preds": "i32"},
        # long tour, capacity above 254 (16-bit staging), costs only: scoring one candidate of a large instance
        {"name": "split_long", "op": "split", "n": 1000, "Q": 400, "S": 100_000, "demand": "uniform", "hi": 30,
         "tour": "random", "preds": ""},
        # the penalised model: every split allowed, excess load priced
        {"name": "split_soft", "op": "split", "n": 500, "Q": 200, "S": 200_000, "demand": "uniform", "hi": 30,
         "tour": "sweep", "preds": "u16", "beta": 10.0},
        # a training step: mean cost and its gradient with respect to the distance matrix
        {"name": "split_gradient", "op": "gradient", "n": 300, "Q": 120, "S": 100_000, "demand": "poisson", "lam": 10.0,
         "tour": "random"},
        # a bounded fleet: at most K routes, with the route of every customer
        {"name": "split_fleet", "op": "fleet", "n": 500, "Q": 200, "S": 65_536, "K": 42, "demand": "uniform", "hi": 30,
         "tour": "random"},
        # a generation of candidates of uneven length, each with its own scenarios, in one replay of a plan
        {"name": "plan_uneven", "op": "plan", "B": 1024, "n_lo": 20, "n_hi": 1000, "Q": 150, "S": 2048, "lam": 12.0},
        # the candidate loop: a few iterations of 1024 neighbours on one scenario set
        {"name": "search", "op": "search", "n": 100, "Q": 100, "S": 10_000, "B": 1024, "iters": 4, "lam": 10.0},
        # a few customers' reinsertion, with a unit cost: latency again
        {"name": "reinsert_small", "op": "reinsert", "T": 30, "U": 100, "S": 1000, "lam": 8.0, "unit": 0.5, "table": False,
         "value0": False, "K": 0},
        # the large reinsertion: value and policy of every scenario
        {"name": "reinsert_large", "op": "reinsert", "T": 60, "U": 200, "S": 1_000_000, "lam": 8.0, "unit": 0.0, "table": False,
         "value0": False, "K": 0},
        # the same with four candidate routes a day, each with its residual capacity per scenario
        {"name": "reinsert_routes", "op": "reinsert", "T": 60, "U": 200, "S": 1_000_000, "lam": 8.0, "unit": 0.0, "table": False,
         "value0": False, "K": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["split", "split", "split", "gradient", "fleet", "plan", "search", "reinsert", "reinsert", "reinsert"])
    if op in ("split", "gradient", "fleet"):
        # capacity over mean demand (customers on a route) stays that of the listed cases
        c = {"op": op, "demand": rng.choice(["poisson", "uniform"]), "tour": rng.choice(["random", "sweep"])}
        if c["demand"] == "poisson":
            c["lam"] = rng.uniform(6.0, 14.0)
            mean = c["lam"]
        else:
            c["hi"] = rng.randint(15, 40)
            mean = (1 + c["hi"]) / 2
        c["Q"] = int(mean * rng.uniform(9.0, 26.0))
    if op == "split":
        c["n"] = _log(rng, 50, 1000)
        c["S"] = _log(rng, 1000, min(1_000_000, 500_000_000 // c["n"]))
        c["preds"] = rng.choice(["", "u16", "u16", "i32"])
        if rng.random() < 0.3:
            c["beta"] = rng.uniform(2.0, 20.0)
            c["S"] = min(c["S"], 200_000)
        return c
    if op == "gradient":
        c["n"] = _log(rng, 50, 500)
        c["S"] = _log(rng, 1000, 200_000)
        return c
    if op == "fleet":
        c["n"] = _log(rng, 60, 600)
        c["S"] = _log(rng, 1000, min(65_536, 33_000_000 // c["n"]))
        c["Q"] = max(c["Q"], int(c["n"] * mean / 50))  # at most about 50 routes are needed
        need = c["n"] * mean / c["Q"]
        c["K"] = max(2, min(64, int(need * rng.uniform(1.04, 1.3)) + 1))
        return c
    if op == "plan":
        lo = _log(rng, 20, 200)
        c = {"op": op, "B": _log(rng, 16, 1024), "n_lo": lo, "n_hi": rng.randint(lo + 20, 1000),
             "Q": rng.randint(100, 250), "lam": rng.uniform(8.0, 14.0)}
        c["S"] = _log(rng, 500, max(600, min(4096, 1_000_000_000 // (c["B"] * c["n_hi"]))))
        return c
    if op == "search":
        n = _log(rng, 40, 200)
        return {"op": op, "n": n, "Q": rng.randint(80, 140), "S": _log(rng, 1000, 10_000), "B": _log(rng, 64, 1024),
                "iters": rng.randint(1, 4), "lam": rng.uniform(6.0, 12.0)}
    T, U = rng.randint(14, 90), _log(rng, 40, 255)
    K = rng.choice([0, 0, 2, 3, 4, 6])
    return {"op": op, "T": T, "U": U, "S": _log(rng, 1000, min(1_000_000, 60_000_000 // T)), "lam": rng.uniform(4.0, 12.0),
            "unit": rng.choice([0.0, 0.0, 0.25]), "table": K == 0 and rng.random() < 0.25,
            "value0": rng.random() < 0.2, "K": K}


# ------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _poisson(g, lam, shape):
    """Poisson draws by inversion of the table of the distribution function."""
    kmax = int(lam + 12.0 * math.sqrt(lam) + 12.0)
    pmf = [math.exp(-lam)]
    for k in range(1, kmax):
        pmf.append(pmf[-1] * lam / k)
    cdf = torch.tensor(np.cumsum(pmf), dtype=torch.float32, device="cuda")
    out = torch.empty(shape, dtype=torch.int32, device="cuda")
    flat = out.view(-1)
    step = 1 << 26
    for k in range(0, flat.numel(), step):
        part = flat[k:k + step]
        part.copy_(torch.bucketize(torch.rand(part.numel(), generator=g, device="cuda"), cdf, out_int32=True, right=True))
    return out


def _demands(g, c, S, n):
    if c.get("demand", "poisson") == "uniform":
        return torch.randint(1, c["hi"] + 1, (S, n), generator=g, dtype=torch.int32, device="cuda")
    return _poisson(g, c["lam"], (S, n)).clamp_(1, c["Q"])


def _coords(rng, n):
    xy = rng.uniform(0.0, 100.0, (n + 1, 2)).astype(np.float32)
    xy[0] = 50.0  # the depot
    return xy


def _tour(rng, xy, kind):
    n = len(xy) - 1
    if kind == "sweep":  # customers by their angle around the depot
        d = xy[1:].astype(np.float64) - xy[0]
        return (np.argsort(np.arctan2(d[:, 1], d[:, 0]), kind="stable") + 1).astype(np.int32)
    return (rng.permutation(n) + 1).astype(np.int32)


def _inputs(case, seed):
    """Everything a program has in hand before the call, on the GPU."""
    c, op = case, case["op"]
    rng, g = np.random.default_rng(seed), _gen(seed)
    if op == "reinsert":
        T, K = c["T"], c["K"]
        s = {"cons": _poisson(g, c["lam"], (c["S"], T))}
        s["fixed"] = torch.from_numpy(rng.uniform(5.0, 50.0, T).astype(np.float32)).cuda() if K == 0 else None
        s["table"] = None
        if c["table"]:  # holding cost of the stock left, a penalty for none
            t = np.arange(c["U"] + 1, dtype=np.float32)
            t[0] = 60.0
            s["table"] = torch.from_numpy(t).cuda()
        s["rcost"] = s["rcap"] = None
        if K:
            s["rcost"] = torch.from_numpy(rng.uniform(5.0, 50.0, (T, K)).astype(np.float32)).cuda()
            s["rcap"] = torch.randint(0, int(1.25 * c["U"]) + 1, (c["S"], T, K), generator=g, dtype=torch.int32, device="cuda")
        return s
    if op == "plan":
        ns = rng.integers(c["n_lo"], c["n_hi"] + 1, c["B"]).astype(np.int32)
        xys = [_coords(rng, int(n)) for n in ns]
        off = np.zeros(c["B"], np.int64)  # each block starts on 16 bytes
        sizes = (ns.astype(np.int64) * c["S"] + 3) // 4 * 4
        off[1:] = np.cumsum(sizes[:-1])
        return {"ns": ns, "xys": xys, "off": off,
                "tours": torch.from_numpy(np.concatenate([_tour(rng, x, "random") for x in xys])).cuda(),
                "coords": torch.from_numpy(np.concatenate(xys)).cuda(),
                "dem": _poisson(g, c["lam"], (int(sizes.sum()),)).clamp_(1, c["Q"])}
    xy = _coords(rng, c["n"])
    s = {"xy": torch.from_numpy(xy).cuda(), "tour": torch.from_numpy(_tour(rng, xy, c.get("tour", "random"))).cuda(),
         "dem": _demands(g, c, c["S"], c["n"])}
    if op == "gradient":
        x = s["xy"].double()
        s["dist"] = (x[:, None, :] - x[None, :, :]).square().sum(-1).sqrt().float().contiguous().requires_grad_(True)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = dict(case)
    if case["op"] == "plan":
        s["plan"] = api.SplitPlan(s["ns"], s["tours"], s["coords"], s["dem"], case["Q"], case["S"], dem_off=s["off"])
    if case["op"] == "search":
        s["search"] = api.SaaSearch(s["tour"], s["xy"], s["dem"], case["Q"], case["B"], seed=seed, moves=SEARCH_MOVES)
    return s


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "split":
        return api.split_eval(s["tour"], c["Q"], s["dem"], coords=s["xy"], preds=c["preds"] or None,
                              overload_penalty=c.get("beta"))
    if op == "gradient":
        mean = api.SplitMeanCost.apply(s["dist"], s["tour"], s["dem"], c["Q"])
        grad, = torch.autograd.grad(mean, s["dist"])
        return {"mean": mean, "grad": grad}
    if op == "fleet":
        return api.split_fleet_eval(s["tour"], c["Q"], s["dem"], c["K"], coords=s["xy"])
    if op == "plan":
        costs, means = s["plan"].run()
        return {"costs": costs, "means": means}
    if op == "search":
        trace, accepted = s["search"].run(c["iters"])
        tour, means = s["search"].state()
        return {"trace": trace, "accepted": accepted, "tour": tour, "means": means}
    return api.reinsert_eval(c["T"], c["U"], c["U"] // 2, 1.0, 20.0, c["unit"], s["fixed"], s["cons"], table=s["table"],
                             value0=c["value0"], route_cost=s["rcost"], route_cap=s["rcap"])


def work(case):
    c, op = case, case["op"]
    if op == "reinsert":
        S, T, U, K = c["S"], c["T"], c["U"], c["K"]
        by = 4 * S * T * (1 + K) + 4 * S + S * T + (4 * S * (U + 1) if c["value0"] else 0)
        # an addition, a comparison and a minimum for each state that a day can start in
        states = T * (U + 1) if c["value0"] else sum(min(t + 1, U + 1) for t in range(T))
        return {"bytes": by, "flops": 3 * S * states}
    if op == "plan":
        n = c["B"] * (c["n_lo"] + c["n_hi"]) / 2
        return {"bytes": c["S"] * (4 * n + 4 * c["B"]), "flops": 4 * c["S"] * n}
    if op == "search":
        tours = c["iters"] * (c["B"] + 1)
        return {"bytes": 4 * c["S"] * c["n"] + 8 * tours, "flops": 4 * tours * c["S"] * c["n"]}
    n, S = c["n"], c["S"]
    by = 4 * n * S + 4 * S
    if op == "fleet":
        by += 4 * S + n * S
    if op == "gradient":
        by += 8 * (n + 1) * (n + 1) - 4 * S  # the matrix in, its gradient out, no costs
    by += {"": 0, "u16": 2, "i32": 4}[c.get("preds", "")] * n * S
    return {"bytes": by, "flops": 4 * n * S}


# ------------------------------------------------------------- 64-bit values
def _legs(xy, tour, dist=None):
    """(c(0,s_i) - c(s_{i-1},s_i), c(s_i,0)) of every position and the tour's inner length."""
    t = tour.long()
    if dist is None:
        x = xy.double()
        pts = x[t]
        out = (pts - x[0]).square().sum(-1).sqrt()
        back = out
        inner = (pts[1:] - pts[:-1]).square().sum(-1).sqrt()
    else:
        d = dist.detach().double()
        out, back, inner = d[0, t], d[t, 0], d[t[:-1], t[1:]]
    a = out.clone()
    a[1:] -= inner
    return a, back, float(inner.sum())


def _windows(L, Q):
    """The most candidates that any scenario has at each position (L: prefix loads [..., n+1])."""
    n = L.shape[-1] - 1
    flat = L.reshape(-1, n + 1)
    lo = torch.searchsorted(flat, flat[:, 1:] - Q)
    idx = torch.arange(1, n + 1, device=L.device)
    return (idx - lo).amax(0).clamp(min=1).tolist()


def _split64(q, a, ce, Q, beta=None, want_pred=False):
    """K(i) [C, S, n+1] of the hard or soft Split; q [C, S, n] in tour order, a / ce [C, n]."""
    C, S, n = q.shape
    L = torch.zeros((C, S, n + 1), dtype=torch.int64, device="cuda")
    torch.cumsum(q.clamp(min=0), -1, out=L[..., 1:])
    K = torch.zeros((C, S, n + 1), dtype=torch.float64, device="cuda")
    pred = torch.zeros((S, n), dtype=torch.int32, device="cuda") if want_pred else None
    w = _windows(L, Q) if beta is None else list(range(1, n + 1))
    for i in range(1, n + 1):
        lo = max(0, i - min(w[i - 1], i))
        over = (L[..., i:i + 1] - L[..., lo:i]) - Q
        cand = K[..., lo:i] + a[:, None, lo:i]
        cand = cand.masked_fill(over > 0, math.inf) if beta is None else cand + beta * over.clamp(min=0)
        best, at = cand.min(-1)
        K[..., i] = best + ce[:, i - 1:i]
        if want_pred:
            pred[:, i - 1] = (at[0] + lo).int()
    return (K, pred) if want_pred else K


def _chunks(total, size):
    return [(k, min(total, k + size)) for k in range(0, total, size)]


def _exact_split(c, s, dist=None):
    a, ce, D = _legs(s["xy"], s["tour"], dist)
    cols = s["tour"].long() - 1
    beta = float(np.float32(c["beta"])) if c.get("beta") is not None else None
    size = max(64, (40_000_000 if beta is None else 8_000_000) // c["n"])
    cost, counts = [], torch.zeros((3, c["n"]), dtype=torch.float64, device="cuda")
    for lo, hi in _chunks(c["S"], size):
        q = s["dem"][lo:hi].long()[:, cols][None]
        if dist is None:
            cost.append(_split64(q, a[None], ce[None], c["Q"], beta)[0, :, -1] + D)
            continue
        K, pred = _split64(q, a[None], ce[None], c["Q"], want_pred=True)
        cost.append(K[0, :, -1] + D)
        i = torch.full((hi - lo,), c["n"], dtype=torch.int64, device="cuda")
        while bool((i > 0).any()):  # the routes of each scenario, from the last to the first
            on = i[i > 0] - 1
            counts[1] += torch.bincount(on, minlength=c["n"])
            p = pred.long().gather(1, (i - 1).clamp(min=0)[:, None])[:, 0]
            counts[0] += torch.bincount(p[i > 0], minlength=c["n"])
            i = torch.where(i > 0, p, i)
    return torch.cat(cost), counts


def _moved(z, n, tour):
    """The neighbour that draw z makes of `tour`: 2-opt, relocate or swap of two positions."""
    a = (z & 0xFFFFFFFF) % n
    b = (z >> 40) % (n - 1)
    b += b >= a
    kind = ((z >> 32) & 0xFF) % 3
    t = list(tour)
    if kind == 0:
        lo, hi = min(a, b), max(a, b)
        t[lo:hi + 1] = t[lo:hi + 1][::-1]
    elif kind == 1:
        t.insert(b, t.pop(a))
    else:
        t[a], t[b] = t[b], t[a]
    return t


def _splitmix(seed, k):
    m = (1 << 64) - 1
    z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _exact_search(c, s, seed):
    tour, means, trace = s["tour"].tolist(), None, []
    dem = s["dem"].long()
    for it in range(c["iters"]):
        cand = [tour] + [_moved(_splitmix(seed, it * c["B"] + k), c["n"], tour) for k in range(c["B"])]
        t = torch.tensor(cand, dtype=torch.int64, device="cuda")
        means = []
        for lo, hi in _chunks(len(cand), max(1, 12_000_000 // (c["S"] * c["n"]))):
            legs = [_legs(s["xy"], t[k]) for k in range(lo, hi)]
            q = torch.stack([dem[:, t[k] - 1] for k in range(lo, hi)])
            K = _split64(q, torch.stack([x[0] for x in legs]), torch.stack([x[1] for x in legs]), c["Q"])
            means += (K[..., -1].mean(-1) + torch.tensor([x[2] for x in legs], dtype=torch.float64, device="cuda")).tolist()
        best = int(np.argmin(means[1:]))
        if means[1 + best] < means[0]:
            tour = cand[1 + best]
        trace.append(min(means[0], means[1 + best]))
    f = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
    return {"trace": f(trace), "accepted": None, "tour": None, "means": f(means)}


def _exact_plan(c, s):
    ns, S = s["ns"], c["S"]
    toff = np.concatenate([[0], np.cumsum(ns[:-1], dtype=np.int64)])
    costs = torch.empty((c["B"], S), dtype=torch.float64, device="cuda")
    order = np.argsort(-ns, kind="stable")
    k = 0
    while k < len(order):  # tours of like length together, padded to the longest
        N = int(ns[order[k]])
        group = order[k:k + max(1, 60_000_000 // (S * N))]
        k += len(group)
        q = torch.zeros((len(group), S, N), dtype=torch.int64, device="cuda")
        a = torch.zeros((len(group), N), dtype=torch.float64, device="cuda")
        ce = torch.zeros_like(a)
        Ds = []
        for j, b in enumerate(group):
            n = int(ns[b])
            t = s["tours"][toff[b]:toff[b] + n]
            x = torch.from_numpy(s["xys"][b]).cuda()
            a[j, :n], ce[j, :n], D = _legs(x, t)
            Ds.append(D)
            q[j, :, :n] = s["dem"][s["off"][b]:s["off"][b] + n * S].view(S, n).long()[:, t.long() - 1]
        K = _split64(q, a, ce, c["Q"])
        for j, b in enumerate(group):
            costs[b] = K[j, :, int(ns[b])] + Ds[j]
    return {"costs": costs, "means": costs.mean(1)}


def _exact_fleet(c, s):
    a, ce, D = _legs(s["xy"], s["tour"])
    cols, n, Q = s["tour"].long() - 1, c["n"], c["Q"]
    cost = []
    for lo, hi in _chunks(c["S"], max(64, 33_000_000 // n)):
        q = s["dem"][lo:hi].long()[:, cols].clamp(min=0)
        L = torch.zeros((hi - lo, n + 1), dtype=torch.int64, device="cuda")
        torch.cumsum(q, 1, out=L[:, 1:])
        wmax = max(_windows(L, Q))
        K = torch.full((hi - lo, n + 1), math.inf, dtype=torch.float64, device="cuda")
        K[:, 0] = 0.0
        best = torch.full((hi - lo,), math.inf, dtype=torch.float64, device="cuda")
        closed = [(L[:, j:] - L[:, :n + 1 - j]) > Q for j in range(1, wmax + 1)]
        for _ in range(c["K"]):
            psi = K[:, :n] + a
            new = torch.full_like(K, math.inf)
            for j in range(1, min(wmax, n) + 1):  # p = i - j
                torch.minimum(new[:, j:], psi[:, :n + 1 - j].masked_fill(closed[j - 1], math.inf), out=new[:, j:])
            new[:, 1:] += ce
            K = new
            best = torch.minimum(best, K[:, n])
        cost.append(best + D)
    cost = torch.cat(cost)
    return {"cost": cost, "nroutes": None, "route": None, "mean": cost.mean()}


def _exact_reinsert(c, s):
    T, U, K = c["T"], c["U"], c["K"]
    unit = float(np.float32(c["unit"]))
    states = torch.arange(U + 1, device="cuda")
    refill = U - states
    value, value0 = [], []
    for lo, hi in _chunks(c["S"], 60_000_000 // (U + 1)):
        d = s["cons"][lo:hi].long().clamp(min=0)
        C = torch.zeros((hi - lo, U + 1), dtype=torch.float64, device="cuda")

        def after(j, C):  # end-of-day cost and cost-to-go of the inventory j left
            if s["table"] is not None:
                e = s["table"].double()[j.clamp(min=0)]
            else:
                e = torch.where(j >= 0, j * 1.0, j * -20.0)
            return e + C.gather(1, j.clamp(min=0))

        for t in range(T - 1, -1, -1):
            none = after(states[None, :] - d[:, t:t + 1], C)
            full = after(U - d[:, t:t + 1], C)
            if K:
                fee = torch.full_like(none, math.inf)
                for r in range(K):
                    fits = s["rcap"][lo:hi, t, r:r + 1] >= refill
                    fee = torch.where(fits, torch.minimum(fee, s["rcost"][t, r].double()), fee)
            else:
                fee = s["fixed"][t].double()
            deliver = fee + unit * refill + full
            C = torch.where(refill > 0, torch.minimum(none, deliver), none)
        value.append(C[:, U // 2].clone())
        value0.append(C if c["value0"] else None)
    value = torch.cat(value)
    return {"value": value, "policy": None, "value0": torch.cat(value0) if c["value0"] else None, "mean": value.mean()}


def exact(case, seed):
    c, op = case, case["op"]
    s = _inputs(c, seed)
    if op == "split":
        cost, _ = _exact_split(c, s)
        return {"cost": cost, "pred": None, "mean": cost.mean()}
    if op == "gradient":
        cost, counts = _exact_split(c, s, s["dist"])
        n, t = c["n"], s["tour"].long()
        g = torch.zeros((n + 1, n + 1), dtype=torch.float64, device="cuda")
        g[0, t], g[t, 0] = counts[0], counts[1]
        g[t[:-1], t[1:]] = c["S"] - counts[1][:-1]
        return {"mean": cost.mean(), "grad": g / c["S"]}
    if op == "fleet":
        return _exact_fleet(c, s)
    if op == "plan":
        return _exact_plan(c, s)
    if op == "search":
        return _exact_search(c, s, seed)
    return _exact_reinsert(c, s)
