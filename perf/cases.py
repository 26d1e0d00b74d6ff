"""The evaluator's work as a user's program has it done, one call or step per case.

Every case is a dict of plain values.  ``prepare`` makes its inputs on the GPU
from the seed alone (order books, slottings and plans by the laws of the
benchmark's generator), ``run`` is one pass through the package's public entry
points, ``work`` the bytes and floating-point operations the path cannot do
without, and ``exact`` the floating-point outputs in 64 bits by plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2110_13693_gb300 as wh
from paper_2110_13693_gb300 import search

BOTH = wh.WH_ROUTE_SSHAPE | wh.WH_ROUTE_OPTIMAL

# Workload families.  A, L: aisles and slots per side; max_orders / max_lines:
# caps of a tour (0: none); chunks: tours are cut at random lengths up to
# max_orders; own: every plan has its own slotting.
TINY = dict(A=10, L=30, n_sku=600, n_orders=200, order_lines=5, geom=0.5, zipf=0.0, max_orders=8, max_lines=0,
            chunks=True)
MIDSIZE = dict(A=40, L=100, n_sku=8000, n_orders=4000, order_lines=12, geom=0.4, zipf=1.1, max_orders=20,
               max_lines=60, chunks=False)
PAPER = dict(A=500, L=200, n_sku=50000, n_orders=4000, order_lines=12, geom=0.4, zipf=1.0, max_orders=24,
             max_lines=0, chunks=False)


def listed():
    return [
        # a few dozen candidate plans of a small depot, rescored as they are edited: the smallest call
        dict(TINY, name="evaluate_small", kind="evaluate", n_plans=64, own=False, mask=BOTH),
        # a population of plans over one slotting, both routing rules
        dict(MIDSIZE, name="evaluate_population", kind="evaluate", n_plans=4096, own=False, mask=BOTH),
        # the same population under the S-shape rule alone (the picker's simple rule)
        dict(MIDSIZE, name="evaluate_sshape", kind="evaluate", n_plans=4096, own=False, mask=wh.WH_ROUTE_SSHAPE),
        # a population whose plans differ in slotting too, at the paper's scale (200,000 locations)
        dict(PAPER, name="evaluate_own_slottings", kind="evaluate", n_plans=8192, own=True, mask=BOTH),
        # many candidate warehouses of uneven size in one launch (the benchmark's headline, a quarter of it)
        dict(name="batch_of_warehouses", kind="batch", n_inst=256, n_plans=64, ids16=True),
        # a step of plain local search: 64 moves a plan scored exactly, the best applied
        dict(PAPER, name="search_step", kind="search", n_plans=4096, own=True, moves=64, relocations=False),
        # a step with the learned prescreen: 64 moves predicted, 4 scored exactly, the best applied
        dict(PAPER, name="screened_step", kind="screened", n_plans=4096, own=True, moves=64, keep=4),
        # every tour of a population predicted by the network: its features, then inference
        dict(PAPER, name="predict_tours", kind="predict", n_plans=2048, own=True),
        # training of the network: a few steps of 4,096 rows, then the weights read
        dict(name="train_network", kind="train", rows=4096, steps=16),
        # orders clustered into tours under many slottings
        dict(MIDSIZE, name="form_batches", kind="grow", n_maps=304),
        # products clustered and placed by co-occurrence and picking frequency
        dict(PAPER, name="kmeans_slotting", kind="kmeans", k=256, iters=20),
        # the pick sequences of the tours of a few chosen plans
        dict(PAPER, name="routes", kind="routes", n_plans=64, own=False),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _family(rng, max_loc, max_orders_in_book=5000):
    """A layout, catalogue and order book between the listed ones, odd sizes among them."""
    for _ in range(100):
        A, L = _log(rng, 8, 500), _log(rng, 20, 200)
        if 2 * A * L <= max_loc:
            break
    else:
        A, L = 40, 100
    n_sku = max(64, min(2 * A * L, int(2 * A * L * rng.choice([0.25, 0.6, 1.0])), 50000))
    cap, lines = rng.choice([(20, 60), (24, 0), (8, 0), (13, 41)])
    return dict(A=A, L=L, n_sku=n_sku, n_orders=_log(rng, 100, max_orders_in_book), order_lines=12, geom=0.4,
                zipf=rng.choice([0.0, 1.0, 1.1]), max_orders=cap, max_lines=lines, chunks=False)


def _plans(rng, c, lo, hi, own):
    """A number of plans that keeps the case within the listed ones' size."""
    most = min(hi, int(3.2e7 // c["n_orders"]))
    if own:
        most = min(most, int(4.0e8 // c["n_sku"]))
    return _log(rng, min(lo, most), most)


def draw(rng):
    kind = rng.choice(["evaluate", "evaluate", "evaluate", "batch", "search", "screened", "predict", "train", "grow",
                       "kmeans", "routes"])
    if kind == "batch":
        return dict(kind=kind, n_inst=_log(rng, 16, 256), n_plans=_log(rng, 8, 64), ids16=rng.random() < 0.7)
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 300, 4096), steps=rng.randint(2, 16))
    c = _family(rng, 200000)
    if kind not in ("evaluate", "routes") and c["max_lines"]:
        # tours cut by orders alone (their number is then the case's); moves may still have a line cap
        c["move_lines"], c["max_lines"] = rng.choice([0, 90]), 0
    if kind == "evaluate":
        own = rng.random() < 0.4
        return dict(c, kind=kind, n_plans=_plans(rng, c, 16, 8192, own), own=own, mask=rng.choice([1, 2, 3, 3]))
    if kind == "search":
        return dict(c, kind=kind, n_plans=_plans(rng, c, 16, 4096, True), own=True, moves=rng.randint(16, 64),
                    relocations=rng.random() < 0.5)
    if kind == "screened":
        m = rng.randint(16, 64)
        return dict(c, kind=kind, n_plans=_plans(rng, c, 16, 4096, True), own=True, moves=m,
                    keep=search.keep_count(m))
    if kind == "predict":
        own = rng.random() < 0.7
        return dict(c, kind=kind, n_plans=_plans(rng, c, 16, 2048, own), own=own)
    if kind == "grow":
        c = _family(rng, 20000, 3000)
        c["A"] = min(c["A"], 200)
        c["n_sku"] = min(c["n_sku"], 2 * c["A"] * c["L"])
        return dict(c, kind=kind, n_maps=_log(rng, 1, 152))
    if kind == "kmeans":
        return dict(c, kind=kind, k=min(_log(rng, 8, 256), c["n_sku"]), iters=rng.randint(5, 20))
    own = rng.random() < 0.3
    return dict(c, kind=kind, n_plans=_plans(rng, c, 1, 64, own), own=own)


# ------------------------------------------------------------------- inputs

def _rand(g, *shape, dtype=torch.float32):
    return torch.rand(*shape, device="cuda", generator=g, dtype=dtype)


def _order_book(g, n_orders, n_sku, order_lines, geom, zipf):
    """CSR order book: truncated geometric sizes, SKUs by popularity, distinct within an order."""
    w = (1.0 - geom) ** torch.arange(order_lines, device="cuda", dtype=torch.float64)
    cdf = torch.cumsum(w, 0) / w.sum()
    sizes = torch.clamp(torch.searchsorted(cdf, _rand(g, n_orders, dtype=torch.float64)) + 1, max=order_lines)
    off = torch.zeros(n_orders + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(sizes, 0)
    order = torch.repeat_interleave(torch.arange(n_orders, device="cuda"), sizes)
    n = int(order.numel())
    pop = torch.arange(1, n_sku + 1, device="cuda", dtype=torch.float64) ** -zipf
    pop = torch.cumsum(pop, 0) / pop.sum()
    sku = torch.clamp(torch.searchsorted(pop, _rand(g, n, dtype=torch.float64)), max=n_sku - 1)
    for _ in range(12):   # repeats within an order are drawn again
        key, at = torch.sort(order * n_sku + sku, stable=True)
        again = torch.zeros(n, dtype=torch.bool, device="cuda")
        again[at[1:]] = key[1:] == key[:-1]
        fresh = torch.clamp(torch.searchsorted(pop, _rand(g, n, dtype=torch.float64)), max=n_sku - 1)
        sku = torch.where(again, fresh, sku)
    return off.to(torch.int32), sku.to(torch.int32)


def _abc(A, L, n_sku):
    """SKU ranks on the locations nearest the depot (pitch 3, slot pitch 1, cross-aisle width 2)."""
    loc = torch.arange(2 * A * L, device="cuda")
    return torch.sort(loc // (2 * L) * 3 + 1 + loc % L, stable=True).indices[:n_sku].to(torch.int32)


def _swapped(g, base, n_maps):
    """n_maps slottings [n_maps, n_sku]: the base with a tenth of its SKUs in swapped places, others in each."""
    n = base.numel()
    pair = torch.randperm(n, device="cuda", generator=g)[:n // 2 * 2].view(2, -1)
    maps = base.repeat(n_maps, 1)
    for lo in range(0, n_maps, 1024):
        part = maps[lo:lo + 1024]
        a, b = part[:, pair[0]], part[:, pair[1]]
        swap = _rand(g, part.shape[0], pair.shape[1]) < 0.1
        part[:, pair[0]] = torch.where(swap, b, a)
        part[:, pair[1]] = torch.where(swap, a, b)
    return maps


def _cut(g, lines, n, max_orders, max_lines, chunks):
    """Tour ends [rounds, rows] of order sequences with line counts `lines` [rows, longest]; row r has n[r] orders."""
    rows = lines.shape[0]
    cum = torch.zeros(rows, lines.shape[1] + 1, dtype=torch.int32, device="cuda")
    cum[:, 1:] = torch.cumsum(lines, 1)
    pos, ends = torch.zeros(rows, dtype=torch.int64, device="cuda"), []
    while True:
        take = torch.randint(1, max_orders + 1, (rows,), device="cuda", generator=g) if chunks else max_orders
        nxt = torch.minimum(pos + take, n)
        if max_lines:
            full = cum.gather(1, pos[:, None]) + max_lines
            nxt = torch.minimum(nxt, torch.maximum(torch.searchsorted(cum, full, right=True)[:, 0] - 1, pos + 1))
        ends.append(nxt)
        pos = nxt
        if len(ends) % 8 == 0 and bool((pos >= n).all()):
            return torch.stack(ends)


def _plan_arrays(g, off, n_plans, max_orders, max_lines, chunks):
    """Random plans over one order book: (plan_tour_off, tour_off, order_seq), int32."""
    n = off.numel() - 1
    sizes = off[1:] - off[:-1]
    seq = torch.empty(n_plans, n, dtype=torch.int32, device="cuda")
    counts, ends = [], []
    for lo in range(0, n_plans, 4096):
        m = min(4096, n_plans - lo)
        part = torch.argsort(_rand(g, m, n), dim=1)
        seq[lo:lo + m] = part
        e = _cut(g, sizes[part], torch.full((m,), n, device="cuda"), max_orders, max_lines, chunks).t()
        new = torch.ones_like(e, dtype=torch.bool)
        new[:, 1:] = e[:, 1:] > e[:, :-1]
        counts.append(new.sum(1))
        ends.append((e + n * torch.arange(lo, lo + m, device="cuda")[:, None])[new])
    zero = torch.zeros(1, dtype=torch.int64, device="cuda")
    pto = torch.cat([zero, torch.cumsum(torch.cat(counts), 0)])
    return pto.to(torch.int32), torch.cat([zero] + ends).to(torch.int32), seq.view(-1)


def _problem(c, g, n_plans):
    off, sku = _order_book(g, c["n_orders"], c["n_sku"], c["order_lines"], c["geom"], c["zipf"])
    if c["zipf"] == 0.0:
        base = torch.randperm(2 * c["A"] * c["L"], device="cuda", generator=g)[:c["n_sku"]].to(torch.int32)
    else:
        base = _abc(c["A"], c["L"], c["n_sku"])
    own = c.get("own", False)
    maps = _swapped(g, base, n_plans if own else 1)
    pto, to, seq = _plan_arrays(g, off, n_plans, c["max_orders"], c["max_lines"], c["chunks"])
    return wh.DeviceProblem(off, sku, maps.view(-1), pto, to, seq, c["n_sku"], c["n_sku"] if own else 0)


def _moves(c, g, prob):
    """[n_plans * moves, 4] order swaps, relocations of orders and SKU swaps (or SKU relocations too)."""
    P, M = prob.n_plans, c["moves"]
    n = P * M

    def below(hi):
        return (_rand(g, n, dtype=torch.float64) * hi).long()

    plan = torch.arange(P, device="cuda").repeat_interleave(M)
    tours = (prob.plan_tour_off[1:] - prob.plan_tour_off[:-1])[plan]
    pool = torch.unique(prob.line_sku)
    kind = below(4 if c.get("relocations") else 3)
    a = torch.where(kind < 2, below(c["n_orders"]), pool[below(pool.numel())].long())
    b = torch.where(kind == 0, below(c["n_orders"]), torch.where(kind == 1, below(tours), below(c["n_sku"])))
    b = torch.where(kind == 3, below(2 * c["A"] * c["L"]), b)
    return torch.stack([kind, a, b, plan], 1).to(torch.int32)


def _params(seed):
    """Packed network parameters: Xavier-uniform weights, small biases."""
    r = np.random.default_rng(seed)

    def xavier(i, o):
        return r.uniform(-1.0, 1.0, (i, o)) * math.sqrt(6.0 / (i + o))

    return wh.pack_params(dict(w1=xavier(192, 256), b1=r.normal(0, 0.02, 256), w2=xavier(256, 256),
                               b2=r.normal(0, 0.02, 256), w3=xavier(256, 1), b3=r.normal(0, 0.02, 1)))


def _training_rows(c, g):
    """Feature rows like a population's tours (histogram counts and scaled scalars) and targets of order one."""
    n = c["rows"] * c["steps"]
    X = torch.poisson(_rand(g, n, 192) ** 4 * 1.5, generator=g)
    X[:, 128:131] = _rand(g, n, 3)
    X[:, 131] = torch.randint(20, 80, (n,), device="cuda", generator=g) / 64.0
    t = 0.5 + 0.3 * X[:, 129] + 0.05 * X[:, 132:].sum(1) / 6.0 + 0.02 * _rand(g, n)
    return X.to(torch.bfloat16), t


def _cost_buffers(c, n_tours, n_plans):
    """Output buffers that a program keeps for populations of this kind: room for more tours than this one has where
    their number differs from population to population."""
    room = n_tours
    if c["max_lines"] or c["chunks"]:
        room = int(1.6 * n_plans * _mean_tours(c)) + 64 * n_plans
        if n_tours > room:
            raise RuntimeError("more tours than the buffers have room for")
    return wh.Costs(*(torch.zeros(n, dtype=t, device="cuda") for n, t in ((room, torch.int32), (room, torch.int32),
                                                                         (n_plans, torch.int64), (n_plans, torch.int64))))


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    c, kind = dict(case), case["kind"]
    if kind == "train":
        sg = wh.Surrogate(0)
        sg.set_params(_params(seed))
        X, t = _training_rows(c, g)
        return dict(c=c, sg=sg, X=X.view(c["steps"], c["rows"], 192), t=t.view(c["steps"], c["rows"]))
    if kind == "batch":
        return _batch(c, g)
    lay = wh.Layout(c["A"], c["L"])
    if kind == "grow":
        prob = _problem(c, g, 1)
        return dict(c=c, lay=lay, prob=prob, maps=_swapped(g, _abc(c["A"], c["L"], c["n_sku"]), c["n_maps"]))
    if kind == "kmeans":
        prob = _problem(c, g, 1)
        signs = (torch.randint(0, 2, (c["n_sku"], 32), device="cuda", generator=g) * 2 - 1).to(torch.int8)
        u = torch.randint(0, 1 << 62, (c["k"],), device="cuda", generator=g)
        return dict(c=c, lay=lay, prob=prob, signs=signs, u=u)
    prob = _problem(c, g, c["n_plans"])
    s = dict(c=c, lay=lay, prob=prob)
    if kind == "routes":
        # as many of the plans' tours as there are at least (none holds more than max_orders orders)
        s["tours"] = torch.arange(c["n_plans"] * max(1, c["n_orders"] // c["max_orders"]), dtype=torch.int32,
                                  device="cuda")
        return s
    if kind in ("predict", "screened"):
        s["sg"] = wh.Surrogate(0)
        s["sg"].set_params(_params(seed))
    if kind != "predict":
        s["costs"] = _cost_buffers(c, prob.n_tours, prob.n_plans)
    if kind in ("search", "screened"):
        if c.get("relocations"):
            lay.occupancy(prob)
        lay.eval_plans(prob, s["costs"], BOTH)
        s["moves"] = _moves(c, g, prob)
    if kind == "screened":
        s["cache"] = search.new_cache(prob)
    return s


def _batch(c, g):
    """Warehouses of uneven size: aisles U[8, 64], slots per side U[20, 200], orders U[100, 5000], SKUs = locations."""
    n_inst, n_plans = c["n_inst"], c["n_plans"]
    host = torch.Generator().manual_seed(g.initial_seed())
    r = torch.rand(n_inst, 3, generator=host)
    r[:, 2] = (torch.randperm(n_inst, generator=host) + r[:, 2]) / n_inst   # order books of all sizes
    dims = [(8 + int(x * 57), 20 + int(y * 181), 100 + int(z * 4900)) for x, y, z in r.tolist()]
    books = [_order_book(g, n, 2 * A * L, 12, 0.4, 1.1) for A, L, n in dims]
    n = torch.tensor([d[2] for d in dims], device="cuda").repeat_interleave(n_plans)
    longest = int(n.max())
    key = _rand(g, n_inst * n_plans, longest)
    key.masked_fill_(torch.arange(longest, device="cuda") >= n[:, None], 2.0)
    seq = torch.argsort(key, dim=1)
    del key
    lines = torch.zeros(n_inst, longest, dtype=torch.int32, device="cuda")
    for i, (off, _) in enumerate(books):
        lines[i, :dims[i][2]] = off[1:] - off[:-1]
    ends = _cut(g, lines.repeat_interleave(n_plans, 0).gather(1, seq), n, 20, 60, False).t()
    new = torch.ones_like(ends, dtype=torch.bool)
    new[:, 1:] = ends[:, 1:] > ends[:, :-1]
    counts = new.sum(1).view(n_inst, n_plans)
    zero = torch.zeros(1, dtype=torch.int64, device="cuda")
    # every warehouse's outputs in one array a rule, one part each
    per_inst = counts.sum(1).tolist()
    mean = dict(MIDSIZE, n_orders=2550)
    out = _cost_buffers(mean, sum(per_inst), n_inst * n_plans)
    items, t0 = [], 0
    for i, ((A, L, k), (off, sku)) in enumerate(zip(dims, books)):
        rows = slice(i * n_plans, (i + 1) * n_plans)
        pto = torch.cat([zero, torch.cumsum(counts[i], 0)]).to(torch.int32)
        to = (ends[rows] + k * torch.arange(n_plans, device="cuda")[:, None])[new[rows]]
        to = torch.cat([zero, to]).to(torch.int32)
        ids = seq[rows, :k].reshape(-1)
        slot = _swapped(g, _abc(A, L, 2 * A * L), 1).view(-1)
        prob = wh.DeviceProblem(off, sku, slot, pto, to, None if c["ids16"] else ids.to(torch.int32), 2 * A * L,
                                order_seq16=ids.to(torch.int16) if c["ids16"] else None)
        tours = slice(t0, t0 + per_inst[i])
        t0 += per_inst[i]
        items.append(((A, L, 3, 1, 2), prob, wh.Costs(out.tour_s[tours], out.tour_rr[tours], out.plan_s[rows],
                                                      out.plan_rr[rows])))
    batch = wh.Batch(items)
    batch.autotune(BOTH)
    return dict(c=c, batch=batch, items=items, out=[out.tour_s, out.tour_rr, out.plan_s, out.plan_rr])


# --------------------------------------------------------------------- pass

def _costs_of(s, mask):
    costs = s["costs"]
    out = []
    if mask & wh.WH_ROUTE_SSHAPE:
        out += [costs.tour_s, costs.plan_s]
    if mask & wh.WH_ROUTE_OPTIMAL:
        out += [costs.tour_rr, costs.plan_rr]
    return out


def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "evaluate":
        s["lay"].eval_plans(s["prob"], s["costs"], c["mask"])
        return _costs_of(s, c["mask"])
    if kind == "batch":
        s["batch"].eval(BOTH, graph=True)
        return s["out"]
    if kind == "search":
        applied = search.plain_step(s["lay"], s["prob"], s["costs"], s["moves"], c["moves"], c["max_orders"],
                                    c.get("move_lines", 0))
        p = s["prob"]
        return [applied] + _costs_of(s, BOTH) + [p.tour_off, p.order_seq, p.slot_map]
    if kind == "screened":
        applied = search.screened_step(s["lay"], s["sg"], s["prob"], s["costs"], s["moves"], c["moves"], c["keep"],
                                       c["max_orders"], c.get("move_lines", 0), s["cache"])
        p = s["prob"]
        return [applied] + _costs_of(s, BOTH) + [p.tour_off, p.order_seq, p.slot_map, s["cache"][0]]
    if kind == "predict":
        X = wh.features(s["lay"], s["prob"])
        return [X, s["sg"].predict(X)]
    if kind == "train":
        losses = [s["sg"].train_step(s["X"][i], s["t"][i], 2e-3) for i in range(c["steps"])]
        params, grads = s["sg"].params()
        return losses + [params, grads]
    if kind == "grow":
        return list(s["lay"].batch_grow(s["prob"], s["maps"], c["max_orders"], c["max_lines"]))
    if kind == "kmeans":
        return list(s["lay"].kmeans_slotting(s["prob"], s["signs"], c["k"], c["iters"], u=s["u"]))
    return list(s["lay"].routes(s["prob"], s["tours"]))


# --------------------------------------------------------------------- work

def _mean_lines(c):
    w = [(1.0 - c["geom"]) ** k for k in range(c["order_lines"])]
    return sum((k + 1) * v for k, v in enumerate(w)) / sum(w)


def _mean_tours(c):
    """Tours a plan is cut into, about."""
    per = (c["max_orders"] + 1) / 2 if c["chunks"] else c["max_orders"]
    if c["max_lines"]:
        per = min(per, max(1.0, c["max_lines"] / _mean_lines(c)))
    return c["n_orders"] / per


def _inputs(c, n_plans):
    """Bytes of the order book, the plans and the slottings' entries that its lines name, each once."""
    lines = c["n_orders"] * _mean_lines(c)
    maps = n_plans if c.get("own") else 1
    return 4 * (c["n_orders"] + lines) + n_plans * 4 * (c["n_orders"] + _mean_tours(c)) + \
        maps * 4 * min(c["n_sku"], lines)


MLP_FLOPS = 2 * (192 * 256 + 256 * 256 + 256)


def work(case):
    c, kind = case, case["kind"]
    if kind == "train":
        n = c["rows"] * c["steps"]
        return {"bytes": n * (192 * 2 + 4) + 2 * 4 * wh.WH_MLP_NPARAM, "flops": 3 * MLP_FLOPS * n}
    if kind == "batch":
        plans = c["n_inst"] * c["n_plans"]   # 2,550 orders a plan, mean, in tours of about 19.7
        return {"bytes": plans * (2550 * (2 if c["ids16"] else 4) + 2550 / 19.7 * 12 + 16) + c["n_inst"] * 80000,
                "flops": 0}
    tours = _mean_tours(c)
    lines = c["n_orders"] * _mean_lines(c)
    if kind == "evaluate":
        rules = 2 if c["mask"] == BOTH else 1
        return {"bytes": _inputs(c, c["n_plans"]) + rules * c["n_plans"] * (4 * tours + 8), "flops": 0}
    if kind in ("search", "screened"):
        # the plans and the moves read, both costs of the changed tours read, every plan's outcome written
        n = c["n_plans"]
        b = _inputs(c, n) + n * c["moves"] * 16 + n * (16 * 2 + 4) + n * tours * 8
        tasks = n * c["moves"] * 1.6
        return {"bytes": b, "flops": MLP_FLOPS * tasks if kind == "screened" else 0}
    if kind == "predict":
        n = c["n_plans"] * tours
        return {"bytes": _inputs(c, c["n_plans"]) + n * (384 + 4), "flops": MLP_FLOPS * n}
    if kind == "grow":
        return {"bytes": 4 * (c["n_orders"] + lines) + c["n_maps"] * (4 * min(c["n_sku"], lines) + 8 * c["n_orders"]),
                "flops": 0}
    if kind == "kmeans":
        # every round compares every SKU with every centroid (and a seed with every SKU)
        ops = 2 * 32 * c["n_sku"] * c["k"] * (c["iters"] + 2)
        return {"bytes": 4 * (c["n_orders"] + lines) + c["n_sku"] * (32 + 128 + 8) + c["k"] * 136, "flops": ops}
    return {"bytes": _inputs(c, c["n_plans"]) + c["n_plans"] * (8 * tours + 4 * lines), "flops": 0}


# -------------------------------------------------------------------- exact

def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _unpacked(seed):
    p = torch.from_numpy(np.asarray(_params(seed), np.float64)).cuda()
    at, out = 0, []
    for shape in ((192, 256), (256,), (256, 256), (256,), (256,), (1,)):
        n = math.prod(shape)
        out.append(p[at:at + n].reshape(shape).clone())
        at += n
    return out


def _exact_features(c, g):
    """The 192 features of every tour in 64 bits, from the inputs alone."""
    p = _problem(c, g, c["n_plans"])
    A, L = c["A"], c["L"]
    sizes = (p.order_off[1:] - p.order_off[:-1]).long()
    per_tour = (p.tour_off[1:] - p.tour_off[:-1]).long()
    n = per_tour.numel()
    F = torch.zeros(n, 192, dtype=torch.float64, device="cuda")
    tour_of = torch.repeat_interleave(torch.arange(n, device="cuda"), per_tour)
    per_plan = (p.plan_tour_off[1:] - p.plan_tour_off[:-1]).long()
    plan_of = torch.repeat_interleave(torch.arange(p.n_plans, device="cuda"), per_plan)
    step = 1 << 22
    book = p.order_off.long()
    cuts = list(range(0, tour_of.numel(), step)) + [tour_of.numel()]
    lo_all, hi_all = [], []
    keys = []
    for q0, q1 in zip(cuts[:-1], cuts[1:]):
        o = p.order_seq[q0:q1].long()
        k = sizes[o]
        t = torch.repeat_interleave(tour_of[q0:q1], k)
        first = torch.repeat_interleave(book[o] - (torch.cumsum(k, 0) - k), k)
        sku = p.line_sku[first + torch.arange(t.numel(), device="cuda")].long()
        loc = p.slot_map[plan_of[t] * p.slot_map_stride + sku].long()
        F[:, 131].index_add_(0, t, torch.ones(t.numel(), dtype=torch.float64, device="cuda"))
        key, at = torch.unique(t * A + loc // (2 * L), return_inverse=True)
        slot = loc % L
        lo = torch.full((key.numel(),), L, device="cuda").scatter_reduce_(0, at, slot, "amin")
        hi = torch.full((key.numel(),), -1, device="cuda").scatter_reduce_(0, at, slot, "amax")
        keys.append(key), lo_all.append(lo), hi_all.append(hi)
    # a tour that spans two parts has its aisles in both
    key, at = torch.unique(torch.cat(keys), return_inverse=True)
    lo = torch.full((key.numel(),), L, device="cuda").scatter_reduce_(0, at, torch.cat(lo_all), "amin")
    hi = torch.full((key.numel(),), -1, device="cuda").scatter_reduce_(0, at, torch.cat(hi_all), "amax")
    t, a = key // A, key % A
    one = torch.ones(key.numel(), dtype=torch.float64, device="cuda")
    flat = F.view(-1)
    flat.index_add_(0, t * 192 + hi * 64 // L, one)
    flat.index_add_(0, t * 192 + 64 + lo * 64 // L, one)
    flat.index_add_(0, t * 192 + 132 + a * 60 // A, one)
    visits = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, t, torch.ones_like(t))
    left = torch.full((n,), A, device="cuda").scatter_reduce_(0, t, a, "amin")
    right = torch.full((n,), -1, device="cuda").scatter_reduce_(0, t, a, "amax")
    F[:, 128], F[:, 129], F[:, 130] = left / A, right / A, visits / A
    F[:, 131] /= 64.0
    return F


def exact(case, seed):
    c = dict(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    if c["kind"] == "predict":
        F = _exact_features(c, g)
        w1, b1, w2, b2, w3, b3 = _unpacked(seed)
        y = torch.cat([_gelu(_gelu(f @ w1 + b1) @ w2 + b2) @ w3 + b3 for f in F.split(1 << 18)])
        return [F, y]
    if c["kind"] != "train":
        return None
    X, t = _training_rows(c, g)
    X, t = X.double().view(c["steps"], c["rows"], 192), t.double().view(c["steps"], c["rows"])
    P = [p.requires_grad_() for p in _unpacked(seed)]
    mo, ve = [torch.zeros_like(p) for p in P], [torch.zeros_like(p) for p in P]
    losses = []
    for k in range(c["steps"]):
        w1, b1, w2, b2, w3, b3 = P
        y = _gelu(_gelu(X[k] @ w1 + b1) @ w2 + b2) @ w3 + b3
        loss = 0.5 * ((y - t[k]) ** 2).mean()
        grads = torch.autograd.grad(loss, P)
        losses.append(loss.detach().reshape(1))
        with torch.no_grad():
            for p, m, v, d in zip(P, mo, ve, grads):
                m.mul_(0.9).add_(0.1 * d)
                v.mul_(0.999).add_(0.001 * d * d)
                p -= 2e-3 * (m / (1 - 0.9 ** (k + 1))) / (torch.sqrt(v / (1 - 0.999 ** (k + 1))) + 1e-8)

    def packed(v):
        return torch.cat([x.detach().reshape(-1) for x in v]).cpu().numpy()

    return losses + [packed(P), packed(grads)]
