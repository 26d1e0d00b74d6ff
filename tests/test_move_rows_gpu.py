"""Moves on tours at the edges of the rows they are costed in: line counts
around the lane groups' sizes and the 128 lines of a row, more than 32 orders
a tour, moves whose plans come in any order, and few
moves (a warp's lanes partly idle).  Deltas and status against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_moves_gpu import check, gpu_moves
from test_parity_gpu import make_instance

pytestmark = pytest.mark.gpu

TOURS = [0, 1, 2, 15, 16, 17, 31, 32, 33, 60, 63, 64, 65, 66, 96, 126, 127, 128, 129, 130, 190, 300] + [50] * 8


def instance(rng, lay, n_plans, n_sku, sizes=(1,)):
    """Plans with tours of about the given line counts, of orders of the given sizes."""
    orders, need = [], sum(TOURS)
    while need > 0:
        k = int(rng.choice(sizes))
        orders.append(rng.choice(n_sku, k, replace=False).tolist())
        need -= k
    plans = []
    for _ in range(n_plans):
        perm, tours, i = rng.permutation(len(orders)).tolist(), [], 0
        for lines in rng.permutation(TOURS).tolist():
            tour, have = [], 0
            while have < lines and i < len(perm):
                tour.append(perm[i])
                have += len(orders[perm[i]])
                i += 1
            tours.append(tour)
        plans.append(tours + [perm[i:]])
    return make_instance(lay, orders, rng.permutation(lay.n_loc)[:n_sku].astype(np.int32), plans, n_sku)


def random_moves(rng, inst, n):
    kind = rng.integers(0, 4, n)
    n_t = int(inst.plan_tour_off[1])
    a = np.where(kind < 2, rng.integers(0, inst.n_orders, n), rng.choice(inst.line_sku, n))
    b = np.where(kind == 0, rng.integers(0, inst.n_orders, n), np.where(kind == 1, rng.integers(0, n_t, n),
                                                                       rng.integers(0, inst.n_sku, n)))
    b = np.where(kind == 3, rng.integers(0, inst.layout.n_loc, n), b)
    return np.stack([kind, a, b, rng.integers(0, inst.n_plans, n)], 1).astype(np.int32)


@pytest.mark.parametrize("n", [3, 70, 1500])
@pytest.mark.parametrize("lay", [wh_gen.Layout(23, 31), wh_gen.Layout(280, 9, 4, 2, 6)], ids=["narrow", "wide"])
@pytest.mark.parametrize("own", [True, False])
def test_moves(gpu_lib, own, lay, n):
    rng = np.random.default_rng(n)
    inst = instance(rng, lay, 4, 600, (1, 1, 2, 9) if n == 70 else (1,))
    maps = np.stack([rng.permutation(lay.n_loc)[:600] for _ in range(4)]).astype(np.int32) if own else None
    s, st = check(gpu_lib, inst, random_moves(rng, inst, n), maps=maps)
    assert st == 0 and (n < 70 or (s == 0).sum() > n // 4)


def test_unusable_location(gpu_lib):
    """A SKU without a usable location: exactly the moves whose changed tours hold it score status 3."""
    rng = np.random.default_rng(4)
    inst = instance(rng, wh_gen.Layout(23, 31), 2, 600)
    maps = np.stack([rng.permutation(inst.layout.n_loc)[:600] for _ in range(2)]).astype(np.int32)
    sku = int(inst.line_sku[5])
    mv = random_moves(rng, inst, 600)
    mv = mv[(mv[:, 0] < 2)]
    want_d, want_s = oracle.eval_moves(inst, mv, 0, 0, slot_map=maps.ravel(), slot_map_stride=inst.n_sku)
    broken = maps.copy()
    broken[:, sku] = inst.layout.n_loc
    d, s, _ = gpu_moves(gpu_lib, inst, mv, maps=broken, occupancy=False)
    holders = set(np.nonzero(inst.line_sku == sku)[0].tolist())   # one line an order
    tour_of = {}
    for p in range(2):
        for t in range(inst.plan_tour_off[p], inst.plan_tour_off[p + 1]):
            for o in inst.order_seq[inst.tour_off[t]:inst.tour_off[t + 1]]:
                tour_of[p, int(o)] = t
    for m, (kind, a, b, p) in enumerate(mv.tolist()):
        ta = tour_of[p, a]
        tb = tour_of[p, b] if kind == 0 else inst.plan_tour_off[p] + b
        held = want_s[m] == 0 and any(tour_of[p, o] in (ta, tb) for o in holders)
        if held:
            assert s[m] == 3 and (d[m] == 0).all()
        else:
            assert s[m] == want_s[m] and (d[m] == want_d[m]).all()
    assert (s == 3).sum() > 0 and (s == 0).sum() > 100
