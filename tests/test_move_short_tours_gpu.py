"""Moves on tours of few orders, which every lane walks by itself, around the
numbers of orders where the lanes take a tour together: few moves (four tours
a warp) and many (32).  Deltas and status against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_moves_gpu import gpu_moves
from test_parity_gpu import make_instance

pytestmark = pytest.mark.gpu

N_SKU = 300


def instance(rng, lay, per, n_plans=3):
    """Orders of 0 .. 9 lines, one SKU on many of them and on some twice, `per` orders a tour, and an empty tour."""
    orders = [rng.integers(0, N_SKU, k).tolist() for k in rng.integers(0, 10, 240)]
    for k in range(0, 240, 5):
        orders[k] += [7] * (1 + k % 2)
    plans = []
    for _ in range(n_plans):
        perm = rng.permutation(len(orders)).tolist()
        plans.append([perm[i:i + per] for i in range(0, len(perm), per)] + [[]])
    return make_instance(lay, orders, np.zeros(N_SKU, np.int32), plans, N_SKU)


def moves(rng, inst, n):
    kind = np.arange(n) % 4
    n_t = int(inst.plan_tour_off[1])
    a = np.where(kind < 2, rng.integers(0, inst.n_orders, n), rng.integers(0, inst.n_sku, n))
    b = np.choose(kind, [rng.integers(0, inst.n_orders, n), rng.integers(0, n_t, n), rng.integers(0, inst.n_sku, n),
                         rng.integers(0, inst.layout.n_loc, n)])
    mv = np.stack([kind, a, b, rng.integers(0, inst.n_plans, n)], 1).astype(np.int32)
    mv[2], mv[6], mv[5] = [2, 7, 30, 0], [2, 31, 7, 1], [1, mv[5, 1], n_t - 1, 0]
    return mv


COPIES = (1, 500)   # of the moves: four tours a warp and 32


@pytest.mark.parametrize("per", [1, 2, 3, 20, 21, 22])
@pytest.mark.parametrize("lay", [wh_gen.Layout(23, 31), wh_gen.Layout(280, 9, 4, 2, 6)], ids=["narrow", "wide"])
def test_short_tours(gpu_lib, lay, per):
    rng = np.random.default_rng(per)
    inst = instance(rng, lay, per)
    maps = np.stack([rng.permutation(lay.n_loc)[:N_SKU] for _ in range(3)]).astype(np.int32)
    mv = moves(rng, inst, 240)
    want_d, want_s = oracle.eval_moves(inst, mv, 0, 0, slot_map=maps.ravel(), slot_map_stride=N_SKU)
    assert (want_s == 0).sum() > 150
    for copies in COPIES:
        d, s, st = gpu_moves(gpu_lib, inst, np.tile(mv, (copies, 1)), maps=maps)
        assert st == 0
        assert np.array_equal(s, np.tile(want_s, copies)) and np.array_equal(d, np.tile(want_d, (copies, 1)))


def test_unusable_lines(gpu_lib):
    """A line without a usable location gives status 3 to the moves that rewrite its tour, and to no others."""
    rng, lay = np.random.default_rng(9), wh_gen.Layout(23, 31)
    inst = instance(rng, lay, 2)
    maps = np.stack([rng.permutation(lay.n_loc)[:N_SKU] for _ in range(3)]).astype(np.int32)
    mv = moves(rng, inst, 240)
    mv = mv[mv[:, 0] < 2]
    want_d, want_s = oracle.eval_moves(inst, mv, 0, 0, slot_map=maps.ravel(), slot_map_stride=N_SKU)
    maps[1, 40] = lay.n_loc
    bad = {k for k in range(inst.n_orders) if 40 in inst.line_sku[inst.order_off[k]:inst.order_off[k + 1]]}
    tour_of = {(p, int(o)): t for p in range(3) for t in range(inst.plan_tour_off[p], inst.plan_tour_off[p + 1])
               for o in inst.order_seq[inst.tour_off[t]:inst.tour_off[t + 1]]}
    for m, (kind, a, b, p) in enumerate(mv.tolist()):
        if want_s[m] or p != 1:
            continue
        changed = {tour_of[p, a], tour_of[p, b] if kind == 0 else int(inst.plan_tour_off[p]) + b}
        if any(tour_of[1, o] in changed for o in bad):
            want_s[m], want_d[m] = 3, 0
    assert (want_s == 3).sum() > 0
    for copies in COPIES:
        d, s, _ = gpu_moves(gpu_lib, inst, np.tile(mv, (copies, 1)), maps=maps, occupancy=False)
        assert np.array_equal(s, np.tile(want_s, copies)) and np.array_equal(d, np.tile(want_d, (copies, 1)))
