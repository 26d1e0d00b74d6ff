"""Plan evaluation by one CTA per plan: tours that it hands to the long-tour
pass, the empty ones among them.  Whole numbers, bit by bit against the
oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_eval_plan_gpu import LAYOUTS, own_maps
from test_parity_gpu import assert_exact, gpu_eval, make_instance

pytestmark = pytest.mark.gpu


def cut(rng, n_orders, n_plans, per, empty=()):
    """Plans over all orders, shuffled, `per` orders a tour, with empty tours put in at the given places."""
    plans = []
    for _ in range(n_plans):
        perm = rng.permutation(n_orders).tolist()
        tours = [perm[i:i + per] for i in range(0, n_orders, per)]
        for k in empty:
            tours.insert(k, [])
        plans.append(tours)
    return plans


@pytest.mark.parametrize("case", ["twice", "long_order", "bad_offset"])
def test_empty_tours_beside_long_ones(gpu_lib, case):
    """A tour of no lines costs 0 also where its plan's tours go to the long-tour pass."""
    import paper_2110_13693_gb300 as wh
    lay, rng, n_sku = LAYOUTS["wide"], np.random.default_rng(7), 700
    sizes = rng.integers(1, 9, 400)
    if case == "long_order":
        sizes[7] = 260
    orders = [rng.integers(0, n_sku, k).tolist() for k in sizes]
    plans = cut(rng, len(orders), 3, 9, empty=(0, 1, 2, 3, 17, 48))
    if case == "twice":
        for plan in plans:
            plan[5] = plan[5] + plan[9][:2]
    maps = own_maps(lay, rng, 3, n_sku)
    inst = make_instance(lay, orders, np.zeros(n_sku, np.int32), plans, n_sku)
    want = oracle.eval_plans(inst, slot_map=maps, slot_map_stride=n_sku)
    if case == "bad_offset":
        inst.order_off[31] = inst.n_lines + 7     # orders 30 and 31
    got = gpu_eval(gpu_lib, inst, slot_map=maps, stride=n_sku, prefill=-9)
    if case != "bad_offset":
        assert got[4] == 0
        assert_exact(got, want)
        return
    assert got[4] == wh.WH_STATUS_BAD_OFFSET
    hit = np.asarray([any(o in (30, 31) for o in t) for plan in plans for t in plan])
    plan_of = np.repeat(np.arange(3), [len(p) for p in plans])
    for k in (0, 1):
        w = np.where(hit, -1, want[k])
        assert np.array_equal(got[k], w)
        assert np.array_equal(got[2 + k], np.bincount(plan_of, np.where(hit, 0, w)).astype(np.int64))


@pytest.mark.parametrize("own", [True, False])
@pytest.mark.parametrize("case", ["long_unused", "long_in_some", "empty_twice", "all_twice", "twice_in_one", "rows_full"])
def test_tours_handed_over_one_by_one(gpu_lib, case, own):
    """Orders of over 128 and over 255 lines, and orders taken twice: beside tours without them."""
    lay, rng, n_sku = LAYOUTS["wide"], np.random.default_rng(8), 700
    sizes = rng.integers(0, 9, 1500)
    sizes[[5, 6]] = 3
    if case.startswith("long"):
        sizes[[40, 41, 42, 43, 44]] = 128, 129, 254, 255, 900
    if case == "empty_twice":
        sizes[5] = 0
    orders = [rng.integers(0, n_sku, k).tolist() for k in sizes]
    plans = cut(rng, len(orders), 24, 9, empty=(4,))
    for k, plan in enumerate(plans):
        if case == "long_unused":
            plan[:] = [[o for o in t if o not in range(40, 45)] for t in plan]
        elif case in ("empty_twice", "twice_in_one"):
            a, b = (3, 3) if case == "twice_in_one" else (2 * k, 60)
            plan[a], plan[b] = plan[a] + [5], plan[b] + [5]
        elif case == "all_twice":
            plan[:] = plan + cut(rng, len(orders), 1, 9)[0]
        elif case == "rows_full":                          # the same orders over and over: more lines than the book has
            plan[:] = plan + [t[::-1] for t in plan[:120]] * 2
    inst = make_instance(lay, orders, rng.permutation(lay.n_loc)[:n_sku], plans, n_sku)
    maps = own_maps(lay, rng, len(plans), n_sku) if own else None
    got = gpu_eval(gpu_lib, inst, slot_map=maps, stride=n_sku if own else 0, prefill=-9)
    assert got[4] == 0
    assert_exact(got, oracle.eval_plans(inst, **(dict(slot_map=maps, slot_map_stride=n_sku) if own else {})))
