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
