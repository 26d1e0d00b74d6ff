"""Plan offsets that do not cover the tours, or decrease: flagged, and every
tour is still scored once, under one plan.  Whole numbers, bit by bit against
the oracle on the offsets that stand for them."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_eval_plan_edges_gpu import cut
from test_eval_plan_gpu import own_maps
from test_parity_gpu import assert_exact, gpu_eval, make_instance

pytestmark = pytest.mark.gpu


# a CTA a plan, CTAs of several plans, those under a shared slotting
@pytest.mark.parametrize("n_plans,own", [(5, True), (700, True), (700, False)])
@pytest.mark.parametrize("case", ["first", "last", "decreasing", "outside"])
def test_malformed_plan_offsets(gpu_lib, case, own, n_plans):
    import paper_2110_13693_gb300 as wh
    lay, rng, n_sku = wh_gen.Layout(260, 4), np.random.default_rng(n_plans), 300
    orders = [rng.integers(0, n_sku, k).tolist() for k in rng.integers(1, 8, 512)]
    inst = make_instance(lay, orders, rng.permutation(lay.n_loc)[:n_sku], cut(rng, len(orders), n_plans, 8), n_sku)
    maps = own_maps(lay, rng, n_plans, n_sku) if own else None
    off = inst.plan_tour_off.copy()
    if case == "first":
        off[0] = 5
    elif case == "last":
        off[-2:] = off[-2] - 3, off[-1] - 20
    elif case == "decreasing":
        off[2] += 100                     # past the next one
        if n_plans > 5:
            off[300], off[690] = off[640], 7
    else:
        off[1], off[-1] = -4, off[-1] + 100
    # the offsets that stand for them: a tour belongs to the first plan that ends behind it, else to the last
    inst.plan_tour_off = np.clip(np.maximum.accumulate(np.concatenate([[0], off[1:-1], [inst.n_tours]])), 0,
                                 inst.n_tours).astype(np.int32)
    inst.plan_tour_off[-1] = inst.n_tours
    kw = dict(slot_map=maps, slot_map_stride=n_sku) if own else {}
    want = oracle.eval_plans(inst, **kw)
    inst.plan_tour_off = off.astype(np.int32)
    got = gpu_eval(gpu_lib, inst, slot_map=maps, stride=n_sku if own else 0, prefill=-9)
    assert got[4] == wh.WH_STATUS_BAD_OFFSET
    assert_exact(got, want)
