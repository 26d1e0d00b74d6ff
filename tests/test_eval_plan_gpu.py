"""Plan evaluation by one CTA per plan (own slottings, layouts of 32-bit keys)
where its phases turn over: tours at the edges of the sort's lane groups and
of its 128 lines, plans of more tours than a round takes, orders taken twice,
order books without a line -> order table, unusable ids.  Whole numbers, bit
by bit against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_parity_gpu import assert_exact, gpu_eval, make_instance

pytestmark = pytest.mark.gpu

LAYOUTS = {"narrow": wh_gen.Layout(20, 30), "wide": wh_gen.Layout(301, 23, 4, 3, 6), "deep": wh_gen.Layout(17, 311)}


def one_line_orders(lay, rng, tours_of, n_plans, n_sku):
    """Plans over orders of one line each: every plan has tours of the given line counts, orders shuffled."""
    n = sum(tours_of)
    plans = []
    for _ in range(n_plans):
        perm = rng.permutation(n).tolist()
        cuts = np.concatenate([[0], np.cumsum(rng.permutation(tours_of))])
        plans.append([perm[a:b] for a, b in zip(cuts[:-1], cuts[1:])])
    return make_instance(lay, [[int(s)] for s in rng.integers(0, n_sku, n)], np.zeros(n_sku, np.int32), plans, n_sku)


def own_maps(lay, rng, n_plans, n_sku):
    return np.stack([rng.permutation(lay.n_loc)[:n_sku] for _ in range(n_plans)]).astype(np.int32).ravel()


@pytest.mark.parametrize("mask", [3, 2])
@pytest.mark.parametrize("name", sorted(LAYOUTS))
@pytest.mark.parametrize("shared", [False, True])
def test_line_counts(gpu_lib, name, shared, mask):
    lay, rng = LAYOUTS[name], np.random.default_rng(5)
    tours = [0, 1, 2, 3, 15, 16, 17, 31, 32, 33, 48, 63, 64, 65, 66, 80, 96, 97, 127, 128, 129, 200]
    tours += [40] * 50 + [70] * 9
    n_sku = min(lay.n_loc, 900)
    inst = one_line_orders(lay, rng, tours, 5, n_sku)
    if shared:
        inst.slot_map[:] = rng.permutation(lay.n_loc)[:n_sku]
        got = gpu_eval(gpu_lib, inst, mask=mask, prefill=0)
        want = oracle.eval_plans(inst)
    else:
        maps = own_maps(lay, rng, 5, n_sku)
        got = gpu_eval(gpu_lib, inst, mask=mask, slot_map=maps, stride=n_sku, prefill=0)
        want = oracle.eval_plans(inst, slot_map=maps, slot_map_stride=n_sku)
    assert got[4] == 0
    if mask == 2:
        want = (np.zeros_like(want[0]), want[1], np.zeros_like(want[2]), want[3])
    assert_exact(got, want)


@pytest.mark.parametrize("case", ["many_tours", "twice", "long_order", "some_orders", "empty"])
def test_plans(gpu_lib, case):
    lay, rng = LAYOUTS["wide"], np.random.default_rng(len(case))
    n_sku = 700
    sizes = rng.integers(0, 9, 2300)
    if case == "long_order":
        sizes[7] = 260
    orders = [rng.integers(0, n_sku, k).tolist() for k in sizes]
    plans = []
    for p in range(4):
        perm = rng.permutation(len(orders)).tolist()
        if case == "many_tours":   # more than 1,024, of uneven length
            cuts = np.sort(rng.choice(np.arange(1, len(perm)), 2101, replace=False)).tolist()
        elif case == "some_orders":
            perm = perm[:len(perm) // (p + 2)]
            cuts = list(range(8, len(perm), 8))
        else:
            cuts = list(range(9, len(perm), 9))
        plans.append([perm[a:b] for a, b in zip([0] + cuts, cuts + [len(perm)])])
    if case == "twice":
        plans[1][3] = plans[1][3] + plans[1][60][:2]     # in two tours
        plans[2][5] = plans[2][5] + [plans[2][5][0]]     # in one tour
    if case == "empty":
        plans[1] = []
        plans[2] = [[] for _ in range(40)]
    inst = make_instance(lay, orders, np.zeros(n_sku, np.int32), plans, n_sku)
    maps = own_maps(lay, rng, 4, n_sku)
    got = gpu_eval(gpu_lib, inst, slot_map=maps, stride=n_sku)
    assert got[4] == 0
    assert_exact(got, oracle.eval_plans(inst, slot_map=maps, slot_map_stride=n_sku))


def test_unusable_ids(gpu_lib):
    """Each unusable id is flagged and costs its tours -1; every other tour keeps its cost."""
    import paper_2110_13693_gb300 as wh
    lay, rng = LAYOUTS["narrow"], np.random.default_rng(2)
    n_sku = lay.n_loc
    orders = [rng.integers(0, n_sku - 1, 3).tolist() for _ in range(90)]
    plans = [[list(range(i, i + 9)) for i in range(0, 90, 9)] for _ in range(3)]
    maps = own_maps(lay, rng, 3, n_sku).reshape(3, n_sku)
    good = make_instance(lay, orders, np.zeros(n_sku, np.int32), plans, n_sku)
    want = oracle.eval_plans(good, slot_map=maps.ravel(), slot_map_stride=n_sku)

    def check(inst, m, bit, tours):
        got = gpu_eval(gpu_lib, inst, slot_map=m.ravel(), stride=n_sku)
        assert got[4] == bit
        for g, w in zip(got[:2], want[:2]):
            w = w.copy()
            w[tours] = -1
            assert np.array_equal(g, w)

    def fresh():
        return make_instance(lay, orders, np.zeros(n_sku, np.int32), plans, n_sku)

    inst = fresh()
    inst.order_seq[94] = 90
    check(inst, maps, wh.WH_STATUS_BAD_ORDER, [10])
    inst = fresh()
    inst.line_sku[3 * 13] = n_sku
    check(inst, maps, wh.WH_STATUS_BAD_SKU, [1, 11, 21])
    bad = maps.copy()
    bad[2, orders[50][1]] = lay.n_loc
    hit = [20 + k for k, t in enumerate(plans[2]) if any(orders[50][1] in orders[o] for o in t)]
    check(fresh(), bad, wh.WH_STATUS_BAD_LOC, hit)
    # a SKU out of every slotting that no order asks for is no fault
    bad = maps.copy()
    bad[:, n_sku - 1] = -5
    check(fresh(), bad, 0, [])
    inst = fresh()
    inst.order_off[31] = inst.n_lines + 7     # orders 30 and 31
    check(inst, maps, wh.WH_STATUS_BAD_OFFSET, [3, 13, 23])
