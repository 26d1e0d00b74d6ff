"""S-shape costs from packed per-order records: the widest and deepest layouts
that pack and the first that do not, the largest packed order book and one
order more, empty orders and tours, and unusable ids; against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_parity_gpu import gpu_eval, make_instance

pytestmark = pytest.mark.gpu


def instance(lay, n_orders, seed, n_plans=2):
    rng = np.random.default_rng(seed)
    n_sku = min(lay.n_loc, 3000)
    orders = [rng.integers(0, n_sku, k).tolist() for k in rng.integers(0, 5, n_orders)]
    orders[0] = [n_sku - 1, 0]
    slot = rng.permutation(lay.n_loc)[:n_sku].astype(np.int32)
    slot[n_sku - 1], slot[np.nonzero(slot == lay.n_loc - 1)[0]] = lay.n_loc - 1, slot[n_sku - 1]   # the last slot
    plans = []
    for _ in range(n_plans):
        perm, tours, i = rng.permutation(n_orders).tolist(), [[]], 0
        while i < n_orders:
            k = int(rng.integers(1, 30))
            tours.append(perm[i:i + k])
            i += k
        plans.append(tours)
    return make_instance(lay, orders, slot, plans, n_sku)


def same(got, want):
    assert got[4] == 0
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[2], want[2])
    assert (got[1] == -7).all() and (got[3] == -7).all()


@pytest.mark.parametrize("A,L,n_orders", [(50, 256, 700), (51, 256, 700), (50, 257, 700), (1, 1, 40), (33, 100, 1),
                                          (32, 40, 12288), (32, 40, 12289)])
def test_layouts_and_books(gpu_lib, A, L, n_orders):
    inst = instance(wh_gen.Layout(A, L), n_orders, A + L)
    same(gpu_eval(gpu_lib, inst, mask=1, prefill=-7), oracle.eval_plans(inst))


def test_unusable_ids(gpu_lib):
    import paper_2110_13693_gb300 as wh
    lay = wh_gen.Layout(50, 256)
    good = instance(lay, 300, 9)
    want = oracle.eval_plans(good)[0]
    owner = np.zeros(good.order_seq.size, np.int64)
    for t in range(good.n_tours):
        owner[good.tour_off[t]:good.tour_off[t + 1]] = t

    def check(inst, bit, tours):
        got = gpu_eval(gpu_lib, inst, mask=1)
        w = want.copy()
        w[sorted(tours)] = -1
        assert got[4] == bit and np.array_equal(got[0], w)

    inst = instance(lay, 300, 9)
    inst.order_seq[100] = 300
    check(inst, wh.WH_STATUS_BAD_ORDER, {owner[100]})
    inst = instance(lay, 300, 9)
    line = int(inst.order_off[77 + int(np.argmax(np.diff(inst.order_off)[77:] > 0))])
    order = int(np.searchsorted(inst.order_off, line, side="right") - 1)
    inst.line_sku[line] = inst.n_sku
    check(inst, wh.WH_STATUS_BAD_SKU, {int(owner[q]) for q in np.nonzero(inst.order_seq == order)[0]})
