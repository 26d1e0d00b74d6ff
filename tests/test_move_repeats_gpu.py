"""SKU moves of SKUs that an order asks for on several of its lines: a
tour's picks are a set, so the order counts once.  Deltas and status against
the oracle, and the search's costs kept current against a full evaluation."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_moves_gpu import check
from test_parity_gpu import gpu_eval, make_instance

pytestmark = pytest.mark.gpu


def instance(rng, lay, n_plans, n_sku):
    """Orders of a few SKUs, most of them asked for again and again: around a warp's lines, and far beyond them."""
    sizes = np.concatenate([rng.integers(1, 9, 150), [31, 32, 33, 40, 64, 65, 97, 150, 260]])
    orders = [rng.integers(0, n_sku, max(1, k // 2))[rng.integers(0, max(1, k // 2), k)].tolist() for k in sizes]
    orders[0], orders[1] = [3, 3], [3, 5, 3, 5, 5]
    plans = []
    for _ in range(n_plans):
        perm = rng.permutation(len(orders)).tolist()
        plans.append([perm[i:i + 7] for i in range(0, len(perm), 7)])
    return make_instance(lay, orders, np.zeros(n_sku, np.int32), plans, n_sku)


def sku_moves(rng, inst, n):
    kind = rng.integers(2, 4, n)
    a = rng.choice(inst.line_sku, n)
    b = np.where(kind == 2, rng.choice(inst.line_sku, n), rng.integers(0, inst.layout.n_loc, n))
    mv = np.stack([kind, a, b, rng.integers(0, inst.n_plans, n)], 1)
    mv[:2] = [[2, 3, 5, 0], [2, 5, 3, 1]]
    return mv.astype(np.int32)


@pytest.mark.parametrize("lay", [wh_gen.Layout(23, 31), wh_gen.Layout(280, 9, 4, 2, 6)], ids=["narrow", "wide"])
def test_repeated_lines(gpu_lib, lay):
    rng = np.random.default_rng(1)
    inst = instance(rng, lay, 3, 80)
    maps = np.stack([rng.permutation(lay.n_loc)[:80] for _ in range(3)]).astype(np.int32)
    s, st = check(gpu_lib, inst, sku_moves(rng, inst, 900), maps=maps)
    assert st == 0 and (s == 0).sum() > 600


@pytest.mark.parametrize("screened", [False, True])
def test_search_keeps_costs(gpu_lib, screened):
    """After local-search steps over such moves the kept costs are those of the plans as they are then."""
    import torch
    import paper_2110_13693_gb300 as wh
    from paper_2110_13693_gb300 import search
    rng, lay = np.random.default_rng(2), wh_gen.Layout(23, 31)
    inst = instance(rng, lay, 3, 80)
    maps = np.stack([rng.permutation(lay.n_loc)[:80] for _ in range(3)]).astype(np.int32)
    h = wh.Layout.of(lay)
    prob = wh.to_device(inst, slot_map=maps.ravel(), slot_map_stride=80)
    h.occupancy(prob)
    costs = wh.evaluate(h, prob)
    sg = wh.Surrogate(0) if screened else None
    for _ in range(6):
        mv = sku_moves(rng, inst, 3 * 40)
        mv[:, 3] = np.repeat(np.arange(3), 40)
        mv = torch.as_tensor(mv).cuda()
        if screened:
            search.screened_step(h, sg, prob, costs, mv, 40, 8, 0, 0)
        else:
            h.ls_step(prob, costs, mv, 40)
    torch.cuda.synchronize()
    assert h.status() == 0
    inst.slot_map = prob.slot_map.cpu().numpy()
    want = oracle.eval_plans(inst, slot_map=inst.slot_map, slot_map_stride=80)
    for g, w in zip((costs.tour_s, costs.tour_rr, costs.plan_s, costs.plan_rr), want):
        assert np.array_equal(g[:w.size].cpu().numpy(), w)
    h.close()
