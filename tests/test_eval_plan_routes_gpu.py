"""Which kernel a plan evaluation goes to, and its results on either side of
the rule's lines, every plan with a slotting of its own or all with one: all
tours against wh_eval_plans_noalloc (always k_eval_short), a sample of the
plans against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen

pytestmark = pytest.mark.gpu

K16, K32 = wh_gen.Layout(30, 30), wh_gen.Layout(301, 23, 4, 3, 6)
N_SKU = 700


def instance(rng, lay, n_orders, lines, n_plans, held, per):
    """Plans that hold `held` of the orders (1 .. 2 * lines - 1 lines each), `per` a tour; per: one number, or one a plan."""
    sizes = rng.integers(1, 2 * lines, n_orders)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    seq = np.argsort(rng.random((n_plans, n_orders)), axis=1)[:, :held].astype(np.int32)
    ends = [np.minimum(np.arange(0, held + p, p)[1:], held) for p in np.broadcast_to(per, n_plans)]
    pto = np.concatenate([[0], np.cumsum([e.size for e in ends])]).astype(np.int32)
    to = np.concatenate([[0]] + [e + k * held for k, e in enumerate(ends)]).astype(np.int32)
    return wh_gen.Instance(lay, N_SKU, off, rng.integers(0, N_SKU, off[-1]).astype(np.int32),
                           rng.permutation(lay.n_loc)[:N_SKU].astype(np.int32), pto, to, seq.ravel())


# (layout, own slottings, orders, mean lines, plans, orders held, orders a tour, kernel)
LONG_AND_SHORT = [2 if k % 8 == 3 else 24 for k in range(700)]
CASES = {
    "an_order_a_tour": (K32, True, 1000, 3, 16, 1000, 1, "k_eval_short"),
    "an_order_a_tour_16": (K16, True, 1000, 3, 16, 1000, 1, "k_eval_short"),
    "part_of_the_book": (K32, True, 2500, 3, 700, 128, 2, "k_eval_short"),
    "part_of_the_book_shared": (K32, False, 2500, 3, 700, 128, 2, "k_eval_short"),
    "few_tours_many_plans": (K32, True, 300, 3, 640, 300, 10, "k_eval_short"),
    "few_tours_many_plans_16": (K16, True, 300, 3, 640, 300, 10, "k_eval_short"),
    "large_book": (K32, True, 4700, 3, 20, 4700, 20, "k_eval_short"),
    "large_book_16": (K16, True, 4700, 3, 20, 4700, 20, "k_eval_short"),
    "lists_of_512": (K32, True, 640, 4, 700, 640, 9, "k_eval_plan"),
    "lists_of_512_16": (K16, True, 640, 4, 700, 640, 9, "k_eval_plan"),
    "lists_of_512_shared": (K32, False, 640, 4, 700, 640, 9, "k_eval_plan"),
    "lists_of_1024": (K32, True, 3000, 3, 500, 3000, 12, "k_eval_plan"),
    "lists_of_1024_16": (K16, True, 3000, 3, 500, 3000, 12, "k_eval_plan"),
    "lists_of_1024_shared": (K32, False, 3900, 3, 500, 3900, 13, "k_eval_plan"),
    "rounds": (K32, True, 2200, 4, 320, 2200, 2, "k_eval_plan"),
    "rounds_of_some_plans": (K32, True, 2200, 2, 700, 2200, LONG_AND_SHORT, "k_eval_plan"),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_routes(gpu_lib, case):
    import torch
    wh = gpu_lib
    lay, own, n_orders, lines, n_plans, held, per, kernel = CASES[case]
    rng = np.random.default_rng(len(case))
    inst = instance(rng, lay, n_orders, lines, n_plans, held, per)
    maps = np.argsort(rng.random((n_plans, lay.n_loc)), axis=1)[:, :N_SKU].astype(np.int32) if own else None
    stride = N_SKU if own else 0
    h = wh.Layout.of(lay)
    prob = wh.to_device(inst, slot_map=maps.ravel() if own else None, slot_map_stride=stride)
    got, general = (wh.alloc_costs(prob.n_tours, prob.n_plans) for _ in range(2))
    h.set_timing(True)
    h.eval_plans(prob, got, 3)
    ran = {k for k, v in h.timing().items() if v[0]}
    assert ran == {"k_prep", kernel, "k_eval_long"}
    assert h.status() == 0
    h.close()
    desc = wh.wh_layout_desc(lay.n_aisles, lay.slots_per_side, lay.aisle_pitch, lay.slot_pitch, lay.cross_aisle_width)
    wh.wh_eval_plans_noalloc(desc, prob.orders(), prob.plans(), 3, general.c())
    torch.cuda.synchronize()
    outs = [(g[:n].cpu().numpy(), w[:n].cpu().numpy()) for g, w, n in
            zip((got.tour_s, got.tour_rr, got.plan_s, got.plan_rr),
                (general.tour_s, general.tour_rr, general.plan_s, general.plan_rr),
                (prob.n_tours, prob.n_tours, n_plans, n_plans))]
    for g, w in outs:
        assert np.array_equal(g, w)
    some = np.unique(np.concatenate([[0, n_plans - 1], rng.choice(n_plans, min(n_plans, 12), replace=False)]))
    want = oracle.eval_plans(inst.subset_plans(some),
                             **(dict(slot_map=maps[some].ravel(), slot_map_stride=N_SKU) if own else {}))
    idx = np.concatenate([np.arange(inst.plan_tour_off[p], inst.plan_tour_off[p + 1]) for p in some])
    for (g, _), w, at in zip(outs, want, (idx, idx, some, some)):
        assert np.array_equal(g[at], w)
