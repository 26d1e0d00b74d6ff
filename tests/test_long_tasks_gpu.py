"""Moves whose changed tours all have more than a row's 128 lines: from a task
a warp to more than 32 (a warp's matrix of records filled and filled again),
tours of fewer and of more aisles than the matrix holds, SKUs that are in
many of a tour's orders.  Deltas and status against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_moves_gpu import gpu_moves, long_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lay", [wh_gen.Layout(30, 5), wh_gen.Layout(300, 4), wh_gen.Layout(60, 3)],
                         ids=["few_aisles", "many_aisles", "around_the_matrix"])
def test_long_tasks(gpu_lib, lay):
    rng = np.random.default_rng(lay.n_aisles)
    inst = long_instance(lay, 5, per_tour=16)
    lines = inst.tour_lines()
    assert (lines > 128).mean() > 0.9
    inst.line_sku[rng.random(inst.n_lines) < 0.1] = 7      # one SKU in most orders, in some of them twice
    maps = np.stack([rng.permutation(lay.n_loc)[:inst.n_sku] for _ in range(3)]).astype(np.int32)
    n = 150
    kind = np.arange(n) % 3
    a = np.where(kind < 2, rng.integers(0, inst.n_orders, n), rng.integers(0, inst.n_sku, n))
    b = np.where(kind == 0, rng.integers(0, inst.n_orders, n),
                 np.where(kind == 1, rng.integers(0, inst.plan_tour_off[1], n), rng.integers(0, inst.n_sku, n)))
    mv = np.stack([kind, a, b, rng.integers(0, 3, n)], 1).astype(np.int32)
    mv[2], mv[5] = [2, 7, 11, 0], [2, 12, 7, 1]
    want_d, want_s = oracle.eval_moves(inst, mv, 0, 0, slot_map=maps.ravel(), slot_map_stride=inst.n_sku)
    assert (want_s == 0).sum() > n // 2
    for copies in (1, 120):
        d, s, st = gpu_moves(gpu_lib, inst, np.tile(mv, (copies, 1)), maps=maps)
        assert st == 0
        assert np.array_equal(s, np.tile(want_s, copies))
        assert np.array_equal(d, np.tile(want_d, (copies, 1)))
