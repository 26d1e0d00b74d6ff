"""Order ids that the short-tour kernel has not looked at when it hands a tour to the long-tour pass."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_parity_gpu import gpu_eval, make_instance

pytestmark = pytest.mark.gpu


def test_bad_order_behind_the_short_limit(gpu_lib):
    """An order id out of range behind the 64th line of a tour: flagged, the tour's costs -1."""
    import paper_2110_13693_gb300 as wh
    lay = wh_gen.Layout(20, 30)
    orders = [[(7 * i + j) % lay.n_loc for j in range(20)] for i in range(12)]
    plans = [[[0, 1, 2, 3, 4], [5, 6], [7, 8, 9, 10, 11]]]
    inst = make_instance(lay, orders, np.arange(lay.n_loc, dtype=np.int32), plans)
    want = oracle.eval_plans(inst)
    inst.order_seq[4] = 1 << 20
    got = gpu_eval(gpu_lib, inst)
    assert got[4] == wh.WH_STATUS_BAD_ORDER
    for g, w in zip(got[:2], want[:2]):
        assert g[0] == -1 and np.array_equal(g[1:], w[1:])
