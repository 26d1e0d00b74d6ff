"""S-shape costs of order books around the sizes where an SM holds three and two
tables of packed records, in tours on both sides of the orders a tour that
packing takes then; against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_parity_gpu import gpu_eval

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orders", [9600, 9601, 12288])
@pytest.mark.parametrize("per", [1, 7, 8, 9])
def test_books(gpu_lib, n_orders, per):
    rng, lay, n_plans = np.random.default_rng(per), wh_gen.Layout(50, 256), 3
    off = np.concatenate([[0], np.cumsum(rng.integers(0, 4, n_orders))]).astype(np.int32)
    seq = np.argsort(rng.random((n_plans, n_orders)), axis=1).astype(np.int32).ravel()
    ends = np.minimum(np.arange(0, n_orders + per, per)[1:], n_orders)
    to = np.concatenate([[0]] + [ends + p * n_orders for p in range(n_plans)]).astype(np.int32)
    inst = wh_gen.Instance(lay, 2000, off, rng.integers(0, 2000, off[-1]).astype(np.int32),
                           rng.permutation(lay.n_loc)[:2000].astype(np.int32),
                           (np.arange(n_plans + 1) * ends.size).astype(np.int32), to, seq)
    got, want = gpu_eval(gpu_lib, inst, mask=1), oracle.eval_plans(inst)
    assert got[4] == 0 and np.array_equal(got[0], want[0]) and np.array_equal(got[2], want[2])
