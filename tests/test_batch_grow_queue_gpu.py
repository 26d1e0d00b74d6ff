"""Batch formation where a growth step has more candidates than its queue
holds: every order adds two picks to the tour, each cheap alone (what bounds
its length) and dear together, so all of them are bounded below the first one
scored.  Tour by tour against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_batch_grow_edges_gpu import check

pytestmark = pytest.mark.gpu

QUEUE = 1024   # candidates queued by a step; more are scored in place


def orders(lay, rng, n, seeds):
    """`seeds` orders of six far picks, the longest alone, among n orders of a pick in one of aisles 2 .. 5 and one in
    6 .. 9, their depths alike."""
    near = [[lay.loc(int(a), int(j), int(s)), lay.loc(int(b), int(k), int(t))] for a, b, j, k, s, t in
            zip(rng.integers(2, 6, n), rng.integers(6, 10, n), rng.integers(8, 15, n), rng.integers(8, 15, n),
                rng.integers(0, 2, n), rng.integers(0, 2, n))]
    far = [[lay.loc(19, 3 + k + i) for i in range(6)] for k in range(seeds)]
    return [(near + far)[i] for i in rng.permutation(n + seeds)]


@pytest.mark.parametrize("n", [1100, 1500])
def test_queue_overflows(gpu_lib, n):
    lay, rng = wh_gen.Layout(20, 60), np.random.default_rng(n)
    book = orders(lay, rng, n, 12)
    # the premise, by the oracle: a seed's tour with every candidate, and with either of its picks alone
    far, near = next(o for o in book if len(o) > 2), [o for o in book if len(o) == 2]
    tours = [far + o for o in near] + [far + o[:1] for o in near] + [far + o[1:] for o in near]
    cut = np.concatenate([[0], np.cumsum([len(t) for t in tours])]).astype(np.int32)
    one = np.arange(len(tours) + 1, dtype=np.int32)
    alone = wh_gen.Instance(lay, lay.n_loc, cut, np.concatenate(tours).astype(np.int32),
                            np.arange(lay.n_loc, dtype=np.int32), np.asarray([0, len(tours)], np.int32), one, one[:-1])
    cost = oracle.eval_plans(alone)[1].reshape(3, -1)
    assert np.maximum(cost[1], cost[2]).max() < cost[0].min() < cost[0].max() and len(near) > QUEUE + 12 * 2
    off = np.concatenate([[0], np.cumsum([len(o) for o in book])]).astype(np.int32)
    # 10 lines: a seed takes two of the others and no other seed
    check(gpu_lib, lay, off, np.concatenate(book).astype(np.int32), np.arange(lay.n_loc, dtype=np.int32), 0, 10)
