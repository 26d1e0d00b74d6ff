"""Routes of tours with more lines than a gathering chunk of 256 but at most
256 distinct points: lines repeat points, within orders and across the chunks'
borders; and one point too many, found in a later chunk."""
import numpy as np
import pytest

import oracle
import wh_gen
from test_routes_gpu import check, run

pytestmark = pytest.mark.gpu


def book(lay, tours):
    """One plan; tours[i] a list of orders, each a list of locations."""
    orders = [o for t in tours for o in t]
    off = np.concatenate([[0], np.cumsum([len(o) for o in orders])]).astype(np.int32)
    lines = np.concatenate([np.asarray(o, np.int32) for o in orders])
    to = np.concatenate([[0], np.cumsum([len(t) for t in tours])]).astype(np.int32)
    return wh_gen.Instance(lay, lay.n_loc, off, lines, np.arange(lay.n_loc, dtype=np.int32),
                           np.array([0, len(tours)], np.int32), to, np.arange(len(orders), dtype=np.int32))


@pytest.mark.parametrize("n_lines", [255, 256, 257, 511, 513, 900])
def test_more_lines_than_points(gpu_lib, n_lines):
    lay = wh_gen.Layout(50, 30, 4, 2, 6)
    rng = np.random.default_rng(n_lines)
    pool = rng.choice(lay.n_loc, 200, replace=False)
    tours = []
    for per in (1, 7, 40, n_lines):
        locs = rng.choice(pool, n_lines)
        tours.append([locs[i:i + per].tolist() for i in range(0, n_lines, per)])
    check(gpu_lib, book(lay, tours), list(range(len(tours))))


def test_point_257_in_a_later_chunk(gpu_lib):
    lay = wh_gen.Layout(40, 20)
    front = [(a * 2) * 20 + k for a in range(40) for k in range(20)]   # one location per point
    many = front[:256]
    tours = [[many, many, [front[256]]], [many, many, [many[3]]]]
    pts, npt, length, st = run(gpu_lib, book(lay, tours), [0, 1])
    assert st == gpu_lib.WH_STATUS_TOUR_TOO_LONG
    assert npt.tolist() == [-1, 256] and length[0] == -1
    assert length[1] == oracle.rr(lay, many)
