"""Batch formation where its lists turn over: orders of more lines than a warp
has lanes, tours of more aisles than that, order books around the block's
size, the largest layout the 16-bit keys allow, and more candidates in one
step than its queue holds; tour by tour against the oracle."""
import numpy as np
import pytest

import oracle
import wh_gen

pytestmark = pytest.mark.gpu


def book(rng, n_sku, sizes):
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    return off, rng.integers(0, n_sku, off[-1]).astype(np.int32)


def check(wh, lay, off, lines, slot, max_orders, max_lines):
    import torch
    one = np.zeros(2, np.int32)
    inst = wh_gen.Instance(lay, slot.size, off, lines, slot, one, one, np.zeros(0, np.int32))
    h = wh.Layout.of(lay)
    to, seq, nt = h.batch_grow(wh.to_device(inst), torch.as_tensor(slot[None]).cuda(), max_orders, max_lines)
    torch.cuda.synchronize()
    assert h.status() == 0
    h.close()
    wto, wseq = oracle.batch_grow(lay, off, lines, slot.size, slot, max_orders, max_lines)
    n = int(nt[0])
    assert n == len(wto) - 1
    assert np.array_equal(to[0, :n + 1].cpu().numpy(), wto)
    assert np.array_equal(seq[0].cpu().numpy(), wseq)


@pytest.mark.parametrize("case", ["long_orders", "one", "two", "wide", "largest_layout", "block_sized"])
def test_edges(gpu_lib, case):
    rng = np.random.default_rng(len(case))
    lay, caps = wh_gen.Layout(30, 40, 5, 2, 4), (6, 0)
    if case == "long_orders":
        sizes, caps = rng.integers(20, 90, 24), (4, 250)
    elif case == "one":
        sizes = np.array([7])
    elif case == "two":
        sizes = np.array([1, 2])
    elif case == "wide":
        lay, sizes, caps = wh_gen.Layout(120, 11), rng.integers(1, 14, 90), (0, 150)
    elif case == "largest_layout":
        lay, sizes, caps = wh_gen.Layout(255, 256), rng.integers(1, 9, 60), (0, 60)
    else:
        sizes, caps = rng.integers(0, 4, 513), (9, 11)
    off, lines = book(rng, lay.n_loc, sizes)
    slot = rng.permutation(lay.n_loc).astype(np.int32)
    check(gpu_lib, lay, off, lines, slot, *caps)


def test_more_candidates_than_the_queue(gpu_lib):
    """1,300 orders of the same two picks: every one is bounded below the
    first one scored, so a step's second round overflows its queue."""
    lay = wh_gen.Layout(12, 20)
    n = 1300
    off = np.arange(0, 2 * n + 1, 2, dtype=np.int32)
    lines = np.tile(np.array([lay.loc(3, 5), lay.loc(9, 12)], np.int32), n)
    check(gpu_lib, lay, off, lines, np.arange(lay.n_loc, dtype=np.int32), 3, 0)
