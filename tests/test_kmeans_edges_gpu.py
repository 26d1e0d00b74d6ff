"""K-means slotting at the edges of its parts, bit-exact with the oracle: no
ordered SKU at all, one SKU, SKU counts around the sort's tiles, clusters that
are no multiple of the threads of a row, pick counts of more than one byte, and
more ordered SKUs than one seeding cluster holds."""
import numpy as np
import pytest

import oracle
import wh_gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_sku,n_orders,lines,k,iters,fw,zipf", [
    (700, 0, 0, 5, 3, 64, 0.0),        # nothing ordered: every row is zero
    (1, 4, 1, 1, 2, 64, 0.0),
    (1023, 90, 5, 3, 4, 64, 0.0),
    (1025, 90, 5, 9, 4, 0, 0.0),
    (2048, 2500, 3, 31, 3, 256, 1.6),  # the most popular SKU picked over 1,000 times
    (40000, 30000, 1, 12, 2, 64, 0.0), # lines and SKUs beyond a cluster's shared memory
    (26000, 60000, 1, 6, 1, 64, 0.0),
])
def test_edges(gpu_lib, n_sku, n_orders, lines, k, iters, fw, zipf):
    import torch
    rng = np.random.default_rng(n_sku + k)
    p = (np.arange(n_sku) + 1.0) ** -zipf
    sku = rng.choice(n_sku, n_orders * lines, p=p / p.sum()).astype(np.int32)
    off = (np.arange(n_orders + 1) * lines).astype(np.int32)
    lay = wh_gen.Layout(max(1, (n_sku + 199) // 200), 100)
    signs = wh_gen.gen_signs(4, (n_sku, 32))
    u = rng.integers(0, 1 << 63, k, dtype=np.uint64)
    one = np.zeros(2, np.int32)
    inst = wh_gen.Instance(lay, n_sku, off, sku, np.zeros(n_sku, np.int32), one, one, np.zeros(0, np.int32))
    h = gpu_lib.Layout.of(lay)
    prob = gpu_lib.to_device(inst)
    if n_orders * lines == 0:
        prob.line_sku = torch.zeros(1, dtype=torch.int32, device="cuda")[:0]
    got = h.kmeans_slotting(prob, torch.as_tensor(signs).cuda(), k, iters, fw,
                            u=torch.as_tensor(u.view(np.int64)).cuda())
    torch.cuda.synchronize()
    assert h.status() == 0
    h.close()
    want = oracle.kmeans_slotting(lay, off, sku, n_sku, signs, fw, k, iters, u=u)
    for name, a, b in zip(("x", "seeds", "centroids", "assign", "slot_map"), got, want):
        assert np.array_equal(a.cpu().numpy(), b), name
