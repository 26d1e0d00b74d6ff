"""wh_get_timing books every launch of a plan evaluation under the kernel that ran."""
import pytest

import wh_gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask,own,names", [(3, False, {"k_prep", "k_eval_short", "k_eval_long"}),
                                            (3, True, {"k_prep", "k_eval_plan", "k_eval_long"}),
                                            (1, True, {"k_prep", "k_eval_sshape"}),
                                            (1, False, {"k_prep", "k_eval_sshape"})])
def test_names(gpu_lib, mask, own, names):
    import numpy as np
    wh = gpu_lib
    inst = wh_gen.midsize(seed=3, n_plans=8)
    maps = np.tile(inst.slot_map, 8) if own else None
    lay = wh.Layout.of(inst.layout)
    prob = wh.to_device(inst, slot_map=maps, slot_map_stride=inst.n_sku if own else 0)
    costs = wh.alloc_costs(prob.n_tours, prob.n_plans)
    lay.set_timing(True)
    lay.eval_plans(prob, costs, mask)
    ran = {k: v[0] for k, v in lay.timing().items() if v[0]}
    lay.close()
    assert ran == dict.fromkeys(names, 1)
