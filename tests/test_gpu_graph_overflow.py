"""A replayed find whose records outgrow the sizes it was captured for emits
nothing from the holes among its first slots, ends, and is run again."""
import numpy as np
import pytest
import torch

import oracle as O
import population as P

pytestmark = pytest.mark.gpu


def _dense(n, seed):
    """Objects on one orbit within 0.02 rad: most pairs meet all the time."""
    els = P.uniform_leo(n, seed=seed, radius_km=50.0)
    spread = els[:, 5].copy() / (2 * np.pi)
    els[:, :5] = els[0, :5]
    els[:, 5] = 0.02 * spread
    return els


@pytest.mark.parametrize("decomp", [None, (2, 0, 3)])
def test_records_past_the_captured_capacity(decomp):
    import paper_1901_10475_gb300 as scd
    torch.cuda.set_device(0)
    n, T = 600, 600
    pol = scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=100)  # the same boxes a scene
    sparse, dense = P.uniform_leo(n, seed=91, radius_km=5.0), _dense(n, 92)
    g = scd.Scene(sparse, float(T), 1.0, pol, tuning=dict(use_graph=1)).build_boxes()
    g.find_pairs_device(decomp)
    g.find_pairs_device(decomp)
    assert g.metrics()["graph"] == 2
    for els in (dense, dense, sparse):
        g.set_elements(els)
        g.build_boxes()
        got = g.find_pairs(decomp).view(np.int32).reshape(-1, 4)
        lo, hi, obj = (x.cpu().numpy() for x in g.boxes())
        want = O.canonicalize(O.raw_cells_sweep(lo, hi, obj.view(np.uint32)))
        want = want.view(np.int32).reshape(-1, 4)
        assert np.array_equal(got, want)
        if els is dense:  # starts and ends both past the first capacity, 65,536 slots
            assert (want[:, 3] - want[:, 2] > 100).sum() > 65536
    g.close()
