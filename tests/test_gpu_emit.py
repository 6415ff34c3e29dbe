"""The canonical list where a pair has many runs within a few ticks: the
record sorts leave out the lowest bits of the tick, and the pass that writes
the pairs ranks each group of runs that differ in those bits alone.  Groups
of 1 to some 30 runs over one and several tiles, with 1 to 8 bits left out."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T", [(40, 250), (40, 1000), (70, 500), (120, 1000), (250, 250),
                                 (250, 500), (250, 2100)])
def test_runs_a_few_ticks_apart(n, T):
    import paper_1901_10475_gb300 as scd
    torch.cuda.set_device(0)
    # coplanar circles with steps of 5 and 6 ticks: the boxes of a pair about
    # its range apart meet and part at every step
    els = np.zeros((n, 7))
    els[:, 0] = np.linspace(6900.0, 7600.0, n)
    els[:, 2], els[:, 3] = 0.9, 0.3
    els[:, 5] = 0.0002 * np.arange(n)
    els[:, 6] = 230.0
    pol = scd.make_step_policy(scd.SCD_STEP_PERIOD_FRACTION, period_fraction=1000.0)
    sc = scd.Scene(els, float(T), 1.0, pol).build_boxes()
    got = sc.find_pairs().view(np.int32).reshape(-1, 4)
    lo, hi, obj = (x.cpu().numpy() for x in sc.boxes())
    want = O.canonicalize(O.raw_cells_sweep(lo, hi, obj.view(np.uint32)))
    assert np.array_equal(got, want.view(np.int32).reshape(-1, 4))
    dev = sc.find_pairs_device()
    assert np.array_equal(dev.cpu().numpy().view(np.int32).reshape(-1, 4), got)
    same = (got[1:, :2] == got[:-1, :2]).all(1) & (got[1:, 2] - got[:-1, 2] < 16)
    assert same.sum() > 10
    sc.close()
