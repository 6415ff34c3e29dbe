"""A captured find is not replayed once another call on its scene has moved the
buffers it was captured with."""
import numpy as np
import pytest
import torch

import population as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("other", ["decomposed", "raw"])
def test_plain_graph_after_another_find(other):
    import paper_1901_10475_gb300 as scd
    torch.cuda.set_device(0)
    els = P.catalog_mixture(n=900, seed=81, radius_km=25.0)
    pol = scd.make_step_policy(scd.SCD_STEP_PERIOD_FRACTION, period_fraction=100.0)
    eager = scd.Scene(els, 20000.0, 1.0, pol).build_boxes()
    want = eager.find_pairs()
    eager.close()
    g = scd.Scene(els, 20000.0, 1.0, pol, tuning=dict(use_graph=1)).build_boxes()
    for replayed in (False, True):
        assert np.array_equal(g.find_pairs(), want)
        g.find_pairs_device()
        assert g.metrics()["graph"] == 2
        if replayed:
            break
        if other == "raw":  # (never a graph) more cells than boxes: larger sort scratch
            assert len(g.find_raw_cells_device()) > g.metrics()["boxes"]
        else:               # more references than boxes: larger sorted boxes, links, tree
            g.set_tuning(dict(g.tuning(), use_graph=0))
            assert np.array_equal(g.find_pairs((2, 0, 16)), want)
            g.set_tuning(dict(g.tuning(), use_graph=1))
        g.find_pairs_device()
        assert g.metrics()["graph"] == 1  # captured anew
    g.close()
