"""The implicit 8-wide tree at the sizes where it can go wrong: box counts at
and beside whole nodes and whole levels, cells that start and end inside
nodes, nodes that span more ticks than a frame has cells, and boxes whose
faces are not finite.  The pair list equals the oracle's on the same FP32
boxes, exactly."""
import numpy as np
import pytest
import torch

import oracle as O
import population as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scd():
    import paper_1901_10475_gb300 as m
    torch.cuda.set_device(0)
    return m


def _check(sc):
    got = sc.find_pairs()
    lo, hi, obj = (x.cpu().numpy() for x in sc.boxes())
    want = O.canonicalize(O.raw_cells_sweep(lo, hi, obj.view(np.uint32)))
    assert np.array_equal(got.view(np.int32).reshape(-1, 4), want.view(np.int32).reshape(-1, 4))
    return got


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 63, 64, 65, 511, 512, 513, 4095, 4097])
@pytest.mark.parametrize("curve", [dict(), dict(morton_bits=8), dict(morton_bits=16, space_warp=1)])
def test_box_counts_at_node_and_level_edges(scd, n, curve):
    els = P.uniform_leo(n, seed=900 + n, radius_km=400.0)
    pol = scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=100)  # one box per object
    sc = scd.Scene(els, 10.0, 1.0, pol, tuning=curve).build_boxes()
    got = _check(sc)
    assert n < 63 or len(got) > 0
    sc.close()


def test_scenes_that_start_and_end_inside_nodes(scd):
    sizes = [1, 8, 9, 2, 65, 1, 1, 512, 7, 70]
    scenes = [P.uniform_leo(m, seed=950 + k, radius_km=400.0) for k, m in enumerate(sizes)]
    hz = [600.0 + 60.0 * k for k in range(len(sizes))]
    pol = scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=60)
    b = scd.BatchScene(scenes, hz, 1.0, pol).build_boxes()
    got = b.find_pairs_per_scene()
    for els, h, g in zip(scenes, hz, got):
        one = scd.Scene(els, h, 1.0, pol).build_boxes()
        assert np.array_equal(_check(one).view(np.int32), np.ascontiguousarray(g).view(np.int32))
        one.close()
    assert sum(map(len, got)) > 0
    b.close()


@pytest.mark.parametrize("step", [1, 50, 700])
def test_consecutive_segments_in_wide_frames(scd, step):
    # few objects over a long horizon: nodes that span up to thousands of ticks
    els = P.uniform_leo(6, seed=970, radius_km=900.0)
    pol = scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=step)
    sc = scd.Scene(els, 6000.0, 1.0, pol).build_boxes()
    assert len(_check(sc)) > 0
    sc.close()


def test_boxes_with_faces_that_are_not_finite(scd):
    els = P.uniform_leo(200, seed=980, radius_km=300.0)
    els[::40, 0] = 1e200  # their faces overflow FP32
    els[::40, 1] = 0.0  # (circular: an eccentric orbit of this size is refused)
    pol = scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=20)
    sc = scd.Scene(els, 600.0, 1.0, pol).build_boxes()
    hi = sc.boxes()[1].cpu().numpy()
    assert not np.isfinite(hi).all()
    assert len(_check(sc)) > 0
    sc.close()
