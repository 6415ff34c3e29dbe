"""Narrow phase over lists too short to keep a warp busy, whose long intervals
are split over its lanes: every candidate's first witness and witness count
equal the oracle's tick-by-tick ones, with either output left out."""
import numpy as np
import pytest
import torch

import oracle as O
import population as P

pytestmark = pytest.mark.gpu

T = 9000


def _elements():
    els = P.uniform_leo(12, seed=1300, radius_km=60.0)
    els[1] = els[0]            # twins: a witness at every tick
    els[3] = els[2]
    els[3, 4] += 0.02          # a slow chase: in and out of reach
    els[4, 1] = 0.6            # eccentric, above the starter's switch
    els[4, 0] = 30000.0
    els[5] = els[4]
    els[5, 5] += 0.004
    els[6, 1] = 0.0
    return els


@pytest.mark.parametrize("m", [1, 2, 31, 33, 64, 300])
def test_split_intervals_against_oracle(m):
    import paper_1901_10475_gb300 as scd
    torch.cuda.set_device(0)
    els = _elements()
    g = np.random.Generator(np.random.Philox(1301 + m))
    c = np.zeros((m, 4), np.int32)
    pairs = [(i, j) for i in range(12) for j in range(i + 1, 12)]
    pick = [(0, 1), (2, 3), (4, 5)] + [pairs[k] for k in g.integers(0, len(pairs), m)]
    for q in range(m):
        c[q, :2] = pick[q]
        lo = int(g.integers(0, T // 2)) if q % 3 else 0
        c[q, 2:] = lo, (T if q % 2 == 0 else int(g.integers(lo, T + 1)))
    of, oc, om, _ = O.narrow_phase(els, c.view(O.CELL_DTYPE).reshape(-1), 1.0)
    sure = om > 2e-6  # the oracle's distances stay off r_i + r_j
    assert sure.sum() >= m - 2
    sc = scd.Scene(els, float(T), 1.0).build_boxes()
    d = torch.as_tensor(c, device="cuda")
    first, count, _ = sc.narrow_phase(d)
    assert (first.cpu().numpy()[sure] == of[sure]).all()
    assert (count.cpu().numpy().view(np.uint32)[sure] == oc[sure]).all()
    only = torch.full((m,), 7, dtype=torch.int32, device="cuda")
    scd.scd_narrow_phase(sc.handle, d.data_ptr(), m, only.data_ptr(), 0)
    assert torch.equal(only, first)
    scd.scd_narrow_phase(sc.handle, d.data_ptr(), m, 0, only.data_ptr())
    assert torch.equal(only, count)
    sc.close()
