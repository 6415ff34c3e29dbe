"""The canonical list delivered into pinned memory is the device list on both
sides of the size where it starts to be streamed in buckets (8.4 M pairs) and
with several buckets."""
import numpy as np
import pytest
import torch

import population as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,buckets", [(3700, 1), (4300, 2), (5300, 3)])
def test_host_list_equals_device_list_in_buckets(n, buckets):
    import paper_1901_10475_gb300 as scd
    torch.cuda.set_device(0)
    sc = scd.Scene(P.catalog_mixture(n, seed=44), 86400.0, 1.0).build_boxes()
    want = sc.find_pairs_device().cpu()
    assert max(1, len(want) >> 22) == buckets
    out = torch.full((len(want) + 3, 4), -7, dtype=torch.int32).pin_memory()
    host = out.numpy().view(scd.PAIR_DTYPE).reshape(-1)
    for _ in range(2):
        out.fill_(-7)
        assert scd.scd_find_pairs_into(sc.handle, host) == len(want)
        assert torch.equal(out[:-3], want) and (out[-3:] == -7).all()
    sc.close()
