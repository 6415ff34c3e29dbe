"""A screen of more than 2^30 boxes, where the tree has eleven levels and a
pending node takes 64 bits: the pairs among its first objects are those of a
screen of these objects alone, which stays below 2^30 boxes.  In a process of
its own, so that it has the device's memory and no earlier screen's records
per box as its guess."""
import os
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
def test_more_than_2_to_the_30_boxes():
    import torch
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 220e9:
        pytest.skip("needs 220 GB of free device memory")
    subprocess.run([sys.executable, os.path.abspath(__file__)], cwd=ROOT, timeout=300, check=True,
                   env=dict(os.environ, PYTHONPATH=ROOT))


def main():
    import torch

    import paper_1901_10475_gb300 as scd
    import population as P
    torch.cuda.set_device(0)
    T, ticks = (1 << 24) - 2, 16  # 2^20 boxes an object
    pol = scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=ticks)
    els = P.uniform_leo(1025, seed=4100)

    def pairs(n):
        sc = scd.Scene(els[:n], float(T), 1.0, pol, mode=1).build_boxes()  # INTERVAL boxes
        got = sc.find_pairs_device().cpu().numpy().view(np.int32).reshape(-1, 4).copy()
        assert sc.metrics()["boxes"] == n << 20
        sc.close()
        torch.cuda.empty_cache()
        return got

    whole, part = pairs(1025), pairs(1000)
    assert len(part) > 10000
    assert np.array_equal(whole[whole[:, 1] < 1000], part)


if __name__ == "__main__":
    main()
