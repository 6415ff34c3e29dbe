"""A refinement that runs out of memory leaves no captured rounds behind that
point into buffers it gave back."""
import ctypes

import numpy as np
import pytest
import torch

import population as P

pytestmark = pytest.mark.gpu


class _KeepingAllocator:
    """Device memory from torch tensors, zeroed, kept alive when it is freed;
    requests of more than `limit` bytes fail."""

    def __init__(self, B):
        self.B, self.limit, self.blocks = B, None, []

        def _alloc(nbytes, stream, ctx):
            if self.limit is not None and nbytes > self.limit:
                return None
            t = torch.zeros(max(int(nbytes), 16), dtype=torch.uint8, device="cuda")
            self.blocks.append(t)
            return t.data_ptr()

        self.hooks = (B.ALLOC_FN(_alloc), B.FREE_FN(lambda ptr, stream, ctx: None))

    def __enter__(self):
        assert self.B.lib().scd_set_allocator(self.hooks[0], self.hooks[1], None) == 0
        return self

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        prev = self.B._torch_hooks
        self.B.lib().scd_set_allocator(*(prev or (self.B.ALLOC_FN(), self.B.FREE_FN())), None)


def test_replay_after_a_failed_call():
    import paper_1901_10475_gb300 as scd
    from paper_1901_10475_gb300 import _binding as B
    torch.cuda.set_device(0)
    n, T = 60, 900
    pol = scd.make_step_policy(scd.SCD_STEP_FIXED, fixed_ticks=10)
    few = P.uniform_leo(n, seed=17, radius_km=60.0)
    many = np.repeat(few[:1], n, axis=0)  # every pair meets in every tick: 1.6 M candidates
    many[:, 5] += np.arange(n) * 1e-6
    ref = scd.Scene(few, float(T), 1.0, pol).build_boxes()
    want = scd.scd_refine_witnesses(ref.handle)[0]
    ref.close()
    assert len(want) > 0
    with _KeepingAllocator(B) as mem:
        sc = scd.Scene(few, float(T), 1.0, pol).build_boxes()
        for _ in range(2):  # captured, replayed
            assert np.array_equal(scd.scd_refine_witnesses(sc.handle)[0], want)
        sc.set_elements(many)
        sc.build_boxes()
        mem.limit = 4 << 20  # the candidates, 2 x 1.6 M of 8 bytes, do not fit
        with pytest.raises(scd.ScdError):
            scd.scd_refine_witnesses(sc.handle)
        mem.limit = None
        sc.set_elements(few)
        sc.build_boxes()
        for _ in range(3):
            assert np.array_equal(scd.scd_refine_witnesses(sc.handle)[0], want)
        sc.close()
