"""A batch that cannot have the memory for a new work list keeps the one it has."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _bounded():
    from paper_2404_01035_gb300._binding import TorchAllocator

    class Bounded(TorchAllocator):
        limit, used = None, 0

        def __init__(self):
            super().__init__()
            self.sizes = {}

        def _do_alloc(self, nbytes, user):
            if self.limit is not None and self.used + int(nbytes) > self.limit:
                return None
            ptr = super()._do_alloc(nbytes, user)
            self.sizes[ptr] = int(nbytes)
            self.used += int(nbytes)
            return ptr

        def _do_free(self, ptr, user):
            self.used -= self.sizes.pop(ptr, 0)
            super()._do_free(ptr, user)
    return Bounded()


def test_a_batch_without_memory_for_a_new_list_keeps_its_own():
    from paper_2404_01035_gb300 import batch as B
    from paper_2404_01035_gb300._binding import MSError
    ps = [W.binary_problem(f"b{i}", 700, ny=640, delta=0.02, Delta=0.2, R=20.0) for i in range(2)]
    out = []
    alloc = _bounded()
    for bounded in (False, True):
        keep, B.TorchAllocator = B.TorchAllocator, (lambda: alloc) if bounded else B.TorchAllocator
        try:
            b = B.Batch(ps)
        finally:
            B.TorchAllocator = keep
        for i, p in enumerate(ps):
            b.set_fields(i, p.phi0, p.mu0)
        b.step(5)
        if bounded:
            alloc.limit = alloc.used
            with pytest.raises(MSError):
                b.set_tile(16)
            assert b.tile_height() == 8
        b.step(5)
        b.sync()
        out.append(b.get_fields(0))
        b.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
