"""Where memory is short, a split step's scratch is given back: also one that is not in
use, and for the transforms of the elasticity."""
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


def test_scratch_of_a_step_not_in_use_makes_room():
    # the split step's scratch stays when a fused variant is chosen, until memory is short
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=3, N=2, NM=1, nx=64, ny=40, nz=24, seed=4)
    out = []
    for bounded in (False, True):
        alloc = _bounded()
        sim = Simulation(p, dtype="f64", allocator=alloc)
        tiles = sim.tiles()
        sim.set_launch([i for i, t in enumerate(tiles) if t[2] == 0][0])
        if bounded:
            alloc.limit = alloc.used
        sim.set_fields(p.phi0, p.mu0)
        sim.enable_checkpoints(8)
        sim.step(6)
        out.append(sim.get_fields())
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_elastic_transforms_get_the_scratch_back():
    # turned on where the memory holds the fields and the transforms' work area only
    # without the FP64 cell list
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=3, N=2, NM=1, nx=263, ny=30, nz=24, bc=[3, 3, 3], seed=4)   # (a large prime in x: needs a work area)
    C = np.zeros((6, 6))
    C[:3, :3] = 0.6
    C[range(3), range(3)] = 1.0
    C[range(3, 6), range(3, 6)] = 0.4
    eig = np.zeros((2, 3, 3))
    eig[0] = 0.01 * np.eye(3)
    free = _bounded()
    sim = Simulation(p, dtype="f64", allocator=free)
    before = free.used
    sim.update_params(elastic_C=C, eigenstrain=eig)
    fields = 263 * 30 * 24 * 8 + 132 * 30 * 24 * 16
    assert free.used > before + fields   # the work area comes on top, from the same allocator
    top = free.used
    sim.set_fields(p.phi0, p.mu0)
    sim.step(3)
    want = sim.get_fields()
    sim.close()
    alloc = _bounded()
    sim = Simulation(p, dtype="f64", allocator=alloc)
    alloc.limit = top - 1   # one byte short of all of it together
    sim.update_params(elastic_C=C, eigenstrain=eig)
    assert sim.tiles()[sim.launch()[0]][2] == 0
    sim.set_fields(p.phi0, p.mu0)
    sim.step(3)
    got = sim.get_fields()
    sim.close()
    assert np.abs(want[0] - got[0]).max() <= 3 * 32 * 2.0 ** -52
    assert np.abs(want[1] - got[1]).max() <= 3 * 32 * 2.0 ** -52
