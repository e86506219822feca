"""A context whose split step cannot have its scratch starts with, and is tuned
to, the fused step: creating and tuning succeed as they do without that variant."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _refusing(size):
    from paper_2404_01035_gb300._binding import TorchAllocator

    class Refusing(TorchAllocator):
        refused = 0

        def _do_alloc(self, nbytes, user):
            if int(nbytes) == size:
                self.refused += 1
                return None
            return super()._do_alloc(nbytes, user)
    return Refusing()


@pytest.mark.parametrize("dim,dtype,nx,ny,nz", [(3, "f64", 40, 21, 13), (3, "f32", 40, 21, 13), (2, "f32", 1300, 1000, 1)])
def test_starts_and_tunes_without_the_split_step(tmp_path, dim, dtype, nx, ny, nz):
    from paper_2404_01035_gb300 import Simulation
    N = 3 if dim == 3 else 2
    p = W.small_multiphase(n=8, dim=dim, N=N, NM=N - 1, nx=nx, ny=ny, nz=nz, seed=4)
    p = p.copy(G=p.G * 16.0 / max(ny, nz, 16))
    cells, segs = nx * ny * nz, -(-nx // 32)
    up = lambda b: -(-b // 256) * 256  # noqa: E731
    size = (up((cells + 2) * 4) + 2 * up(cells) + up(3 * N * cells * 8) + up((N - 1) ** 2 * cells * 8) if dtype == "f64"
            else 2 * (segs * ny * nz + 2) * 4)
    alloc = _refusing(size)
    sim = Simulation(p, dtype=dtype, allocator=alloc)
    assert alloc.refused == 1 and sim.tiles()[sim.launch()[0]][2] == 0
    sim.set_fields(p.phi0, p.mu0)
    cache = str(tmp_path / "tuned.json")
    sim.tune(cache, steps_per_trial=2)
    assert alloc.refused > 1 and sim.tiles()[sim.launch()[0]][2] == 0
    sim.step(3)
    got = sim.get_fields()
    sim.close()
    # a cache entry that names the split step, read where its scratch cannot be had
    sim = Simulation(p, dtype=dtype)
    split = [i for i, t in enumerate(sim.tiles()) if t[2] == 1][0]
    tx, ty = sim.tiles()[split][:2]
    sim.close()
    text = open(cache).read()
    import re
    text = re.sub(r'"tx": \d+, "ty": \d+, "split": 0', f'"tx": {tx}, "ty": {ty}, "split": 1', text)
    open(cache, "w").write(text)
    sim = Simulation(p, dtype=dtype, allocator=_refusing(size))
    sim.set_fields(p.phi0, p.mu0)
    sim.tune(cache, steps_per_trial=2)
    assert sim.tiles()[sim.launch()[0]][2] == 0
    sim.step(3)
    again = sim.get_fields()
    sim.close()
    assert np.isfinite(got[0]).all() and np.abs(got[0] - again[0]).max() <= 1e-5


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


@pytest.mark.parametrize("what", ["tune", "checkpoints"])
def test_scratch_makes_room(what):
    # room for the state and the FP64 cell list, but not for the tuner's copy of the state
    # or a checkpoint as well
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=3, N=2, NM=1, nx=64, ny=40, nz=24, seed=4)
    out = []
    for bounded in (False, True):
        alloc = _bounded()
        sim = Simulation(p, dtype="f64", allocator=alloc)
        assert sim.tiles()[sim.launch()[0]][2] == 1
        if bounded:
            alloc.limit = alloc.used
        sim.set_fields(p.phi0, p.mu0)
        sim.step(2)
        if what == "tune":
            sim.tune(None, steps_per_trial=2)
        else:
            sim.enable_checkpoints(8)   # one: 2.5 MB padded, beside 3.8 MB of scratch
        sim.step(6)
        out.append(sim.get_fields())
        assert not bounded or sim.tiles()[sim.launch()[0]][2] == 0
        sim.close()
    # the same step in other kernels: a few roundings of values up to 2 per step
    assert np.abs(out[0][0] - out[1][0]).max() <= 8 * 32 * 2.0 ** -52
    assert np.abs(out[0][1] - out[1][1]).max() <= 8 * 32 * 2.0 ** -52
