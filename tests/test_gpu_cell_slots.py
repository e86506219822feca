"""FP64 3-D grids beyond 2^22 cells, where only some listed cells have a place for
their fluxes: few cells listed, and more than there are places, against the fused
step."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [[3, 3, 3], [1, 3, 1]])
@pytest.mark.parametrize("dense", [False, True])
def test_places_for_fluxes(dense, bc):
    import torch
    from paper_2404_01035_gb300 import Simulation
    nx, ny, nz = 173, 170, 171   # 5.0 M cells, 4.2 M places
    p = W.small_multiphase(n=8, dim=3, N=2, NM=1, rotate=True, bc=bc, seed=3)
    p = p.copy(nx=nx, ny=ny, nz=nz, phi0=None, mu0=None, G=0.0)
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) + 0.5 for n in (nz, ny, nx)]
    z, y, x = ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]
    if dense:   # every cell mixed
        a = 0.5 + 0.2 * torch.sin(0.21 * x + 0.1 * y) * torch.cos(0.17 * z - 0.05 * y)
    else:       # a ball in liquid
        r = torch.sqrt((x - 80.0) ** 2 + (y - 75.0) ** 2 + (z - 20.0) ** 2)
        a = 0.5 * (1.0 + torch.sin(4.0 / np.pi * ((30.0 - r) / p.eps).clamp(-np.pi ** 2 / 8, np.pi ** 2 / 8)))
    phi = torch.stack([a, 1.0 - a]).contiguous()
    mu = (1.6 + 0.01 * torch.sin(0.3 * x) * torch.cos(0.2 * y + 0.1 * z))[None].contiguous()
    out = []
    for split in (1, 0):
        sim = Simulation(p, dtype="f64")
        sim.set_launch([i for i, t in enumerate(sim.tiles()) if t[2] == split][0])
        sim.set_fields(phi, mu)
        sim.step(2)
        q, m = torch.empty_like(phi), torch.empty_like(mu)
        sim.get_fields_into(q, m, True)
        out.append((q, m))
        sim.close()
    # a few roundings of values up to 2 a step
    assert float((out[0][0] - phi).abs().max()) > 1e-4
    assert float((out[0][0] - out[1][0]).abs().max()) <= 2 * 16 * 2.0 ** -52
    assert float((out[0][1] - out[1][1]).abs().max()) <= 2 * 16 * 2.0 ** -52


def test_scratch_is_a_fraction_of_the_state():
    from paper_2404_01035_gb300 import Simulation
    from paper_2404_01035_gb300._binding import TorchAllocator

    class Counting(TorchAllocator):
        sizes = []

        def _do_alloc(self, nbytes, user):
            self.sizes.append(int(nbytes))
            return super()._do_alloc(nbytes, user)

    cells = 340 ** 3
    p = W.small_multiphase(n=8, dim=3, N=3, NM=2, seed=3).copy(nx=340, ny=340, nz=340, phi0=None, mu0=None, G=0.0)
    alloc = Counting()
    sim = Simulation(p, dtype="f64", allocator=alloc)
    assert sim.tiles()[sim.launch()[0]][2] == 1
    state = 2 * 5 * 8 * cells
    assert sum(alloc.sizes) <= 1.5 * state   # (rows are padded by 3%)
    sim.close()
