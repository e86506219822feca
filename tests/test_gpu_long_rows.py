"""Grids of more than 2^27 row segments: a thread per lane of each would pass 2^32."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _room(gigabytes):
    import torch
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    if free < gigabytes * 10 ** 9:
        pytest.skip(f"needs {gigabytes} GB of device memory")


def _spec(**kw):
    p = W.small_multiphase(n=4, dim=kw["dim"], N=2, NM=1, seed=2)
    return p.copy(phi0=None, mu0=None, G=0.0, **kw)


def test_fields_of_a_tall_grid():
    import torch
    from paper_2404_01035_gb300 import Simulation
    _room(130)   # two states of 51.5 GB, lists and fields
    ny = (1 << 27) + 1000
    sim = Simulation(_spec(dim=2, nx=1, ny=ny, nz=1), dtype="f32")
    mu = torch.arange(ny, device="cuda", dtype=torch.float32).reshape(1, 1, ny, 1)
    phi = torch.zeros(2, 1, ny, 1, device="cuda")
    phi[1] = 1.0
    phi[0, 0, -5:] = 0.25
    phi[1, 0, -5:] = 0.75
    sim.set_fields(phi, mu)
    p, m = torch.empty_like(phi), torch.empty_like(mu)
    sim.get_fields_into(p, m, True)
    same = bool(torch.equal(p, phi)) and bool(torch.equal(m, mu))
    sim.close()
    del sim, p, m, phi, mu
    torch.cuda.empty_cache()
    assert same


def test_cell_list_of_a_grid_of_single_cells():
    import torch
    from paper_2404_01035_gb300 import Simulation
    _room(150)   # two states of 51.6 GB, 8.3 GB of scratch, fields
    ny, nz = 16384, 8193
    sim = Simulation(_spec(dim=3, nx=1, ny=ny, nz=nz), dtype="f64")
    assert sim.tiles()[sim.launch()[0]][2] == 1
    # pure liquid, mu a parity pattern that one step of diffusion moves everywhere
    mu = torch.ones(1, nz, ny, 1, device="cuda", dtype=torch.float64)
    mu[:, :, ::2] = 1.25
    phi = torch.zeros(2, nz, ny, 1, device="cuda", dtype=torch.float64)
    phi[1] = 1.0
    sim.set_fields(phi, mu)
    del phi
    sim.step(1)
    out = sim.fields()[1].clone()
    sim.close()
    del sim
    moved = bool((out != mu).all())
    # every row of a kind holds the same value
    even, odd = out[:, :, ::2], out[:, :, 1::2]
    same = float(even.max() - even.min()) <= 1e-12 and float(odd.max() - odd.min()) <= 1e-12
    del out, even, odd, mu
    torch.cuda.empty_cache()
    assert moved and same
