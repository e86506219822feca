"""Fields set and read on the device against the same through host memory:
same bits, for rows that allow 16-byte accesses and rows that do not."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _dev(a, dtype, off):
    """A contiguous device copy starting `off` elements into its allocation."""
    t = torch.empty(a.size + off, dtype=dtype, device="cuda")
    v = t[off:].view(a.shape)
    v.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return v


@pytest.mark.parametrize("nx,ny,nz", [(1, 3, 1), (31, 2, 1), (32, 1, 1), (130, 33, 1), (256, 9, 1),
                                      (1, 1, 2), (33, 4, 3), (64, 1, 5), (132, 6, 2)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("N,bc,off", [(2, [3, 3, 3], 0), (3, [1, 1, 1], 0), (3, [3, 1, 3], 1)])
def test_device_fields_equal_host_fields(nx, ny, nz, dtype, N, bc, off):
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=2 if nz == 1 else 3, N=N, NM=N - 1, nx=nx, ny=ny, nz=nz, bc=bc, seed=nx + ny + nz)
    td = torch.float32 if dtype == "f32" else torch.float64
    nd = np.float32 if dtype == "f32" else np.float64
    phi, mu = np.array(p.phi0, dtype=nd), np.array(p.mu0, dtype=nd)
    phi[:, :, ny // 2:] = 0   # pure rows: their segment codes decide what a step rewrites
    phi[1, :, ny // 2:] = 1
    out = []
    for device in (False, True):
        sim = Simulation(p, dtype=dtype)
        for start in range(2):   # a second state over the first one's buffers
            if device:
                sim.set_fields(_dev(np.roll(phi, start, 2), td, off), _dev(mu, td, off))
            else:
                sim.set_fields(np.roll(phi, start, 2), mu)
            sim.step(3)
        if device:
            a, b = _dev(phi, td, off), _dev(mu, td, off)
            sim.get_fields_into(a, b, on_device=True)
            sim.sync()
            out.append((a.cpu().numpy(), b.cpu().numpy()))
        else:
            out.append(sim.get_fields())
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
