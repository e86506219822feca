"""Diagnostics by segment codes (pure segments are not read): regions of one
phase that reach, cross and miss segment and grid edges, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,dtype", [(301, 299, 1, "f32"), (64, 1400, 1, "f32")] + [
    (nx, ny, nz, d) for nx, ny, nz in [(96, 5, 3), (33, 2, 40), (160, 1, 2)] for d in ("f32", "f64")])
@pytest.mark.parametrize("N,bc", [(2, [3, 3, 3]), (3, [1, 1, 1]), (3, [3, 1, 3])])
def test_matches_oracle(nx, ny, nz, dtype, N, bc):
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=2 if nz == 1 else 3, N=N, NM=N - 1, nx=nx, ny=ny, nz=nz, bc=bc, seed=nx + ny)
    p = p.copy(G=p.G * 16.0 / max(ny, nz, 16))
    x, y, z = np.arange(nx)[None, None, :], np.arange(ny)[None, :, None], np.arange(nz)[:, None, None]
    t = np.mod((x + 0.4 * y + 7.0 * z) / 75.0, N)   # stripes of 75 cells, boundaries of 15
    phi = np.stack([np.clip(5.0 * (0.6 - np.abs(np.mod(t - a + 0.5 * N, N) - 0.5 * N)), 0.0, 1.0) for a in range(N)])
    phi = phi / phi.sum(0)
    sim = Simulation(p, dtype=dtype)
    sim.set_fields(phi, p.mu0)
    d = sim.diag()
    m = oracle.diag(p, *sim.get_fields())
    # no segment is pure once a little of every phase is mixed in; the diffusion
    # number moves by a few times that little
    little = 1e-5
    sim.set_fields((1.0 - little) * phi + little / N, p.mu0)
    full = sim.diag()
    sim.close()
    # per-cell values in the state's precision (a few roundings of terms up to ~4), summed in FP64
    eps = 2.0 ** (-24 if dtype == "f32" else -53)
    assert np.abs(d["mass"] - m[:N - 1]).max() <= 64 * eps * nx * ny * nz
    assert abs(d["sum_err"] - m[N - 1]) <= 2 * eps
    assert d["phi_min"] == m[N] and d["phi_max"] == m[N + 1] and d["nonfinite"] == 0
    assert d["mu_diffusion_number"] == pytest.approx(full["mu_diffusion_number"], rel=100 * little)
