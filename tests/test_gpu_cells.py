"""The cell-list FP64 step against the oracle: row lengths on either side of a
segment, every boundary code, many phases, the options."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (31, 4, 5), (32, 5, 3), (33, 3, 6), (65, 6, 4), (96, 2, 7)])
@pytest.mark.parametrize("N,bc,kind", [(2, [3, 3, 3], "noise"), (3, [1, 3, 1], "rotated"), (3, [3, 1, 3], "anti_trapping"),
                                       (8, [3, 3, 1], "rotated"), (8, [1, 1, 1], "grain_growth")])
def test_cells_match_the_oracle(nx, ny, nz, N, bc, kind):
    p = W.small_multiphase(n=8, dim=3, N=N, NM=2 if N == 3 else 1, nx=nx, ny=ny, nz=nz, bc=bc, seed=nx + nz,
                           rotate=kind == "rotated", aniso=kind != "grain_growth", gamma3=0.3 if kind == "rotated" else 0.0)
    p = p.copy(**{"noise": dict(noise_amp=0.02, noise_seed=5), "anti_trapping": dict(anti_trapping=1),
                  "grain_growth": dict(grain_growth=1)}.get(kind, {}))
    from paper_2404_01035_gb300 import Simulation
    sim = Simulation(p, dtype="f64")
    tiles = sim.tiles()
    assert tiles[sim.launch()[0]] == (32, 1, 1)
    sim.set_fields(p.phi0, p.mu0)
    sim.step(6)
    g = sim.get_fields()
    sim.sync()
    sim.close()
    o = oracle.run(p, p.phi0, p.mu0, 6)
    assert max(np.abs(g[0] - o[0]).max(), np.abs(g[1] - o[1]).max()) <= 1e-10


@pytest.mark.parametrize("dtype,tol", [("f64", 1e-10), ("f32", 1e-4)])
def test_sparse_grains_with_a_table_of_gammas(dtype, tol):
    # unequal boundary energies: the pair form of the sparse update
    from paper_2404_01035_gb300.sparse_gg import SparseGrainGrowth
    p = W.sparse_grain_growth(n=64, dim=2, grains=12)
    rng = np.random.default_rng(2)
    gam = 0.85 + 0.15 * rng.random((12, 12))
    gam = np.triu(gam, 1)
    p = p.copy(gamma=gam + gam.T)
    s = SparseGrainGrowth(p, dtype=dtype)
    s.set_fields(p.phi0)
    s.step(25)
    s.sync()
    phi = s.get_fields()
    assert s.stats()[1] == 25 and 0 < s.stats()[0] < 64 * 64
    s.close()
    o, _ = oracle.run(p, p.phi0, p.mu0, 25)
    assert np.abs(phi - o).max() <= tol
