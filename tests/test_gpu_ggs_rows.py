"""Sparse grain growth on rows that allow the four-cell classification and rows
that do not, and on axes of a few cells, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,nx,ny,nz", [(2, 4, 40, 1), (2, 40, 1, 1), (2, 37, 33, 1), (2, 36, 2, 1),
                                          (3, 4, 5, 24), (3, 1, 24, 7), (3, 24, 1, 3), (3, 20, 24, 2), (3, 22, 9, 1)])
@pytest.mark.parametrize("bc", [[3, 3, 3], [1, 1, 1]])
def test_rows_match_the_oracle(dim, nx, ny, nz, bc):
    from paper_2404_01035_gb300.sparse_gg import SparseGrainGrowth
    p = W.sparse_grain_growth(n=40 if dim == 2 else 24, dim=dim, grains=6)
    p = p.copy(nx=nx, ny=ny, nz=nz, bc=bc)
    phi0 = np.ascontiguousarray(np.asarray(p.phi0)[:, :nz, :ny, :nx])
    steps = 12
    s = SparseGrainGrowth(p, dtype="f64")
    s.set_fields(phi0)
    s.step(steps)
    g = np.asarray(s.get_fields(), dtype=np.float64)
    s.close()
    o, _ = oracle.run(p, phi0, np.asarray(p.mu0)[:, :nz, :ny, :nx], steps)
    assert np.abs(g - o).max() <= 1e-10


def test_more_than_32_grains_match_the_oracle():
    # grain indices on both halves of the 64-bit union masks
    from paper_2404_01035_gb300.sparse_gg import SparseGrainGrowth
    p = W.sparse_grain_growth(n=132, dim=2, grains=48)
    steps = 10
    s = SparseGrainGrowth(p, dtype="f64")
    s.set_fields(p.phi0)
    s.step(steps)
    g = np.asarray(s.get_fields(), dtype=np.float64)
    s.close()
    o, _ = oracle.run(p, p.phi0, p.mu0, steps)
    assert np.abs(g - o).max() <= 1e-10
    assert (np.asarray(p.phi0)[32:] > 0).any() and np.abs(o - p.phi0).max() > 1e-3
