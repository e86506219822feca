"""A refused cudaMalloc is reported by the call that asked, and by no other."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_a_refused_cudamalloc_leaves_no_error_behind():
    # without a caller's allocator; an absurd size, so nothing is taken
    import torch
    from paper_2404_01035_gb300 import Simulation
    from paper_2404_01035_gb300._binding import MSError
    p = W.adjoint_well_2d(n=48)
    out = []
    for refuse in (False, True):
        sim = Simulation(p, dtype="f32", torch_alloc=False)
        sim.set_fields(p.phi0, p.mu0)
        sim.enable_checkpoints(1 << 30)   # one segment of 2^30 states: 3e13 bytes
        sim.step(3)
        if refuse:
            with pytest.raises(MSError, match="allocation"):
                sim.grad(torch.ones(2, 1, 48, 48, device="cuda"), None)
        sim.step(3)
        sim.diag()
        out.append(sim.get_fields())
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
