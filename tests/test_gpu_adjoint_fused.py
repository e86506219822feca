"""The one-launch FP32 reverse step against the three-pass FP64 one, at the
edges of its tiles (30 x 8 cells) and on periodic and no-flux axes down to one
cell."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 3
# a few hundred FP32 operations per cell and step whose terms exceed the sums by
# up to 1/|q|^2-sized factors on the anisotropic faces: 2^10 units of 2^-24 a step
TOL = STEPS * 2.0 ** (10 - 24)


@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 9), (30, 8), (31, 7), (61, 17), (29, 33)])
@pytest.mark.parametrize("bc", [[3, 3, 3], [1, 3, 3], [1, 1, 3]])
def test_fused_equals_three_passes(nx, ny, bc):
    import torch
    from paper_2404_01035_gb300 import Simulation
    p = W.binary_problem("fused", nx, ny=ny, delta=0.03, Delta=0.2, R=3.0, potential="well", bc=bc)
    # phases mixed everywhere: where |q|^2 nears the anisotropy's cut-off (1e-12,
    # the tails of a profile) the derivative jumps and FP32 says nothing
    x, y = np.arange(nx)[None, None, :] + 0.5, np.arange(ny)[None, :, None] + 0.5
    s = 0.5 + 0.2 * np.sin(2 * np.pi * x / max(nx, 5) + 0.4) + 0.15 * np.cos(2 * np.pi * y / max(ny, 5) + 0.7)
    p.phi0 = np.stack([s, 1.0 - s])
    p.mu0 = p.mu0 + 0.02 * np.cos(2 * np.pi * x / max(nx, 5))
    rng = np.random.default_rng(nx * 100 + ny)
    lam = [rng.normal(size=p.phi0.shape), rng.normal(size=p.mu0.shape)]
    got = {}
    for dtype in ("f32", "f64"):
        t = torch.float32 if dtype == "f32" else torch.float64
        sim = Simulation(p, dtype=dtype)
        sim.set_fields(p.phi0.astype(np.float32), p.mu0.astype(np.float32))
        sim.enable_checkpoints(2)
        sim.step(STEPS)
        dp, dphi, dmu = sim.grad(torch.tensor(lam[0].astype(np.float32), dtype=t, device="cuda"),
                                 torch.tensor(lam[1].astype(np.float32), dtype=t, device="cuda"))
        got[dtype] = (dp, dphi.double().cpu().numpy(), dmu.double().cpu().numpy())
        sim.close()
    for a, b in zip(got["f32"], got["f64"]):
        assert np.abs(a - b).max() <= TOL * max(1.0, np.abs(b).max())
