"""The anti-trapping current in FP32 whatever the launch.  A face's unit normal is
switched on at |grad phi|^2 >= 1e-12, a few units of FP32 rounding of phi, and has
length 1 however small the gradient: where a trace of liquid lies in a solid-solid
boundary the last bits of phi decide whether the current acts, and a launch that
sums in another order ends up to 1e-2 away in single cells.  So every launch of a
model with the current takes the same sums."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _profile(u):
    return 0.5 * (1.0 + np.sin(4.0 / np.pi * np.clip(u, -np.pi ** 2 / 8, np.pi ** 2 / 8)))


def eutectic(nx, ny, nz, seed):
    """Lamellae of two solids under a wavy front, ternary, the current on; fields in
    multiples of 2^-22 (the same inputs on every machine)."""
    p = W.eutectic_3d(n=32).copy(nx=nx, ny=ny, nz=nz, anti_trapping=1)
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(np.arange(nz) + 0.5, np.arange(ny) + 0.5, np.arange(nx) + 0.5, indexing="ij")
    n = max(1, nx // 24)
    near = nx / (2.0 * n) / np.pi * np.sin(2 * np.pi * n * x / nx + rng.uniform(0, 6))
    front = 0.5 * nz + 2.0 * np.sin(2 * np.pi * x / nx + rng.uniform(0, 6)) * np.cos(2 * np.pi * y / ny + rng.uniform(0, 6))
    a, liquid = _profile(near / p.eps), _profile((z - front) / p.eps)
    phi = np.stack([(1 - liquid) * a, (1 - liquid) * (1 - a), liquid])
    layer = np.exp(-np.maximum(z - front, 0.0) / 12.0) * (a - 0.5)
    q = 2.0 ** 22
    p.phi0 = np.round(phi * q) / q
    p.mu0 = np.round(np.stack([0.8 + 0.02 * layer, 0.8 - 0.02 * layer]) * q) / q
    return p


def run(p, split, steps, dtype="f32"):
    from paper_2404_01035_gb300 import Simulation
    sim = Simulation(p, dtype=dtype)
    if split is not None:
        sim.set_launch([i for i, t in enumerate(sim.tiles()) if t[2] == split][0])
    sim.set_fields(np.asarray(p.phi0, dtype=sim.np_dtype), np.asarray(p.mu0, dtype=sim.np_dtype))
    sim.step(steps)
    out = sim.get_fields()
    sim.sync()
    sim.close()
    return out


def binary(dim, nx, ny, nz):
    p = W.small_multiphase(n=8, dim=dim, N=2, NM=1, nx=nx, ny=ny, nz=nz, rotate=True, seed=nx + ny)
    return p.copy(anti_trapping=1)


@pytest.mark.parametrize("dim,nx,ny,nz", [(2, 77, 60, 1), (2, 160, 33, 1), (3, 45, 17, 20), (3, 64, 12, 9)])
def test_binary_split_and_fused_steps_give_the_same_bits(dim, nx, ny, nz):
    p = binary(dim, nx, ny, nz)
    a, b = run(p, 1, 25), run(p, 0, 25)
    assert np.abs(a[0] - np.asarray(p.phi0)).max() > 1e-3
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def test_ternary_split_and_fused_steps_agree_to_the_last_bit_of_mu():
    # one step (later ones amplify); mu near 1: a unit in the last place is 6e-8
    p = eutectic(72, 20, 44, 3)
    a, b = run(p, 1, 1), run(p, 0, 1)
    assert np.array_equal(a[0], b[0])
    assert np.abs(a[1] - b[1]).max() <= 2.0 ** -24
    assert (a[1] != b[1]).mean() <= 1e-4


def test_values_where_a_trace_switches_the_current():
    # cells beside such a trace after 60 steps, as the fused step gives them (the
    # present one, and the one that every launch was until the split step became the
    # default); sums taken in another order end 1.5e-4 away here
    kept = {(0, 11, 8, 13): 0.7960939407348633, (0, 11, 8, 12): 0.7972019910812378,
            (1, 11, 8, 12): 0.8025597333908081, (1, 11, 8, 13): 0.802801251411438}
    mu = run(eutectic(72, 20, 44, 22), None, 60)[1]
    for cell, value in kept.items():
        assert abs(float(mu[cell]) - value) <= 2e-6   # the other cells' rounding over 60 steps


def test_many_phases_with_the_current_start_fused():
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=12, dim=3, N=8, NM=1, seed=3)
    for current, split in ((0, 1), (1, 0)):
        sim = Simulation(p.copy(anti_trapping=current), dtype="f32")
        assert sim.tiles()[sim.launch()[0]][2] == split
        sim.close()


def test_turning_the_current_on_and_off_with_many_phases():
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=12, dim=3, N=8, NM=1, seed=3)
    out = []
    for how in ("created", "updated", "chosen"):
        sim = Simulation(p.copy(anti_trapping=int(how == "created")), dtype="f32")
        split = [t[2] for t in sim.tiles()]
        if how == "chosen":
            sim.set_launch(split.index(1))
        if how != "created":
            sim.update_params(anti_trapping=1)
        assert split[sim.launch()[0]] == (how == "chosen")
        sim.set_fields(p.phi0, p.mu0)
        sim.step(10)
        out.append(sim.get_fields())
        sim.update_params(anti_trapping=0)
        assert split[sim.launch()[0]] == 1
        sim.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
