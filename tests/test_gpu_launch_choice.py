"""Which kernel a step of a small 2-D grid and of a small batch takes: the
multi-step (unit) kernel until a variant is chosen, the chosen one afterwards, and
after tuning the one that was found the fastest.  The fused 2-D kernels, which such
grids run no other way, against the multi-step kernel."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _kernels(run):
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        run()
        torch.cuda.synchronize()
    return " ".join(e.key for e in prof.key_averages())


@pytest.fixture(scope="module", autouse=True)
def _profiler_is_up():
    # the first session of a process may still be starting when its kernels run
    import torch
    for _ in range(10):
        if "kernel" in _kernels(lambda: torch.ones(1000, device="cuda").add_(1.0)):
            return
    pytest.skip("the profiler names no kernels here")


def _problem(N, nx, ny):
    p = W.small_multiphase(n=8, dim=2, N=N, NM=N - 1, nx=nx, ny=ny, rotate=True, seed=nx + ny)
    return p.copy(G=p.G * 16.0 / ny)


@pytest.mark.parametrize("N,nx,ny", [(2, 65, 70), (3, 65, 70), (3, 160, 130), (3, 33, 5)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_a_chosen_variant_runs_and_agrees(N, nx, ny, dtype):
    from paper_2404_01035_gb300 import Simulation
    p = _problem(N, nx, ny)
    out, steps = [], 20
    for choose in (False, True):
        sim = Simulation(p, dtype=dtype)
        if choose:
            sim.set_launch([i for i, t in enumerate(sim.tiles()) if t[2] == 0][0])
        sim.set_fields(p.phi0, p.mu0)
        if nx == 65:
            names = _kernels(lambda: sim.step(steps))
            assert ("k_gp_multi" in names) != choose and ("k_gp_step" in names) == choose
        else:
            sim.step(steps)
        out.append(sim.get_fields())
        sim.close()
    # a few roundings of values up to 2 a step
    tol = steps * 8 * 2 * (2.0 ** -24 if dtype == "f32" else 2.0 ** -53)
    assert np.abs(out[0][0] - p.phi0).max() > 1e-3
    assert np.abs(out[0][0] - out[1][0]).max() <= tol and np.abs(out[0][1] - out[1][1]).max() <= tol


def test_the_tuner_times_what_a_step_takes(tmp_path):
    from paper_2404_01035_gb300 import Simulation
    p = _problem(2, 128, 128)
    cache = str(tmp_path / "tuned.json")
    sim = Simulation(p, dtype="f32")
    sim.set_fields(p.phi0, p.mu0)
    sim.set_launch(0)
    ms = sim.tune(cache, steps_per_trial=200)
    # 3.9 us a step against 6.2 by one launch each
    assert '"multi": 1' in open(cache).read()
    assert "k_gp_multi" in _kernels(lambda: sim.step(5))
    sim.close()
    sim = Simulation(p, dtype="f32")
    sim.set_fields(p.phi0, p.mu0)
    sim.set_launch(0)
    assert abs(sim.tune(cache, steps_per_trial=200) - ms) <= 1e-6 * ms   # from the file
    assert "k_gp_multi" in _kernels(lambda: sim.step(5))
    # an entry that does not name the multi-step kernel was no comparison with it
    text = open(cache).read()
    open(cache, "w").write(text.replace(', "multi": 1', ""))
    sim.set_launch(0)
    sim.tune(cache, steps_per_trial=200)
    assert '"multi": 1' in open(cache).read() and "k_gp_multi" in _kernels(lambda: sim.step(5))
    # one in which a variant won is obeyed
    open(cache, "w").write(text.replace('"multi": 1', '"multi": 0'))
    sim.tune(cache, steps_per_trial=200)
    assert "k_gp_multi" not in _kernels(lambda: sim.step(5))
    sim.close()


def test_a_chosen_strip_height_runs_and_agrees():
    from paper_2404_01035_gb300.batch import Batch
    ps = [W.binary_problem(f"b{i}", 64 + 13 * i, ny=50 + 7 * i, delta=0.02 * i, Delta=0.2, R=8.0) for i in range(4)]
    out, steps = [], 12
    for choose in (None, 4, 8, "late", "tune"):
        b = Batch(ps)
        for i, p in enumerate(ps):
            b.set_fields(i, p.phi0, p.mu0)
        if choose in (4, 8):
            b.set_tile(choose)
            assert "k_batch<" in _kernels(lambda: b.step(steps))
        elif choose == "late":   # the unit kernel keeps no segment codes
            assert "k_batch_units" in _kernels(lambda: b.step(5))
            b.set_tile(16)
            assert "k_batch<" in _kernels(lambda: b.step(steps - 5))
        elif choose == "tune":
            b.step(3)
            b.tune(steps_per_trial=20)
            assert "k_batch_units" in _kernels(lambda: b.step(steps - 3))   # 4.7 us a step against 14
        else:
            b.step(steps)
        b.sync()
        out.append([b.get_fields(i) for i in range(len(ps))])
        b.close()
    tol = steps * 8 * 2 * 2.0 ** -24
    for o in out[1:]:
        for (p0, m0), (p1, m1) in zip(out[0], o):
            assert np.abs(p0 - p1).max() <= tol and np.abs(m0 - m1).max() <= tol
