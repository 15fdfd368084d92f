"""The FP32 time-step reduction over boxes whose z chunks are one to eight
layers and longer, whole and ragged, with the fastest cell on each layer in
turn near the chunks' ends: the z-march of the step against the plane-parallel
reduction of compute_dt, bit for bit (the same arithmetic, order-independent
maxima)."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(32, 32, 24), (64, 64, 64), (128, 64, 50), (128, 128, 45), (256, 128, 70)])
def test_step_dt_equals_standalone(shape):
    from paper_1908_08557_gb300 import Simulation
    nx, ny, nz = shape
    case = inputs.make_box(nx, ny, nz, seed=3, magnetogram="bipoles", n_mag=6)
    rng = np.random.default_rng(6)
    st = case.state.astype(np.float32)
    st[3:6] += 0.02 * rng.standard_normal(st[3:6].shape).astype(np.float32)
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    sim = Simulation(case.params, dev(st), case.lnrho0, case.lnT0, precision=32)
    sim.set_driver(dev(case.bz), dev(case.v0), dev(case.v1), case.t0, case.t1)
    for k in (3, 4, 5, 6, 10, 11, nz // 2, nz - 5, nz - 4):
        fast = st.copy()
        fast[5, k, int(rng.integers(ny)), int(rng.integers(nx))] = 40.0
        sim.write(dev(fast))
        sim.fill_ghosts()
        dt = sim.compute_dt()
        t = sim.time()[0]
        sim.step(1)
        assert sim.time()[1] == dt, (k, dt, sim.time()[1])
        assert sim.time()[0] == t + dt
    sim.close()
