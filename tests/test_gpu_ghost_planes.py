"""Potential-field ghost layers over plane sizes: one and several lines per
block, one thread per point and per radix-4 butterfly, the chained launches of
small planes and the separate chains of larger ones."""
import numpy as np
import pytest

import inputs
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("plane", [(8, 8), (8, 16), (16, 8), (32, 32), (8, 128), (128, 8), (64, 32), (32, 256),
                                   (64, 128), (128, 64), (512, 16), (16, 512), (128, 128), (8, 1024), (1024, 8),
                                   (256, 128)])
def test_ghost_fill_over_plane_sizes(plane):
    """Against numpy's FFT.  A radix-2 transform in FP64 errs by about
    eps log2 n of the 2-norm per direction (eps = 1.1e-16), here up to 14 stages
    forward and back: 3e-15, and the largest value is within a factor of ten
    of the rms; 1e-13 of the largest value."""
    nx, ny = plane
    from paper_1908_08557_gb300 import Simulation
    case = inputs.make_box(nx, ny, 7, seed=nx + 3 * ny)
    rng = np.random.default_rng(5)
    st = case.state + 0.05 * rng.standard_normal(case.state.shape)
    sim = Simulation(case.params, st, case.lnrho0, case.lnT0, precision=64)
    sim.fill_ghosts()
    got = sim.read_padded(0)
    sim.close()
    u = oracle.to_padded(st)
    oracle.fill_ghosts(case.params, u, case.lnrho0, pfe="fft")
    scale = np.abs(u).max(axis=(1, 2, 3))
    err = np.abs(got - u).max(axis=(1, 2, 3))
    assert np.all(err <= 1e-13 * scale), err / scale


@pytest.mark.parametrize("shape", [(8, 8, 7), (8, 64, 8), (64, 8, 13), (128, 16, 7), (16, 256, 9), (512, 8, 7)])
def test_adjoint_over_plane_sizes(shape):
    """<lam, (F(x + e v) - F(x - e v)) / 2e> = <J^T lam, v> of one FP64 step.
    Central differences with e = 1e-5 leave truncation of order e^2 = 1e-10
    and rounding of order 1e-16 / e = 1e-11 of a cell's response, both times
    the response's curvature and the 40-odd operations of a stencil: 1e-7 of
    the 2-norm of the products, the size a sum of random signs has."""
    torch = pytest.importorskip("torch")
    from paper_1908_08557_gb300 import Simulation
    nx, ny, nz = shape
    case = inputs.make_box(nx, ny, nz, seed=2, magnetogram="bipoles", n_mag=6)
    case.params = dict(case.params, dt_fixed=0.01)
    rng = np.random.default_rng(9)
    st = case.state.copy()
    st[0:8] += 0.01 * rng.standard_normal(st.shape)
    v = 0.01 * rng.standard_normal(st.shape)
    lam = rng.standard_normal(st.shape)
    sim = Simulation(case.params, st, case.lnrho0, case.lnT0, precision=64, adjoint=True)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    sim.set_driver(dev(case.bz), dev(case.v0), dev(case.v1), case.t0, case.t1)

    def forward(x):
        sim.write(dev(x))
        sim.set_time(0.3)
        sim.step(1)
        return sim.read().cpu().numpy()

    e = 1e-5
    jv = (forward(st + e * v) - forward(st - e * v)) / (2 * e)
    sim.write(dev(st))
    sim.set_time(0.3)
    ck = sim.new_checkpoint()
    t = sim.save(ck)
    sim.adjoint_init(dev(lam))
    sim.restore(ck, t)
    sim.adjoint_step()
    got = float(np.sum(sim.adjoint_read()["lam"].cpu().numpy() * v))
    sim.close()
    assert abs(got - float(np.sum(lam * jv))) <= 1e-7 * np.linalg.norm(lam * jv)
