"""The FP64 z-march right-hand side (shared first derivatives) against the
one-thread-per-cell kernel on the same state, over every form the entry points
take: tiles ragged in x and y, the smallest boxes, z chunks of one layer and
more, triply periodic odd sizes, a stretched vertical grid, Newtonian cooling,
A about a background, and the update itself."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu

# Each kernel's FP64 right-hand side is held to 1e-11 of its field's scale
# against the oracle; two of them differ by at most the sum.
TOL = 2e-11


def _case(nx, ny, nz, opt, seed=5):
    kw = {}
    if opt == "z":
        kw["z"] = inputs.stretched_z(nz, 0.5, 1.5, nz / 3.0, nz / 8.0)[0]
    if opt == "cooling":
        kw["nc_tau"] = 0.5
    case = inputs.make_box(nx, ny, nz, seed=seed, **kw)
    rng = np.random.default_rng(seed)
    case.state[3:6] += 0.1 * rng.standard_normal(case.state[3:6].shape)
    case.state[0:3] += 0.1 * rng.standard_normal(case.state[0:3].shape)
    case.state[6:8] += 0.05 * rng.standard_normal(case.state[6:8].shape)
    if opt == "periodic":
        case.params.update(bc_z=1)
    return case


def _sim(case, variant, monkeypatch, opt):
    from paper_1908_08557_gb300 import Simulation
    if variant:
        monkeypatch.setenv("MHD_RK_VARIANT", variant)
    else:
        monkeypatch.delenv("MHD_RK_VARIANT", raising=False)
    bg = np.ascontiguousarray(0.7 * case.state[0:3]) if opt == "background" else None
    sim = Simulation(case.params, case.state, case.lnrho0, case.lnT0, precision=64, a_background=bg)
    if bg is not None:
        sim.set_a_background(bg, np.ascontiguousarray(case.state[0:3] - bg))
    if opt != "periodic":
        sim.set_driver(case.bz, case.v0, case.v1, case.t0, case.t1)
    return sim


@pytest.mark.parametrize("shape,opt", [
    ((8, 8, 7), "plain"), ((32, 8, 9), "plain"), ((64, 16, 33), "plain"), ((128, 64, 40), "plain"),
    ((4, 5, 7), "periodic"), ((37, 11, 13), "periodic"), ((33, 6, 8), "periodic"), ((150, 9, 17), "periodic"),
    ((16, 16, 24), "z"), ((64, 8, 19), "cooling"), ((32, 16, 21), "background")])
def test_rhs_and_step_match_one_thread_per_cell(shape, opt, monkeypatch):
    case = _case(*shape, opt)
    got = {}
    for v in ("", "simple"):
        sim = _sim(case, v, monkeypatch, opt)
        sim.fill_ghosts()
        r = sim.eval_rhs(0.3)
        sim.step(2)
        got[v] = (r, sim.read().cpu().numpy(), sim.read_padded(0))
        sim.close()
    for a, b in zip(got[""], got["simple"]):
        for f in range(8):
            assert np.isfinite(b[f]).all()
            s = max(np.abs(b[f]).max(), 1e-30)
            assert np.abs(a[f] - b[f]).max() <= TOL * s, (f, np.abs(a[f] - b[f]).max(), s)


def test_non_finite_cell_is_reported(monkeypatch):
    """A NaN reaches the time-step reduction through the new kernel's update as through the other's."""
    from paper_1908_08557_gb300 import MHDError
    case = _case(16, 8, 9, "plain")
    case.state[4, 3, 2, 1] = np.nan
    sim = _sim(case, "", monkeypatch, "plain")
    sim.step(2)
    with pytest.raises(MHDError):
        sim.time()
