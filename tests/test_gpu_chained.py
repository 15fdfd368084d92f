"""The launches of a small box's step and of its adjoint, each queued behind its
predecessor, against the same handle's plain launches (a profiled handle records
events between its kernels and chains none of them); and the adjoint's column
transforms one layer at a time (columns of 1024)."""
import numpy as np
import pytest

import inputs
import test_gpu_ghost_planes as planes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# The same arithmetic in the same order; only the ghost rules are compiled into
# another kernel, where a product and a sum may be contracted otherwise: one
# rounding of a value of up to 16 times the fields' scales in each of nine ghost
# values of a column, through stencils of weights below 3 and three substeps of
# dt <= 0.3: below 16 * 9 * 3 * 0.3 = 130 eps of a field's scale.
TOL = {32: 130 * 2.0 ** -23, 64: 130 * 2.0 ** -52}
DT = {32: torch.float32, 64: torch.float64}


def _run(shape, precision, periodic, plain):
    from paper_1908_08557_gb300 import Simulation
    nx, ny, nz = shape
    case = inputs.make_box(nx, ny, nz, seed=3, **({} if periodic else dict(magnetogram="bipoles", n_mag=6)))
    case.params = dict(case.params, dt_fixed=0.0 if periodic else 0.01, bc_z=1 if periodic else 0)
    rng = np.random.default_rng(4)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=DT[precision], device="cuda")  # noqa: E731
    st = case.state + 0.01 * rng.standard_normal(case.state.shape)
    lam = dev(rng.standard_normal(st.shape))
    sim = Simulation(case.params, dev(st), case.lnrho0, case.lnT0, precision=precision, adjoint=not periodic)
    if not periodic:
        sim.set_driver(dev(case.bz), dev(case.v0), dev(case.v1), case.t0, case.t1)
    sim.profile(1 if plain else 0)
    sim.set_time(0.3)
    sim.step(3)
    out = {"state": sim.read()}
    if not periodic:
        tape, ck = sim.new_tape(), sim.new_checkpoint()
        t = sim.save(ck)
        sim.step_taped(tape)
        out["taped"] = sim.read()
        sim.adjoint_init(lam)
        sim.adjoint_step_taped(tape)
        out.update({"taped " + k: v for k, v in sim.adjoint_read().items()})
        sim.adjoint_init(lam)
        sim.restore(ck, t)
        sim.adjoint_step()
        out.update(sim.adjoint_read())
    sim.close()
    return out


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("shape,periodic", [((8, 8, 7), False), ((8, 8, 9), False), ((8, 64, 7), False),
                                            ((64, 8, 8), False), ((32, 16, 7), False), ((64, 128, 11), False),
                                            ((18, 12, 9), True), ((130, 67, 12), True)])
def test_chained_launches_match_plain_ones(shape, periodic, precision):
    got, want = (_run(shape, precision, periodic, plain) for plain in (False, True))
    for name, w in want.items():
        g = got[name]
        for a, b in zip(g, w) if w.dim() == 4 else [(g, w)]:
            assert torch.isfinite(b).all()
            assert (a - b).abs().max() <= TOL[precision] * b.abs().max(), name


@pytest.mark.parametrize("shape", [(8, 1024, 7), (16, 1024, 7)])
def test_adjoint_columns_one_layer_at_a_time(shape):
    """12 * 16 bytes a point and pair exceed 96 KB from columns of 1024 on; the
    first plane takes the chained launches, the second does not."""
    planes.test_adjoint_over_plane_sizes(shape)
