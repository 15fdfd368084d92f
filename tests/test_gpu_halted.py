"""A handle halted by a non-finite value keeps the state its step began from.

The first step after a write finds the value, and no kernel writes from then
on, while the steps go on swapping the two state sets: every read must give
the state written (or restored), never what the other set held before.
"""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DT = {32: torch.float32, 64: torch.float64}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1908_08557_gb300.build import build
    build()


def _used_handle(shape, precision, periodic):
    """A handle some steps into a run, and its case."""
    from paper_1908_08557_gb300 import Simulation
    case = inputs.make_box(*shape, seed=5)
    case.params.update(bc_z=1 if periodic else 0)
    st = torch.tensor(case.state, dtype=DT[precision], device="cuda")
    sim = Simulation(case.params, st, case.lnrho0, case.lnT0, precision=precision)
    if not periodic:
        d = lambda a: torch.tensor(a, dtype=DT[precision], device="cuda")  # noqa: E731
        sim.set_driver(d(case.bz), d(case.v0), d(case.v1), case.t0, case.t1)
    sim.step(3)
    return case, st, sim


def _bad_state(st):
    g = torch.Generator(device="cpu").manual_seed(6)
    bad = st + 0.01 * torch.randn(st.shape, generator=g, dtype=torch.float64).to(st)
    bad[7, 4, 3, 2] = float("nan")
    return bad


def _assert_same(got, want):
    # A and u come back bit for bit; ln rho, ln T through one subtraction and
    # one addition of the profile (|profile| < 16: half an ulp of 16 each)
    tol = 16 * torch.finfo(want.dtype).eps
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(got[:6], want[:6])
    assert (got[6:] - want[6:]).nan_to_num().abs().max().item() <= tol


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("shape,periodic", [((16, 16, 10), False), ((16, 16, 7), False), ((128, 128, 12), False),
                                            ((18, 12, 10), True)])
def test_reads_of_a_halted_handle_return_the_state_written(shape, periodic, precision):
    from paper_1908_08557_gb300 import MHDError
    from paper_1908_08557_gb300.binding import MHD_ERR_NONFINITE
    case, st, sim = _used_handle(shape, precision, periodic)
    bad = _bad_state(st)
    sim.write(bad)
    for n in (1, 1, 2, 1):  # both parities of the swapped sets
        sim.step(n)
        _assert_same(sim.read(), bad)
        assert torch.equal(sim.read_plane(3, 4), bad[3, 4])
        assert np.array_equal(sim.read_padded(0)[0, 3:-3, 3:-3, 3:-3], bad[0].cpu().numpy())
        with pytest.raises(MHDError) as e:
            sim.time()
        assert e.value.code == MHD_ERR_NONFINITE
    # saved and restored on a halted handle: that state, after further steps too
    ck = sim.new_checkpoint()
    sim.save(ck)
    _, _, other = _used_handle(shape, precision, periodic)
    ck2 = other.new_checkpoint()
    other.save(ck2)
    sim.restore(ck2, 0.0)
    for n in (0, 1, 2):
        sim.step(n)
        assert torch.equal(sim.read(), other.read())
    sim.restore(ck, 0.0)
    sim.step(1)
    _assert_same(sim.read(), bad)
    # a good state written clears the flag
    sim.write(st)
    sim.set_time(0.0)
    sim.step(3)
    assert torch.equal(sim.read(), other.read())
    sim.time()
    sim.close()
    other.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_a_taped_step_that_halts_leaves_its_state(precision):
    case, st, sim = _used_handle((16, 16, 10), precision, False)
    bad = _bad_state(st)
    tape = sim.new_tape()
    sim.write(bad)
    for _ in range(2):
        sim.step_taped(tape)
        _assert_same(sim.read(), bad)
    sim.close()
