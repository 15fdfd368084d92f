"""The copies between interior and padded arrays: whole vectors and single
elements (nx no multiple of a vector, arrays that are not 16-byte aligned),
rims, the velocity rows below the photosphere, host and device arrays."""
import ctypes

import numpy as np
import pytest
import torch

import inputs

pytestmark = pytest.mark.gpu


def _sim(shape, prec, periodic, adjoint=False):
    from paper_1908_08557_gb300 import Simulation
    case = inputs.make_box(*shape, seed=3, dt_fixed=0.01 if adjoint else 0.0)
    case.params.update(bc_z=1 if periodic else 0)
    st = np.random.default_rng(4).standard_normal(case.state.shape)
    st = st.astype(np.float32 if prec == 32 else np.float64)
    return case, st, Simulation(case.params, st, case.lnrho0, case.lnT0, precision=prec, adjoint=adjoint)


def _unaligned(a):
    """A device copy of `a` one element past a 16-byte boundary."""
    flat = torch.zeros(a.size + 1, dtype=torch.from_numpy(a).dtype, device="cuda")
    flat[1:] = torch.from_numpy(a).reshape(-1).cuda()
    return flat, ctypes.c_void_p(flat.data_ptr() + a.itemsize)


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("shape,periodic", [((8, 8, 7), False), ((64, 16, 9), False), ((4, 5, 7), True),
                                            ((37, 6, 8), True), ((46, 11, 70), True)])
def test_write_fills_the_padded_set_and_read_returns_it(shape, periodic, prec):
    case, st, sim = _sim(shape, prec, periodic)
    # ln rho and ln T pass through a subtraction and an addition of the profile
    eps = np.finfo(st.dtype).eps
    prof = np.abs(np.concatenate([case.lnrho0, case.lnT0])).max()
    tol = 4 * eps * (prof + np.abs(st).max())
    ref = np.pad(st, ((0, 0), (0, 0), (3, 3), (3, 3)), mode="wrap")
    dev = torch.from_numpy(st).cuda()
    flat, ptr = _unaligned(st)
    for how in ("host", "device", "unaligned"):
        if how == "unaligned":
            assert sim.lib.mhd_write(sim.h, ptr, 0) == 0
        else:
            sim.write(st if how == "host" else dev)
        pad = sim.read_padded(0)
        assert np.array_equal(pad[:6, 3:-3], ref[:6])
        assert np.abs(pad[6:, 3:-3] - ref[6:]).max() <= tol
        if not periodic:
            for m in range(3):
                assert np.array_equal(pad[3:5, m], ref[3:5, 0])
        assert np.abs(pad[5, :3]).max() == 0.0 and np.abs(pad[:6, -3:]).max() == 0.0
        out = sim.read()
        assert torch.equal(out[:6], dev[:6]) and (out[6:] - dev[6:]).abs().max() <= tol
        back = torch.zeros_like(flat)
        assert sim.lib.mhd_read(sim.h, -1, ctypes.c_void_p(back.data_ptr() + st.itemsize), 0) == 0
        assert torch.equal(back[1:].view(out.shape), out)
        assert torch.equal(sim.read(7), out[7])


@pytest.mark.parametrize("prec", [32, 64])
def test_adjoint_seed_and_result_copies(prec):
    """With no reverse step taken, the adjoint read back is the seed (the
    velocity ghost rows it starts with are zero)."""
    case, st, sim = _sim((32, 8, 9), prec, False, adjoint=True)
    dev = torch.from_numpy(st).cuda()
    flat, ptr = _unaligned(st)
    for how in ("host", "device", "unaligned"):
        if how == "unaligned":
            assert sim.lib.mhd_adjoint_init(sim.h, ptr, 0) == 0
        else:
            sim.adjoint_init(st if how == "host" else dev)
        g = sim.adjoint_read()
        assert torch.equal(g["lam"], dev)
        host = np.empty_like(st)
        assert sim.lib.mhd_adjoint_read(sim.h, ctypes.c_void_p(host.ctypes.data), None, None, None, 1) == 0
        assert np.array_equal(host, st)
