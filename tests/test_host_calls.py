"""The host code's launches, copies and their order, without a GPU."""
import ctypes

import pytest

from hostlib import HostLib

P = ctypes.c_void_p


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return HostLib(tmp_path_factory.mktemp("host"))


@pytest.mark.parametrize("precision", [32, 64])
def test_arrays_of_another_device_travel_by_copy(host, precision):
    """A kernel cannot read or write memory of another GPU without peer
    access; a copy can.  Arrays of the handle's own device go without one."""
    h = host.handle(16, 8, 8, precision, adjoint=True, dt_fixed=0.01)
    n = 8 * 16 * 8 * 8 * precision // 8
    own, far = host.memory(n), host.memory(n, foreign=True)
    calls = [("unpack_kernel", 5, lambda p: host.lib.mhd_write(h, P(p), 0)),
             ("unpack_kernel", 5, lambda p: host.lib.mhd_adjoint_init(h, P(p), 0)),
             ("pack_kernel", 6, lambda p: host.lib.mhd_adjoint_read(h, P(p), None, None, None, 0))]
    for kernel, arg, call in calls:
        for array in (own, far):
            host.clear()
            host.ok(call(array), h)
            ops = host.log()
            at = [i for i, o in enumerate(ops) if o[0] == "launch" and kernel in o[1]]
            assert len(at) == 1
            used = int(ops[at[0]][arg + 1], 16)
            copies = [(i, o) for i, o in enumerate(ops) if o[0] == "copy" and int(o[4]) == n]
            if array == own:
                assert used == own and not copies
            else:
                assert used != far and len(copies) == 1
                i, o = copies[0]
                assert o[1] == "3" and int(o[5], 16) == 0x77  # device to device, on the caller's stream
                if kernel == "unpack_kernel":
                    assert i < at[0] and int(o[3], 16) == far and int(o[2], 16) == used
                else:
                    assert i > at[0] and int(o[2], 16) == far and int(o[3], 16) == used
    host.lib.mhd_destroy(h)
