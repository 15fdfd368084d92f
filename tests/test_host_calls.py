"""The host code's launches, copies and their order, without a GPU."""
import ctypes

import pytest

import inputs
from hostlib import STREAM, HostLib
from paper_1908_08557_gb300.binding import GranParams
from paper_1908_08557_gb300.granulation import paper_params

P = ctypes.c_void_p
D = ctypes.c_double


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
                assert o[1] == "3" and int(o[5], 16) == STREAM  # device to device, on the caller's stream
                if kernel == "unpack_kernel":
                    assert i < at[0] and int(o[3], 16) == far and int(o[2], 16) == used
                else:
                    assert i > at[0] and int(o[2], 16) == far and int(o[3], 16) == used
    host.lib.mhd_destroy(h)


def _uploads_on_the_stream(ops):
    """Every host-to-device copy is queued on the caller's stream, so that the
    kernels behind it there find the table: one on the legacy stream may still
    be under way when cudaMemcpy returns."""
    ups = [o for o in ops if o[0] == "copy" and o[1] == "1"]
    assert ups
    for o in ups:
        assert o[5] != "sync" and int(o[5], 16) == STREAM, o


@pytest.mark.parametrize("nx,ny", [(64, 32), (16, 64)])
def test_generator_tables_are_ordered_before_their_kernels(host, nx, ny):
    gp = GranParams(**paper_params(mm_per_unit=0.23))
    n = host.lib.mhd_gran_workspace_bytes(nx, ny, D(1.0), D(1.0), ctypes.byref(gp))
    assert n
    g = P()
    host.clear()
    host.ok(host.lib.mhd_gran_create(nx, ny, D(1.0), D(1.0), ctypes.byref(gp), P(host.memory(n)), ctypes.c_size_t(n),
                                     P(STREAM), ctypes.byref(g)), None)
    ops = host.log()
    assert any(o[0] == "launch" for o in ops)
    _uploads_on_the_stream(ops)
    host.lib.mhd_gran_destroy(g)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("over", [{}, {"z": True}, {"bc_z": 1}])
def test_handle_tables_are_ordered_before_their_kernels(host, precision, over):
    if "z" in over:
        over = dict(z=inputs.stretched_z(12, 0.5, 1.5, 4, 2)[0])
    host.clear()
    h = host.handle(16, 8, 12, precision, **over)
    _uploads_on_the_stream(host.log())
    host.lib.mhd_destroy(h)


def _reaches(ops):
    """after(i, j): operation j can only run once i has (stream order and events)."""
    before = [set() for _ in ops]  # direct predecessors
    last, recorded = {}, {}
    for n, o in enumerate(ops):
        stream = o[2] if o[0] in ("launch", "record") else o[1] if o[0] in ("wait", "sync") else o[-1]
        if stream in last:
            before[n].add(last[stream])
        if o[0] == "record":
            recorded[o[1]] = n
        elif o[0] == "wait":
            before[n].add(recorded[o[2]])
        last[stream] = n
    anc = [set() for _ in ops]
    for n in range(len(ops)):
        for b in before[n]:
            anc[n] |= anc[b] | {b}
    return lambda i, j: i in anc[j]


@pytest.mark.parametrize("nx,ny,fft_kernels", [(128, 128, 9), (64, 64, 3)])
def test_profiled_fft_time_ends_with_its_last_chain(host, nx, ny, fft_kernels):
    """mhd_profile(h, 1): a class's times hold all of its kernels, on whatever
    stream they run, and none of the step's other work."""
    h = host.handle(nx, ny, 8, 32, dt_fixed=0.01)
    host.ok(host.lib.mhd_profile(h, 1), h)
    host.clear()
    host.ok(host.lib.mhd_step(h, 1), h)
    ops = host.log()
    after = _reaches(ops)
    fft = [i for i, o in enumerate(ops) if o[0] == "launch" and ("rows_" in o[1] or "cols_" in o[1])]
    assert len(fft) == 3 * fft_kernels
    at = {}  # where each event is recorded first; a timer's two events are created together
    for i, o in enumerate(ops):
        if o[0] == "record":
            at.setdefault(int(o[1], 16), i)
    rules = [i for i, o in enumerate(ops) if o[0] == "launch" and "bc_kernel" in o[1]]
    assert len(rules) == 3
    for sub in range(3):
        ks = fft[sub * fft_kernels:(sub + 1) * fft_kernels]
        a = max(e for e, i in at.items() if i < ks[0] and e + 0x10 in at and at[e + 0x10] > ks[0])
        start, end = at[a], at[a + 0x10]
        assert all(after(start, k) and after(k, end) for k in ks)
        assert not any(after(start, r) and after(r, end) for r in rules)
    host.lib.mhd_destroy(h)
