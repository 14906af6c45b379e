"""Which call reports a bounded device wait that ran out.  A kernel that gives up
stores to a word of its lattice's handle; here the test stores to it (through an
accessor that only tests use), so no wait runs out on the GPU.  The first call on
that handle reports it, whichever it is, and no other handle does; the lattice
has no state then until a new one is set."""
import ctypes

import numpy as np
import pytest

import paper_1703_00185_gb300 as lbm
from paper_1703_00185_gb300 import serving

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_00185_gb300 import _build
    _build.build()
    lib = lbm.load_library()
    lib.d2q37_late_word.restype = ctypes.POINTER(ctypes.c_uint)
    lib.d2q37_late_word.argtypes = [ctypes.c_void_p]
    lib.d2q37_server_job_handle.restype = ctypes.c_void_p
    lib.d2q37_server_job_handle.argtypes = [ctypes.c_void_p, ctypes.c_int64]
    return lib


def lattice(precision="fp64", seed=1):
    lat = lbm.Lattice(20, 40, precision=precision, device="cuda:0")
    lat.init_rayleigh_taylor(seed)
    lat.step(3)
    lat.synchronize()
    return lat


def late(lib, h):
    lib.d2q37_late_word(h)[0] = 1


CALLS = {
    "synchronize": lambda lat: lat.synchronize(),
    "fields": lambda lat: lat.fields(),
    "fields_device": lambda lat: lat.fields_device(),
    "populations": lambda lat: lat.populations(),
    "step": lambda lat: lat.step(1),
    "graph steps": lambda lat: lat.step(40),
    "run_phases": lambda lat: lat.run_phases(1, lbm.PHASE_ALL),
    "set_timing": lambda lat: lat.set_timing(True),
    "kernel_times": lambda lat: lat.kernel_times(),
    "batch": lambda lat: lbm.Batch([lat]),
    "static": lambda lat: lbm.lbm_batch_step_static([lat._h], 1, 0),
}


@pytest.mark.parametrize("precision", ["fp64", "fp32-df"])
@pytest.mark.parametrize("call", sorted(CALLS))
def test_first_call_reports(lib, call, precision):
    lat, other = lattice(precision), lattice(precision, 2)
    expect = lattice(precision).populations()
    late(lib, lat._h)
    for quiet in ("synchronize", "fields", "populations", "step", "kernel_times"):  # another handle
        CALLS[quiet](other)
    with pytest.raises(lbm.LBMError) as e:
        CALLS[call](lat)
    assert e.value.code == lbm.LBM_ETIMEOUT
    lat.synchronize()  # reported once
    for refused in ("step", "fields", "populations"):
        with pytest.raises(lbm.LBMError) as e:
            CALLS[refused](lat)
        assert e.value.code == lbm.LBM_ESTATE
    lat.init_rayleigh_taylor(1)
    lat.step(3)
    assert np.array_equal(lat.populations(), expect)


def test_a_new_state_drops_an_earlier_time_out(lib):
    lat = lattice()
    f = lat.populations()
    late(lib, lat._h)
    lat.set_populations(f)
    assert np.array_equal(lat.populations(), f)
    late(lib, lat._h)
    lat.init_rayleigh_taylor(4)
    lat.step(1)
    lat.synchronize()


def test_batch_reports_its_lattices(lib):
    lats = [lattice(seed=s) for s in range(3)]
    b = lbm.Batch(lats)
    b.step(5)
    b.synchronize()
    late(lib, lats[1]._h)
    with pytest.raises(lbm.LBMError) as e:
        b.synchronize()
    assert e.value.code == lbm.LBM_ETIMEOUT
    b.synchronize()
    lats[0].populations(), lats[2].populations()
    with pytest.raises(lbm.LBMError) as e:
        lats[1].fields()
    assert e.value.code == lbm.LBM_ESTATE
    late(lib, lats[2]._h)  # and one the batch did not look for
    with pytest.raises(lbm.LBMError) as e:
        lats[2].fields()
    assert e.value.code == lbm.LBM_ETIMEOUT


@pytest.mark.parametrize("when", ["stepping", "waiting for its fields"])
def test_server_ends_the_job_and_no_other(lib, when):
    server = serving.Server(64 << 20, max_steps_per_tick=4)
    ids = [server.submit(24, 40, 16, seed=s) for s in (1, 2)]
    for _ in range(2 if when == "stepping" else 4):
        server.tick()
    h = lib.d2q37_server_job_handle(server._h, ids[0])
    assert h
    late(lib, h)
    done = []
    for _ in range(50):
        server.tick()
        done += server.poll()
    assert sorted(done) == ids
    with pytest.raises(lbm.LBMError) as e:
        server.fetch(ids[0])
    assert e.value.code == lbm.LBM_ETIMEOUT
    rho, u, T = server.fetch(ids[1])
    lat = lbm.Lattice(24, 40, device="cuda:0")
    lat.init_rayleigh_taylor(2)
    lat.step(16)
    assert all(np.array_equal(a, b) for a, b in zip((rho, u, T), lat.fields()))
