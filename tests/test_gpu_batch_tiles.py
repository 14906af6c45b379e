"""Batched steps with one block per tile (GPU, through the C ABI) beyond the
sizes of the other batch tests: more lattices than one collision's constants
serve, each with its own tau and g, walls and periodic ones mixed, the owner of
a tile from the per-tile table (a batch) and from a search (the call without
device allocation); batches of so many sites that their populations are staged
in shared memory; and more lattices than a launch's parameters hold.  Every
lattice ends bit-identical to the same one alone."""
import numpy as np
import pytest

import paper_1703_00185_gb300 as lbm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_00185_gb300 import _build
    _build.build()
    lbm.load_library()


def make(n, precision, shared):
    r = np.random.default_rng(n)
    lats = []
    for i in range(n):
        lat = lbm.Lattice(int(r.integers(3, 30)), int(r.integers(6, 300)), tau=0.8 if shared else 0.75 + 0.005 * i,
                          g0=1e-4 if shared else 1e-6 * i, T_bot=1.3, precision=precision, periodic_y=i % 3 == 2,
                          device="cuda:0")
        lat.init_rayleigh_taylor(i)
        lats.append(lat)
    return lats


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32-df"])
@pytest.mark.parametrize("n,shared", [(1, True), (70, False), (70, True), (140, False)])
def test_tiles_of_many_lattices(n, shared, precision):
    import torch
    alone, batched, static = (make(n, precision, shared) for _ in range(3))
    for lat in alone:
        lat.step(5)
    b = lbm.Batch(batched)  # the default shape: 128 rows a tile
    b.step(5)
    b.synchronize()
    assert b.launch_count == 5
    stream = torch.cuda.Stream(device="cuda:0")
    for lat in static:
        lat.synchronize()
    lbm.lbm_batch_step_static([lat._h for lat in static], 5, stream.cuda_stream)
    stream.synchronize()
    for a, c, d in zip(alone, batched, static):
        f = a.populations()
        assert np.array_equal(f, c.populations()) and np.array_equal(f, d.populations())
    b.close()


# One lattice that makes the batch large, and others whose tiles have every kind of remainder
STAGED = [(1024, 1300, False), (37, 257, True), (5, 6, False), (40, 129, True), (3, 300, False), (64, 66, False),
          (70, 260, False), (21, 512, True)]


def large(shared):
    lats = []
    for i, (Lx, Ly, periodic) in enumerate(STAGED):
        lat = lbm.Lattice(Lx, Ly, tau=0.8 if shared else 0.75 + 0.02 * i, g0=1e-4 if shared else 1e-5 * (i + 1),
                          T_bot=1.3, periodic_y=periodic, device="cuda:0")
        lat.init_rayleigh_taylor(i)
        lats.append(lat)
    return lats


@pytest.mark.parametrize("shared", [True, False])
def test_staged_tiles(shared):
    """FP64 tiles take the staged form above a number of warps of rows per SM."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert sum(Lx * ((Ly + 31) // 32) for Lx, Ly, _ in STAGED) > 250 * sms
    alone, batched, static = (large(shared) for _ in range(3))
    b = lbm.Batch(batched)
    stream = torch.cuda.Stream(device="cuda:0")
    for block_y in (64, 128, 256):
        for lat in alone:
            lat.step(3)
        b.set_config(block_y, 0)
        b.step(3)
        b.synchronize()
        if block_y == 128:  # six steps so far
            for lat in static:
                lat.synchronize()
            lbm.lbm_batch_step_static([lat._h for lat in static], 6, stream.cuda_stream)
            stream.synchronize()
        for k, (a, c) in enumerate(zip(alone, batched)):
            f = a.populations()
            assert np.array_equal(f, c.populations()), (block_y, STAGED[k])
            if block_y == 128:
                assert np.array_equal(f, static[k].populations()), STAGED[k]
    b.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32-df"])
def test_more_lattices_than_one_launch_holds(precision):
    alone, batched = ([], [])
    for lats in (alone, batched):
        for i in range(390):
            lat = lbm.Lattice(3 + i % 5, 6 + i % 11, tau=0.7 + 1e-3 * i, precision=precision, periodic_y=i % 4 == 3,
                              device="cuda:0")
            lat.init_rayleigh_taylor(i)
            lats.append(lat)
    for lat in alone:
        lat.step(5)
    b = lbm.Batch(batched)
    b.step(5)
    b.synchronize()
    assert b.launch_count == 5
    for a, c in zip(alone, batched):
        assert np.array_equal(a.populations(), c.populations())
    b.close()
