"""Batched steps with one block per tile (GPU, through the C ABI) beyond the
sizes of the other batch tests: more lattices than one collision's constants
serve, each with its own tau and g, walls and periodic ones mixed, the owner of
a tile from the per-tile table (a batch) and from a search (the call without
device allocation).  Every lattice ends bit-identical to the same one alone."""
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
