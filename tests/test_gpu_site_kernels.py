"""The forms of the FP64 fused sites kernel (GPU, through the C ABI): the
populations staged in shared memory by bulk copies, in tiles of 256 rows, and
the one for small lattices (all warps resident: at most 8 x SMs warps of 32
rows) that takes them into registers.  The default schedule picks one by the
lattice's size and chains the kernels; the serial schedule always runs the
staged one.  Their results are the same bit for bit, at the edges of tiles, on
both sides of the rule, with sites inside and outside the fixed-point ranges."""
import numpy as np
import pytest

import oracle
import paper_1703_00185_gb300 as lbm
from tests import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_00185_gb300 import _build
    _build.build()
    lbm.load_library()


def initial(Lx, Ly, wild):
    cx, cy = lbm.lbm_velocity_set()
    ocx, ocy = oracle.velocity_set()
    at = {(a, b): i for i, (a, b) in enumerate(zip(ocx.tolist(), ocy.tolist()))}
    perm = np.array([at[(a, b)] for a, b in zip(cx.tolist(), cy.tolist())])
    o = oracle.Lattice(Lx, Ly, tau=0.9, g0=1e-3)
    rho, u, T = ((0.3, 5.0), 0.5, (0.3, 2.4)) if wild else ((0.8, 1.2), 0.05, (0.5, 1.5))
    o.set_equilibrium(*synthetic.random_fields(Lx, Ly, 3, rho=rho, u=u, T=T))
    f = o.populations()[perm]
    if wild:  # zeros, a population above the rest one, tiny values of both signs
        r = np.random.default_rng(1)
        f[r.integers(37, size=40), r.integers(Lx, size=40), r.integers(Ly, size=40)] *= r.choice([0.0, 1e3, 1e-12, -1e-12], 40)
    return f


@pytest.mark.parametrize("wild", [False, True])
@pytest.mark.parametrize("Lx,Ly", [(3, 6), (7, 255), (5, 256), (6, 257), (4, 513), (38, 1024), (39, 1024), (150, 257)])
@pytest.mark.parametrize("periodic_y", [False, True])
def test_forms_agree_bit_for_bit(Lx, Ly, periodic_y, wild):
    f = initial(Lx, Ly, wild)
    out = []
    for kernel in ("fused", "fused_serial"):
        lat = lbm.Lattice(Lx, Ly, tau=0.9, g0=1e-3, periodic_y=periodic_y, kernel=kernel, device="cuda:0")
        lat.set_populations(f)
        lat.step(1 if wild else 5)
        out.append(lat.populations())
    assert np.array_equal(out[0], out[1])
    if not wild and not periodic_y and Lx >= 7:  # and the separate kernels, to rounding
        lat = lbm.Lattice(Lx, Ly, tau=0.9, g0=1e-3, kernel="separate", device="cuda:0")
        lat.set_populations(f)
        lat.step(5)
        assert np.max(np.abs(lat.populations() - out[0])) <= 1e-15 * 5


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32-df"])
@pytest.mark.parametrize("Lx,Ly", [(3, 6), (5, 257), (38, 1024), (130, 257)])
def test_long_chains_equal_the_serial_schedule(Lx, Ly, precision):
    """Steps that start in the tail of the one before them, and a read-out behind
    them, see everything those wrote: 203 steps, with single ones between."""
    out = []
    for kernel in ("fused", "fused_serial"):
        lat = lbm.Lattice(Lx, Ly, kernel=kernel, precision=precision, device="cuda:0")
        lat.init_rayleigh_taylor(7)
        got = []
        for n in (1, 1, 1, 100, 100):
            lat.step(n)
            got += list(lat.fields())
        out.append(got + [lat.populations()])
    assert all(np.array_equal(a, b) for a, b in zip(*out))


# (Lx, Ly) on both sides of every rule that picks a form, and blocks whose last one is nearly empty
FORMS = [(3, 9), (64, 64), (227, 34), (1000, 16), (2000, 35), (76, 512), (100, 512), (142, 515), (152, 515),
         (130, 257), (130, 260), (256, 196), (400, 100), (500, 516), (470, 262), (460, 191), (40, 1030), (1450, 512),
         (1450, 470)]


@pytest.mark.parametrize("Lx,Ly", FORMS)
@pytest.mark.parametrize("periodic_y", [False, True])
def test_every_form_gives_the_same_bits(Lx, Ly, periodic_y):
    """One lattice chained, serial, in a batch of one launch per lattice and with
    separate kernels, each in the form its rule picks, against the batch's table
    kernel (one register form for every size)."""
    f = initial(Lx, Ly, False)
    out = []
    for kernel, config in (("fused", (128, 1)), ("fused", (0, 0)), ("fused", None), ("fused_serial", None),
                           ("separate", None)):
        lat = lbm.Lattice(Lx, Ly, tau=0.9, g0=1e-3, periodic_y=periodic_y, kernel=kernel, device="cuda:0")
        lat.set_populations(f)
        if config:
            b = lbm.Batch([lat])
            b.set_config(*config)
            b.step(5)
            b.synchronize()
            b.close()
        else:
            lat.step(5)
        out.append(lat.populations())
    for got in out[1:]:
        assert np.array_equal(got, out[0])
