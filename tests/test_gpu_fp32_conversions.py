"""FP32 storage with FP64 wide terms converts between FP64 and FP32 by integer
operations (round to nearest even, infinities and NaN kept).  Through the C
ABI: deviations that become infinite or NaN stay so and stay where they are,
and one collision from states over a wide range of densities agrees with the
double-float form, whose conversions are additions, to FP32 rounding."""
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


def collided(f, precision):
    lat = lbm.Lattice(f.shape[1], f.shape[2], tau=0.9, precision=precision, kernel="separate", device="cuda:0")
    lat.set_populations(f)
    lat.run_phases(1, lbm.PHASE_COLLIDE)
    return lat.populations()


@pytest.mark.parametrize("scale", [1e-3, 0.5, 1.0, 3.0, 40.0])
def test_agrees_with_double_float(scale):
    _, w = lbm.lbm_quadrature()
    r = np.random.default_rng(5)
    f = scale * w[:, None, None] * (1.0 + 0.02 * (2.0 * r.random((37, 20, 70)) - 1.0))
    f[:, 3, :] = scale * w[:, None]  # at rest: u and q exactly 0
    a, b = collided(f, "fp32"), collided(f, "fp32-df")
    # a population is a deviation from w rounded to FP32 (2^-24 of w + f) after
    # terms of up to ~10 w rho; each form is within a few such roundings
    bound = 40 * 2.0**-24 * (w[:, None, None] + np.abs(b))
    assert np.all(np.abs(a - b) <= bound + 40 * 2.0**-24 * scale * w[:, None, None])


def test_infinities_and_nan_stay_at_their_site():
    _, w = lbm.lbm_quadrature()
    f = np.ones((37, 12, 40)) * w[:, None, None]
    ref = collided(f, "fp32")
    for (x, y), v in zip([(2, 5), (4, 33), (7, 12)], [np.inf, np.nan, 1e30]):
        f[5, x, y] = v
    got = collided(f, "fp32")
    bad = np.zeros((12, 40), bool)
    bad[[2, 4, 7], [5, 33, 12]] = True
    assert np.array_equal(got[:, ~bad], ref[:, ~bad])
    assert not np.isfinite(got[:, 2, 5]).any() and np.isnan(got[:, 4, 33]).any()
