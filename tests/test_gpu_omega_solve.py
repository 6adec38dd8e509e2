"""The FP64 solve for omega_nu works on bit patterns in place of FP64
comparisons and logarithms: what it does outside the positive, finite range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def clbm():
    from paper_1908_05396_gb300 import build
    build.build()
    from paper_1908_05396_gb300 import clbm as c
    c.lib()
    return c


@pytest.mark.parametrize("n", [0.5, 0.9, 1.3, 1.8])
def test_no_rate_without_a_valid_density_and_moments(clbm, n):
    inf, nan = np.inf, np.nan
    rho = np.array([1.0, 0.7, -0.27, -1e-3, 0.0, -0.0, nan, -nan, inf, -inf] + [1.0] * 4)
    m = np.zeros((6, len(rho)))
    m[0] = 1e-3
    m[2, 10], m[5, 11], m[1, 12], m[5, 13] = nan, nan, inf, -inf
    w, gd = clbm.omega_nodes(rho, m, 1e-3, n, "f64")
    assert np.all(np.isfinite(w[:2]) & (w[:2] > 0) & (w[:2] < 2)) and np.all(gd[:2] > 0)
    assert np.all(np.isnan(w[2:]))


@pytest.mark.parametrize("in_place", [False, True])
def test_negative_density_spreads_and_is_reported(clbm, in_place):
    # one node of negative density: its collision leaves NaN, which its
    # neighbours pull in the next step, and the check step reports it
    kw = dict(face=(clbm.PERIODIC,) * 6, K=0.02, n=0.8, dtype="f64", check_interval=4)
    with clbm.Lattice(9, 8, 7, in_place=in_place, **kw) as lat:
        f = lat.get_state()
        for q, (x, y, z) in enumerate(_E):      # what node (4, 4, 3) pulls
            f[q, (3 - z) % 7, (4 - y) % 8, (4 - x) % 9] *= -0.27
        lat.set_state(f)
        lat.step(2)
        assert np.isnan(lat.get_state()).any(axis=0).sum() >= 19
        lat.step(2)
        assert lat.residual()[1] == clbm.ERR_DIVERGED


_E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1),
      (-1, 0, -1), (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n", [0.7, 1.0, 1.4])
def test_shear_rate_is_a_magnitude(clbm, n, dtype):
    # gamma_dot is the root of an invariant: the density's sign is not its own
    rho = np.array([-0.27, 0.27, -1.5, 1.5])
    m = np.tile(np.array([1e-3, -2e-3, 5e-4, 1e-3, 0.0, 2e-4])[:, None], 4)
    _, gd = clbm.omega_nodes(rho, m, 1e-3, n, dtype)
    assert np.all((gd > 0) | np.isnan(gd)) and np.all(gd[[1, 3]] > 0)


@pytest.mark.parametrize("n", [0.4, 0.8, 1.6, 2.0])
def test_shear_beyond_the_fp32_range_reaches_its_clamp(clbm, n):
    # invariants around and past the largest FP32 value: the viscosity lies on
    # the clamp that n decides, to the rounding of 1 / (3 nu + 1/2): a few 2^-53
    mag = 10.0 ** np.arange(15, 61, 2.5)
    rho = np.ones(len(mag))
    m = mag * np.array([1.0, -0.5, 0.3, 0.2, 0.1, 0.4])[:, None]
    w, _ = clbm.omega_nodes(rho, m, 1e-3, n, "f64")
    nu = 5e-4 if n < 1 else 10.0
    assert np.all(np.abs(w * (3 * nu + 0.5) - 1) <= 1e-15)
