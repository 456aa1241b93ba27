"""The FP64 right-hand side where the pressure is small beside the internal energy (gamma
near 1), the geopotential (a mesh far above z = 0, an element of several kilometres) or the
kinetic energy, against the long-double oracle: each variable and momentum component against
its own terms.  Without dissipation every term is a product of a few rounded factors, so the
bar is 4 x 2^-53 of the norm of the terms (or_rhs_scale).  The volume kernel's fixed-point
pairs hold the pressure at the scale of the energies or some bits above, and leave an
element whose scales do not fit to the FP64 pairs: gamma and temperature move an element
across both lines."""
import numpy as np
import pytest

import oracle as O
from paper_2605_16684_gb300 import inputs

pytestmark = pytest.mark.gpu

GRAV = 9.81


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


def check(lib, N, size=31.0, z0=0.0, gamma=1.4, T=300.0, u=5.0, fold=0.0, warp=0.0):
    K = (3, 3, 2)
    lo, hi = (0.0, 0.0, z0), (K[0] * size, K[1] * size, z0 + K[2] * size)
    box = dict(lo=lo, hi=hi, warp=warp, dissipation=0, gamma=gamma)
    s, o = lib.Solver(*K, N, **box), O.Oracle(*K, N, precision="long", **box)
    x, _, _ = o.geometry()
    f = inputs.perturbation_factors(x, lo, hi, 4, 3, kmin=1, kmax=1)
    z = np.asarray(x[:, 2], float)
    rho = 1.2 * np.exp(-fold * (z - z0) / size) * (1 + 1e-3 * f[3])
    p = rho * 287.0 * T * (1 + 1e-3 * f[0])
    vel = [u * (1 + 0.3 * f[0]), u * (0.6 + 0.3 * f[1]), u * f[2]]
    q = np.empty((s.E, 5, s.np))
    q[:, 0] = rho
    for c in range(3):
        q[:, 1 + c] = rho * vel[c]
    q[:, 4] = p / (gamma - 1) + 0.5 * rho * sum(v * v for v in vel) + rho * GRAV * z
    r, ref, terms = s.rhs(q), np.asarray(o.rhs(q), float), o.rhs_scale(q)
    s.close()
    for v in range(5):
        err = np.linalg.norm(r[:, v] - ref[:, v])
        assert err <= 4 * 2.0 ** -53 * np.linalg.norm(terms[:, v]), (v, err)


@pytest.mark.parametrize("N", [2, 4, 7])
@pytest.mark.parametrize("gamma", [1.001, 1.003, 1.005, 1.02, 1.1, 1.2, 5.0 / 3.0, 2.0])
def test_gamma(lib, N, gamma):
    check(lib, N, gamma=gamma)


@pytest.mark.parametrize("N", [1, 4, 6])
@pytest.mark.parametrize("z0", [-2e5, 1e3, 1e4, 5e4, 2e5])
def test_far_from_the_zero_of_the_geopotential(lib, N, z0):
    check(lib, N, z0=z0, warp=0.05 if z0 == 1e3 else 0.0)


@pytest.mark.parametrize("N", [3, 4, 5])
@pytest.mark.parametrize("size,T", [(2e3, 273.0), (5e3, 273.0), (7.5e3, 220.0), (7.5e3, 300.0),
                                    (1.1e4, 273.0)])
def test_tall_elements(lib, N, size, T):
    # density falling by size / 8 km over an element
    check(lib, N, size=size, T=T, fold=size / 8e3)


@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("T", [1.0, 260.0, 310.0, 323.0, 324.0, 400.0, 3e5])
def test_temperatures(lib, N, T):
    check(lib, N, T=T, u=0.05 * np.sqrt(T))


@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("u", [50.0, 90.0, 110.0, 125.0, 150.0, 200.0, 300.0, 1000.0])
def test_velocities(lib, N, u):
    check(lib, N, u=u)
