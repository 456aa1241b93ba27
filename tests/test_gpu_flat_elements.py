"""The FP64 right-hand side on elements far from cubes against the long-double oracle, each
variable and each momentum component against its own terms.  Without dissipation every
term is a product of a few rounded factors, so the bar is 4 x 2^-53 of the norm of the
terms (or_rhs_scale), the floor that the FP64 right-hand side has on other meshes; nothing
is granted on top of it.  The volume kernel's fixed-point pairs hold an element's metric and
velocity in limbs of a few common scales: their aspect ratio, the balance of the fluxes
through the small and the large faces, and both sides of the rule that gives an element to
the FP64 pairs."""
import numpy as np
import pytest

import oracle as O
from paper_2605_16684_gb300 import inputs

pytestmark = pytest.mark.gpu

GAMMA, GRAV = 1.4, 9.81


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


def check(lib, size, u, N, warp=0.0):
    """Elements of size (dx, dy, dz), velocities up to u = (u, v, w)."""
    K = (3, 2, 2)
    hi = tuple(k * d for k, d in zip(K, size))
    box = dict(lo=(0.0, 0.0, 0.0), hi=hi, warp=warp, dissipation=0)
    s, o = lib.Solver(*K, N, **box), O.Oracle(*K, N, precision="long", **box)
    x, _, _ = o.geometry()
    f = inputs.perturbation_factors(x, box["lo"], hi, 4, 3, kmin=1, kmax=1)
    z = np.asarray(x[:, 2], float)
    rho = 1.2 * np.exp(-z / 8000.0) * (1 + 1e-3 * f[3])
    p = rho * 287.0 * 300.0 * (1 + 1e-3 * f[0])
    vel = [u[0] * (1 + 0.3 * f[0]), u[1] * (0.6 + 0.3 * f[1]), u[2] * f[2]]
    q = np.empty((s.E, 5, s.np))
    q[:, 0] = rho
    for c in range(3):
        q[:, 1 + c] = rho * vel[c]
    q[:, 4] = p / (GAMMA - 1) + 0.5 * rho * sum(v * v for v in vel) + rho * GRAV * z
    r, ref, terms = s.rhs(q), np.asarray(o.rhs(q), float), o.rhs_scale(q)
    s.close()
    for v in range(5):
        err = np.linalg.norm(r[:, v] - ref[:, v])
        assert err <= 4 * 2.0 ** -53 * np.linalg.norm(terms[:, v]), (v, err)


@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("aspect", [1.0, 3.0, 30.0, 1e3, 1e4, 1e5])
def test_aspects(lib, aspect, N):
    check(lib, (10.0 * aspect, 10.0 * aspect, 10.0), (10.0, 10.0, 10.0 / aspect), N)


@pytest.mark.parametrize("warp", [0.0, 1e-4])
@pytest.mark.parametrize("N", [3, 5])
def test_channel_elements(lib, N, warp):
    # 500 km x 375 km x 3.75 km, stratified (density falling by a third)
    check(lib, (500e3, 375e3, 3750.0), (30.0, 30.0, 0.01), N, warp)


@pytest.mark.parametrize("w", [0.0, 1e-9, 0.1, 0.5, 1.0, 1.5, 2.0, 3.0, 50.0])
@pytest.mark.parametrize("N", [2, 4])
def test_fluxes_through_the_large_faces(lib, N, w):
    # 1 km x 1 km x 10 m: w = 0.1 balances u = 10; from w = 1 to 3 the stretched velocity
    # passes the rule's line
    check(lib, (1000.0, 1000.0, 10.0), (10.0, 10.0, w), N)


@pytest.mark.parametrize("size,u", [((2e4, 20.0, 20.0), (10.0, 0.01, 0.01)),
                                    ((2e4, 20.0, 20.0), (10.0, 10.0, 10.0)),
                                    ((20.0, 20.0, 2e4), (0.01, 0.01, 10.0)),
                                    ((20.0, 20.0, 2e4), (1.0, 1.0, 10.0)),
                                    ((1e5, 20.0, 1e5), (10.0, 0.002, 10.0)),
                                    ((1e5, 1e3, 20.0), (10.0, 0.1, 0.002)),
                                    ((1e5, 1e3, 20.0), (10.0, 10.0, 0.01)),
                                    ((1e-3, 1e-3, 1e-6), (10.0, 10.0, 0.01)),
                                    ((1e9, 1e9, 1e3), (10.0, 10.0, 1e-5))])
@pytest.mark.parametrize("N", [4, 6])
def test_other_shapes(lib, N, size, u):
    check(lib, size, u, N)
