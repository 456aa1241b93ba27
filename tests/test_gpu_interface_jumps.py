"""The FP64 interface flux at jumps of every size against the long-double oracle: elements
whose densities, pressures and velocities differ by factors (logarithm branch) down to a
millionth (series branch), with and without the dissipation, at periodic faces and walls.
Bar: an interface value is about 150 operations on terms no larger than its largest, so
150 x 1.1e-16 and as much again for the five terms of a node's sum: 1e-13 of each
variable's largest value."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

CUBE = dict(lo=(0.0, 0.0, 0.0), hi=(1000.0, 1000.0, 1000.0))


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


@pytest.mark.parametrize("dissipation", [0, 1])
@pytest.mark.parametrize("size", [1.0, 1e-2, 1e-6])
@pytest.mark.parametrize("K,N,warp", [((3, 2, 4), 3, 0.05), ((2, 2, 3), 6, 0.0)])
def test_jumps(lib, K, N, warp, size, dissipation):
    s = lib.Solver(*K, N, warp=warp, dissipation=dissipation, **CUBE)
    o = O.Oracle(*K, N, precision="long", warp=warp, dissipation=dissipation, **CUBE)
    rng = np.random.default_rng(11)
    E, n = s.E, s.np
    x, _, _ = o.geometry()
    f = lambda: np.exp(size * rng.uniform(-0.7, 0.7, (E, 1)))
    rho, p = 1.1 * f() * np.ones((E, n)), 9.0e4 * f() * np.ones((E, n))
    u = 40.0 + 300.0 * size * rng.uniform(-1.0, 1.0, (E, 3, 1)) * np.ones((E, 3, n))
    q = np.empty((E, 5, n))
    q[:, 0] = rho
    q[:, 1:4] = rho[:, None] * u
    q[:, 4] = p / 0.4 + rho * (0.5 * (u ** 2).sum(1) + 9.81 * np.asarray(x, float)[:, 2])
    r, e = s.rhs(q), np.asarray(o.rhs(q), float)
    for v in range(5):
        assert np.abs(r[:, v] - e[:, v]).max() <= 1e-13 * np.abs(e[:, v]).max()
