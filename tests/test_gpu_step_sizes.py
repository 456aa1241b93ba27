"""Stage launches with steps at the ends of the range.  A step of zero and steps too small
to change any value leave the state as it was, bit for bit (the increment is zero, or below
half a unit of the last place of every value); an infinite step is reported, not passed
over.  Both precisions, states that take the FP64 volume kernel's fixed-point pairs and one
that takes its FP64 pairs."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GAMMA, GRAV = 1.4, 9.81


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


def _solver(lib, precision, mach, N, warp):
    s = lib.Solver(3, 2, 2, N, precision=precision, warp=warp)
    x, _, _ = s.geometry()
    w = 1.0 + 0.01 * np.sin(2 * math.pi * x[:, 0] / 1000.0)
    rho, u = 1.2 * w, mach * 340.0 * w
    q = np.zeros((s.E, 5, s.np))
    q[:, 0], q[:, 1], q[:, 2], q[:, 3] = rho, rho * u, 0.5 * rho * u, -0.5 * rho * u
    q[:, 4] = 1e5 * w / (GAMMA - 1) + 0.75 * rho * u * u + rho * GRAV * x[:, 2]
    s.set_state(q)
    return s, q


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("mach", [0.01, 1.5])
@pytest.mark.parametrize("N,warp", [(1, 0.0), (4, 0.05), (7, 0.0)])
@pytest.mark.parametrize("dt", [0.0, -0.0, 5e-324, 1e-310, 1e-300, 1e-30])
def test_steps_too_small_to_matter(lib, precision, mach, N, warp, dt):
    s, q = _solver(lib, precision, mach, N, warp)
    s.launch(0)
    s.launch(2, 0, dt)
    s.sync()
    assert np.array_equal(s.get_state(), q)
    s.close()


@pytest.mark.parametrize("mach", [0.01, 1.5])
def test_infinite_step_is_reported(lib, mach):
    s, _ = _solver(lib, "fp64", mach, 4, 0.05)
    s.step(math.inf, 1)
    with pytest.raises(lib.EsDgError) as e:
        s.sync()
    assert e.value.code == -4
    s.close()
