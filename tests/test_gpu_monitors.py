"""The CFL bound (FP32 screen, FP64 near the maximum) and the integrals (table logarithm)
against the oracle: orders, ragged element counts, and states that the screen must hand to
FP64 as a whole.  Bars: 1e-13 relative for the CFL step (both evaluate the same FP64
expression at the same node), 1e-12 for the integrals (round-off of sums of up to 1e5 terms).
"""
import numpy as np
import pytest

import oracle as O
from paper_2605_16684_gb300 import inputs

pytestmark = pytest.mark.gpu

CUBE = dict(lo=(0.0, 0.0, 0.0), hi=(1000.0, 1000.0, 1000.0))


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


@pytest.mark.parametrize("K,N", [((1, 1, 1), 1), ((3, 2, 1), 2), ((5, 7, 3), 3), ((9, 8, 7), 4),
                                 ((33, 1, 1), 5), ((2, 3, 2), 6), ((3, 3, 3), 7)])
def test_orders_and_ragged_counts(lib, K, N):
    s = lib.Solver(*K, N, warp=0.05, **CUBE)
    o = O.Oracle(*K, N, warp=0.05, **CUBE)
    x, _, _ = o.geometry()
    q = inputs.perturb_state(o.bubble(), x, CUBE["lo"], CUBE["hi"], seed=N)
    s.set_state(q)
    assert s.cfl_dt(0.5) == pytest.approx(o.cfl_dt(q, 0.5), rel=1e-13)
    assert np.allclose(s.integrals(), o.integrals(q), rtol=1e-12, atol=0)


@pytest.mark.parametrize("kind", ["supersonic", "vacuum", "huge", "one_nan", "ties"])
def test_states_beyond_the_screen(lib, kind):
    s = lib.Solver(5, 4, 3, 4, warp=0.05 if kind != "ties" else 0.0, **CUBE)
    o = O.Oracle(5, 4, 3, 4, warp=0.05 if kind != "ties" else 0.0, **CUBE)
    q = o.bubble(amp=0.0)
    ref = q.copy()
    if kind == "supersonic":  # one element at Mach 20
        u = 7000.0
        q[17, 1] = q[17, 0] * u
        q[17, 4] += 0.5 * q[17, 0] * u * u
        ref = q
    elif kind == "vacuum":  # a node of almost no pressure: not the maximum
        x, _, _ = o.geometry()
        q[3, 4, 11] = q[3, 0, 11] * 9.81 * x[3, 2, 11] + 1e-6
        ref = q
    elif kind == "huge":  # energies beyond the float range
        q[:, 4] *= 1e60
        ref = q
    elif kind == "one_nan":  # a node without a signal speed is left out
        q[8, 4, 5] = np.nan
    s.set_state(q)
    assert s.cfl_dt(0.5) == pytest.approx(o.cfl_dt(ref, 0.5), rel=1e-13)


def test_logarithm_over_its_range(lib):
    # densities and pressures over many binades in one mesh: the entropy integral
    s = lib.Solver(4, 3, 2, 3, g=0.0, **CUBE)
    o = O.Oracle(4, 3, 2, 3, g=0.0, **CUBE)
    rng = np.random.default_rng(1)
    q = np.zeros(o.shape())
    q[:, 0] = 2.0 ** rng.uniform(-30, 30, q[:, 0].shape)
    q[:, 4] = 2.0 ** rng.uniform(-30, 30, q[:, 0].shape) / 0.4
    s.set_state(q)
    assert np.allclose(s.integrals(), o.integrals(q), rtol=1e-12, atol=0)
