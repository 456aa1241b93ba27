"""A volume kernel's bounded wait that runs out (bytes that are registered on its barrier and
never copied, es_dg_debug_inject_wait_timeout) in the kernels without a background and with a
moving one: it is reported once, by any handle's sync, and the next step of the same handle is
right again."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CHANNEL = dict(lo=(0.0, 0.0, 0.0), hi=(40000e3, 6000e3, 30e3), periodic=(1, 0, 0), f0=1e-4)


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


def _solver(lib, kind):
    if kind == "jet":
        s = lib.Solver(6, 3, 2, 4, precision="mixed", **CHANNEL)
        s.init_channel(background="jet")
        return s
    s = lib.Solver(3, 3, 3, 4, precision="mixed" if kind == "none" else "fp64")
    s.init_bubble()
    if kind == "none":
        assert s.lib.es_dg_clear_background(s.h) == 0
    return s


@pytest.mark.parametrize("kind", ["none", "jet", "fp64"])
@pytest.mark.parametrize("other", [False, True])
def test_reported_once_and_cleared(lib, kind, other):
    s, ref = _solver(lib, kind), _solver(lib, kind)
    q0, dt = s.get_state(), s.cfl_dt(0.25)
    s.lib.es_dg_debug_inject_wait_timeout()
    s.step(dt, 1)
    s.get_state()  # waits for the step
    reader, bystander = (ref, s) if other else (s, ref)
    with pytest.raises(lib.EsDgError) as err:
        reader.sync()
    assert err.value.code == -5  # ES_DG_ETIMEOUT
    bystander.sync()
    s.set_state(q0)
    s.step(dt, 1)
    s.sync()
    ref.step(dt, 1)
    ref.sync()
    assert np.array_equal(s.get_state(), ref.get_state())
