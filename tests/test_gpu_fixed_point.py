"""The FP64 volume kernel's fixed-point pairs against the long-double oracle, at the
edges of their range and of the tiles.

Bar: 1e-12 relative L2 per variable (momentum against the momentum vector's norm), the
bar of the FP64 right-hand side on generic states, plus the round-off floor of the
right-hand side's cancelling terms, 4 * 2^-53 of their norm (or_rhs_scale).
"""
import numpy as np
import pytest

import oracle as O
from paper_2605_16684_gb300 import inputs

pytestmark = pytest.mark.gpu

# a 60 m box: hydrostatic variation of 0.5 % over the whole height, so that every
# element of a smooth state shares its first node's scales
BOX = dict(lo=(0.0, 0.0, 0.0), hi=(60.0, 60.0, 60.0))
GAMMA, GRAV = 1.4, 9.81


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


def check(lib, K, N, q_of, warp=0.05, **phys):
    s = lib.Solver(*K, N, warp=warp, **BOX, **phys)
    o = O.Oracle(*K, N, warp=warp, precision="long", **BOX, **phys)
    x, _, _ = o.geometry()
    q = q_of(o, x)
    r, ref, terms = s.rhs(q), o.rhs(q), o.rhs_scale(q)
    assert np.isfinite(r).all()
    mom = np.sqrt(sum(np.linalg.norm(ref[:, v]) ** 2 for v in (1, 2, 3)))
    for v in range(5):
        norm = mom if v in (1, 2, 3) else np.linalg.norm(ref[:, v])
        err = np.linalg.norm(r[:, v] - ref[:, v])
        assert err <= 1e-12 * norm + 4 * 2.0 ** -53 * np.linalg.norm(terms[:, v]), (v, err, norm)
    s.close()


def smooth(o, x):
    return inputs.perturb_state(o.bubble(amp=0.1, centre=(30.0, 30.0, 30.0), radius=20.0), x,
                                BOX["lo"], BOX["hi"], seed=5, eps=1e-3, kmin=1, kmax=1)


def state(rho, u, p, x):
    z = x[:, 2]
    q = np.empty((x.shape[0], 5, x.shape[2]))
    q[:, 0] = rho
    for c in range(3):
        q[:, 1 + c] = rho * u[c]
    q[:, 4] = p / (GAMMA - 1) + 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2) + rho * GRAV * z
    return q


@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("K", [(1, 1, 1), (5, 3, 1), (7, 5, 3)])
def test_every_order_and_ragged_tiles(lib, K, N):
    if N >= 6 and K == (7, 5, 3):
        K = (3, 3, 2)
    check(lib, K, N, smooth, f0=1e-4 if K == (5, 3, 1) else 0.0)


@pytest.mark.parametrize("ratio", [0.0, 1e-9, 0.0094, 0.0096, 0.03, 0.115, 0.125, 0.3])
def test_density_variation_across_the_series_range(lib, ratio):
    def q_of(o, x):
        t = x[:, 0] / 60.0
        return state(1.2 * (1 + ratio * t), (2.0 + t, -1.0 + 0 * t, t), 1e5 * (1 - 0.3 * ratio * t), x)
    check(lib, (1, 2, 1), 4, q_of, warp=0.0)


@pytest.mark.parametrize("fold", [0.13, 0.5, 1.0, 1.5, 1.56, 1.7])
@pytest.mark.parametrize("N", [3, 4, 7])
def test_stratified_elements_across_the_tall_range(lib, N, fold):
    # density falling by exp(-fold) over the element at a nearly uniform temperature
    def q_of(o, x):
        t = x[:, 2] / 60.0
        rho = 1.2 * np.exp(-fold * t)
        return state(rho, (2.0 + t, -1.0 + 0 * t, t), rho * 287.0 * (300.0 + 10.0 * t), x)
    check(lib, (2, 1, 1), N, q_of, warp=0.0)


def moving(mach):
    c = np.sqrt(GAMMA * 1e5 / 1.2)

    def q_of(o, x):
        f = inputs.perturbation_factors(x, BOX["lo"], BOX["hi"], 4, 3, kmin=1, kmax=1)
        u = [mach * c * (0.5 + 0.4 * f[k]) for k in range(3)]
        return state(1.2 * (1 + 1e-3 * f[3]), u, 1e5 * (1 + 1e-3 * f[0]), x)
    return q_of


@pytest.mark.parametrize("mach", [0.3, 0.62, 0.9, 3.0])
def test_velocities_to_supersonic(lib, mach):
    check(lib, (2, 3, 2), 4, moving(mach))


@pytest.mark.parametrize("mach", [1e-14, 1e-5])
def test_small_velocities(lib, mach):
    # without dissipation: near rest it is the interface's round-off that dominates the
    # mass right-hand side
    check(lib, (2, 3, 2), 4, moving(mach), dissipation=0)


def test_rest_has_no_mass_or_energy_flux(lib):
    s = lib.Solver(2, 3, 2, 4, warp=0.05, dissipation=0, **BOX)
    x, _, _ = s.geometry()
    r = s.rhs(moving(0.0)(None, x))
    assert not r[:, 0].any() and not r[:, 4].any()


@pytest.mark.parametrize("jump", [1.1, 30.0, 1e6])
def test_jumps_between_elements_outside_the_range_of_their_sums(lib, jump):
    # uniform elements, their densities and pressures a checkerboard: the interface
    # terms of the light elements exceed their own fluxes by the jump
    def q_of(o, x):
        e = np.arange(x.shape[0])
        odd = (e % 3 + (e // 3) % 2 + e // 6) % 2
        f = np.where(odd, jump, 1.0)[:, None] * np.ones_like(x[:, 0])
        return state(1.2 * f, (0 * f + 3.0, 0 * f, 0 * f - 1.0), 1e5 * f, x)
    check(lib, (3, 2, 2), 3, q_of)


def test_batched_and_single_launches_agree_bitwise(lib):
    # small bubbles on the 1000 m cube at N = 7: elements on both sides of the range in
    # one mesh, single-mesh tiles against the server's
    srv = lib.Server(8 << 30, 4)
    req = dict(kind="bubble", K=(9, 9, 9), N=7, precision="fp64", nsteps=3, cfl=0.3)
    out = srv.wait(srv.submit(**req), 300)
    srv.close()
    assert out["status"] == 0
    s = lib.Solver(9, 9, 9, 7, lo=(0, 0, 0), hi=(1000.0, 1000.0, 1000.0))
    s.init_bubble()
    s.step(out["dt"], 3)
    s.sync()
    assert np.array_equal(s.get_state().ravel(), out["q"])
