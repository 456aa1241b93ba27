"""The FP64 volume kernel at N = 6 and 7 has a second build for meshes of no more elements
than SMs (152 on this GPU).  Same source, and the tolerance is that of the FP64 right-hand
side: 1e-12 of each variable's norm (momentum: the vector's) and 4 x 2^-53 of the norm of its
terms, against the long-double oracle at both sides of the line, for states on the fixed-point
paths and on the FP64 pairs."""
import numpy as np
import pytest

import oracle as O
from paper_2605_16684_gb300 import inputs

pytestmark = pytest.mark.gpu

BOX = dict(lo=(0.0, 0.0, 0.0), hi=(1000.0, 1000.0, 1000.0), dissipation=0)


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


@pytest.mark.parametrize("N", [6, 7])
@pytest.mark.parametrize("mach", [0.01, 1.2])
@pytest.mark.parametrize("K", [(1, 1, 1), (19, 4, 2), (17, 3, 3)])
def test_both_sides_of_the_line(lib, K, mach, N):
    s, o = lib.Solver(*K, N, warp=0.05, **BOX), O.Oracle(*K, N, warp=0.05, precision="long", **BOX)
    x, _, _ = o.geometry()
    f = inputs.perturbation_factors(x, BOX["lo"], BOX["hi"], 4, 3, kmin=1, kmax=1)
    rho, p = 1.2 * (1 + 1e-2 * f[3]), 1e5 * (1 + 1e-2 * f[0])
    u = [340.0 * mach * (0.5 + 0.4 * f[k]) for k in range(3)]
    q = np.empty((s.E, 5, s.np))
    q[:, 0] = rho
    for c in range(3):
        q[:, 1 + c] = rho * u[c]
    q[:, 4] = p / 0.4 + 0.5 * rho * sum(v * v for v in u) + rho * 9.81 * np.asarray(x[:, 2], float)
    r, ref, terms = s.rhs(q), np.asarray(o.rhs(q), float), o.rhs_scale(q)
    s.close()
    norm = [np.linalg.norm(ref[:, v]) for v in range(5)]
    norm[1] = norm[2] = norm[3] = np.sqrt(sum(norm[c] ** 2 for c in (1, 2, 3)))
    for v in range(5):
        err = np.linalg.norm(r[:, v] - ref[:, v])
        assert err <= 1e-12 * norm[v] + 4 * 2.0 ** -53 * np.linalg.norm(terms[:, v]), (v, err)
