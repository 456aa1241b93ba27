"""The batched volume kernels' CTAs walk several tiles of the work table, reusing their shared
memory and their barrier at alternating parity.  Meshes large enough that with one round of
resident CTAs (the autotuner left out, so the grid is known: at most 4 CTAs of two-element
tiles on each of 152 SMs) every CTA takes at least three tiles, with an odd number of elements
for a partial last tile: bitwise the state of a single handle, whose launches give each tile a
CTA of its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CUBE = dict(lo=(0.0, 0.0, 0.0), hi=(1000.0, 1000.0, 1000.0))


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_every_cta_walks_several_tiles(lib, monkeypatch, precision):
    monkeypatch.setenv("ES_DG_BATCH_VARIANT", "0")
    K, N = (17, 17, 15), 4
    assert (K[0] * K[1] * K[2] + 1) // 2 >= 3 * 4 * 152
    srv = lib.Server()
    out = srv.wait(srv.submit(kind="bubble", K=K, N=N, precision=precision, nsteps=2, warp=0.05), 300)
    srv.close()
    assert out["status"] == 0
    s = lib.Solver(*K, N, precision=precision, warp=0.05, **CUBE)
    s.init_bubble()
    s.step(out["dt"], 2)
    s.sync()
    assert np.array_equal(s.get_state().ravel(), out["q"])
