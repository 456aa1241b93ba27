"""The launches of a step start before the ones they depend on have ended and wait on the
device.  A step gives bitwise what the same kernels give launched one by one, each after a
synchronisation, and what they give captured in a CUDA graph: same kernels, same order, so
the tolerance is zero.  Sizes: fewer face nodes than one CTA, a ragged last CTA, several
waves."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2605_16684_gb300 import _build, _lib
    _build.build()
    return _lib


def _state(s):
    return s.get_state(torch.empty(s.shape(), dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("K,N", [((1, 1, 1), 1), ((5, 3, 2), 4), ((13, 9, 7), 3), ((24, 24, 24), 4),
                                 ((6, 5, 4), 7)])
def test_step_is_its_stages(lib, K, N, precision):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        s = lib.Solver(*K, N, warp=0.05, precision=precision, stream=stream)
        s.init_bubble()
        q0 = _state(s)
        dt = s.cfl_dt(0.5)
        for _ in range(3):
            for stage in range(5):
                for which in (0, 2):
                    s.launch(which, stage, dt)
                    stream.synchronize()
        one_by_one = _state(s)
        s.set_state(q0)
        s.step(dt, 3)
        together = _state(s)
        s.sync()
        assert not torch.equal(one_by_one, q0)
        assert torch.equal(one_by_one, together)
        s.set_state(q0)
        s.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            s.step(dt, 1)
        for _ in range(3):
            graph.replay()
        assert torch.equal(one_by_one, _state(s))
        s.sync()
