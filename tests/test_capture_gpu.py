"""A caller's own CUDA graph over ``Solver.step``: replays between uncaptured
calls continue from the state those leave, as single launches would."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


def _solver(nx, ny, precision):
    from paper_1309_6726_gb300 import inputs as I, lbm
    g = I.random_lattice(nx, ny, seed=nx)
    # (no growth: the host's step count runs ahead of a captured call's)
    return lbm.Solver(g, I.ModelParams(g_ads=0.3, k_r=0.0, inlet=1), precision)


@pytest.mark.parametrize("n", [24, 25, 514, 536, 600, 1025, 1027])
@pytest.mark.parametrize("nx,ny,precision", [(131, 13, "fp16"), (256, 32, "fp32")])
def test_replay_after_uncaptured_steps(nx, ny, precision, n):
    import torch
    stream = torch.cuda.Stream()
    with _solver(nx, ny, precision) as s, _solver(nx, ny, precision) as ref:
        s.set_stream(stream.cuda_stream)
        s.step(2)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            s.step(2)
        with torch.cuda.stream(stream):
            graph.replay()
        s.step(n)
        if n % 2:  # (back to the buffer that the capture reads)
            s.step(1)
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        ref.step(6 + n + n % 2)
        np.testing.assert_array_equal(s.populations(), ref.populations())
