"""lbm_step recorded in a CUDA graph of the caller's: an even number of steps with held
valves ends in the buffer it begins in, so the graph can be replayed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1307_4703_gb300 import lbm, workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1307_4703_gb300 import build
    build.build()
    lbm.load()


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("n", [2, 4, 6, 8, 100])
def test_replays_equal_direct_calls(n, precision):
    """Three replays give the bits of three calls: fields by populations, and totals."""
    s = torch.cuda.Stream()
    chips = [lbm.Chip.from_problem(W.config_small(), stream=s, precision=precision) for _ in range(2)]
    for c in chips:
        c.set_valves(1)
        c.step(5)
        c.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        chips[0].step(n)
    for _ in range(3):
        with torch.cuda.stream(s):
            graph.replay()
        chips[1].step(n)
    torch.cuda.synchronize()
    for a, b in zip(chips[0].populations(), chips[1].populations()):
        assert np.array_equal(a, b)
    assert np.array_equal(chips[0].diagnostics(), chips[1].diagnostics())
    for c in chips:
        c.step(7)  # the handle goes on from the replayed state
    for a, b in zip(chips[0].populations(), chips[1].populations()):
        assert np.array_equal(a, b)
    for c in chips:
        c.close()
