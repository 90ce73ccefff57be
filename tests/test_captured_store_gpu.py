"""A velocity field whose only store was captured in a CUDA graph: the scalar steps after
its replay take several steps a launch, as after a store by itself."""
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


def test_strips_are_planned_with_the_first_scalar_steps():
    """The strips are device memory that the handle reports; captured steps may not plan
    them, later ones do."""
    s = torch.cuda.Stream()
    chips = [lbm.Chip.from_problem(W.config_small(), stream=s, torch_alloc=True) for _ in range(2)]
    for c in chips:
        c.set_valves(1)
        c.step(5)
        c.synchronize()
    without = chips[0].info()["device_bytes"]
    store, steps = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(store, stream=s):
        chips[0].store_velocity(1)
    with torch.cuda.stream(s):
        store.replay()
    field = chips[0].info()["device_bytes"] - without
    with torch.cuda.graph(steps, stream=s):
        chips[0].scalar_step(8)  # (8: the state ends where it began)
    assert chips[0].info()["device_bytes"] == without + field
    with torch.cuda.stream(s):
        steps.replay()
    chips[0].scalar_step(7)
    chips[1].store_velocity(1)
    chips[1].scalar_step(8)
    chips[1].scalar_step(7)
    assert chips[0].info()["device_bytes"] == chips[1].info()["device_bytes"] > without + field
    for a, b in zip(chips[0].populations(), chips[1].populations()):
        assert np.array_equal(a, b)
    for c in chips:
        c.close()
