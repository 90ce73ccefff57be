"""The FP32 register kernel stages its bounce-back entries in shared memory (lattices
without rescaling ports): the bits of the variant that loads them link by link, at
tile edges, for sparse to dense obstacles and blocks of every size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1307_4703_gb300 import lbm, workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("block", [64, 128, 256])
@pytest.mark.parametrize("nx,ny,solid_frac,paper_ports", [
    (4, 8, 0.0, False), (61, 9, 0.5, False), (128, 16, 0.2, False), (131, 40, 0.05, False), (515, 33, 0.3, True)])
def test_staged_bounce_back_is_the_plain_one(nx, ny, solid_frac, paper_ports, block):
    prob, init = W.random_case(nx + block, nx, ny, solid_frac=solid_frac, paper_ports=paper_ports)
    chips = [lbm.Chip.from_problem(prob, variant=v, block_threads=b) for v, b in ((1, block), (4, 128))]
    for c in chips:
        c.init_equilibrium(**init)
        c.set_valve_schedule(1, prob["states"])
        c.step(12)
    for a, b in zip(chips[0].populations(), chips[1].populations()):
        assert np.array_equal(a, b)
    for c in chips:
        c.close()
