"""Every instance of the two-step kernel: both block shapes of each storage type, with and
without ports of the rescaling kinds.  The plan says which shape a lattice takes (on the
CPU, for a GPU of 152 SMs); the populations have the bits of single steps."""
import numpy as np
import pytest

from paper_1307_4703_gb300 import lbm, workloads as W
from test_strip_plan import FP16, FP32, Plan, lib  # noqa: F401  (lib: the plan built for the CPU)

torch = pytest.importorskip("torch")

# precision, warps of a block, lattice
SHAPES = [("fp32", 4, 129, 47), ("fp32", 6, 400, 120), ("fp16", 6, 129, 47), ("fp16", 8, 1025, 90),
          ("bf16", 6, 129, 47), ("bf16", 8, 1025, 90)]


def _case(nx, ny, paper_ports):
    return W.random_case(nx + ny, nx, ny, paper_ports=paper_ports)


@pytest.mark.parametrize("paper_ports", [False, True])
@pytest.mark.parametrize("precision,warps,nx,ny", SHAPES)
def test_the_plan_takes_the_shape(lib, precision, warps, nx, ny, paper_ports):  # noqa: F811
    prob, _ = _case(nx, ny, paper_ports)
    p = Plan(lib, prob["solid"], prob["ports"], precision=FP32 if precision == "fp32" else FP16, rescale=paper_ports)
    assert p.worth and p.warps == warps


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("paper_ports", [False, True])
@pytest.mark.parametrize("precision,warps,nx,ny", SHAPES)
def test_bits_of_single_steps(precision, warps, nx, ny, paper_ports):
    from paper_1307_4703_gb300 import build
    build.build()
    prob, init = _case(nx, ny, paper_ports)
    single = dict(variant=1 if precision == "fp32" else 4, block_threads=128)
    chips = [lbm.Chip.from_problem(prob, precision=precision, **kw) for kw in ({}, single)]
    for c in chips:
        c.init_equilibrium(**init)
        c.set_valve_schedule(1, prob["states"])
    for n in (3, 8, 27):
        for c in chips:
            c.step(n)
        for a, b in zip(chips[0].populations(), chips[1].populations()):
            assert np.array_equal(a, b)
        assert np.array_equal(chips[0].diagnostics(), chips[1].diagnostics())
    for c in chips:
        c.close()
