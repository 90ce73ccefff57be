"""Two steps in one launch (the default of lbm_step): the populations are the bits
of single steps, at the edges of the strips, rows and blocks it is cut into."""
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


def _assert_same(pairs, single, runs):
    """After each run of steps: populations and diagnostics bit for bit (the last step
    of a call is a single one on both handles)."""
    for n in runs:
        pairs.step(n)
        single.step(n)
        for a, b in zip(pairs.populations(), single.populations()):
            assert np.array_equal(a, b)
        assert np.array_equal(pairs.diagnostics(), single.diagnostics())
    assert pairs.step_count() == single.step_count()
    pairs.close()
    single.close()


def _single(precision):
    """The same kernel one step a launch: the launch shape given instead of left to the
    library."""
    return dict(precision=precision, variant=1 if precision == "fp32" else 4, block_threads=128)


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("nx,ny,paper_ports,decay", [
    (4, 8, False, 0.0), (60, 9, True, 1e-3), (124, 13, False, 0.0), (125, 30, False, 1e-3), (128, 31, True, 0.0),
    (129, 47, False, 0.0), (244, 33, True, 0.0), (249, 40, False, 0.0), (513, 64, False, 1e-3)])
def test_random_lattices(nx, ny, paper_ports, decay, precision):
    """Obstacles, every port kind and another valve word each step; one strip to several
    with a partial last one, fewer rows than a block's warps to many."""
    prob, init = W.random_case(nx + ny, nx, ny, paper_ports=paper_ports, decay=decay)
    chips = [lbm.Chip.from_problem(prob, **kw) for kw in (dict(precision=precision), _single(precision))]
    for c in chips:
        c.init_equilibrium(**init)
        c.set_valve_schedule(1, prob["states"])
    _assert_same(*chips, (3, 4, 7, 1, 2, 20))


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("nx,ny", [(256, 128), (777, 401), (2100, 1000)])
def test_two_channel_chips(nx, ny, precision):
    """Side walls of channels and chamber within the strips, valves toggling between the
    steps of a pair (odd period)."""
    prob = W.config_large_chip(nx, ny)
    chips = [lbm.Chip.from_problem(prob, **kw) for kw in (dict(precision=precision), _single(precision))]
    for c in chips:
        c.set_valve_schedule(13, prob["states"])
    _assert_same(*chips, (40, 27))


@pytest.mark.parametrize("graph_steps", [0, 6, 8])
def test_batches_and_graphs(graph_steps):
    """Per-row relaxation rates, a valve program a chip, graphs of three and four
    launches (the state ends in either buffer)."""
    probs = W.config_batch(7, seed=11)
    chips = [lbm.Chip.batch(probs, graph_steps=graph_steps), lbm.Chip.batch(probs, **_single("fp32"))]
    for c in chips:
        for k, p in enumerate(probs):
            c.set_instance_schedule(k, 20 + 9 * k, p["states"])
    _assert_same(*chips, (50, 31))
