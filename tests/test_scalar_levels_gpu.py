"""Several scalar-only steps in one launch (the default of lbm_scalar_step): the
populations and diagnostics are the bits of single steps, at the edges of the
strips, rows and blocks it is cut into."""
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


def _same(a, b):
    for x, y in zip(a.populations(), b.populations()):
        assert np.array_equal(x, y)
    assert np.array_equal(a.diagnostics(), b.diagnostics())


@pytest.mark.parametrize("nx,ny,paper_ports,decay,period", [
    (4, 8, False, 0.0, 5), (60, 9, True, 1e-3, 4), (124, 13, False, 0.0, 3), (125, 30, False, 1e-3, 11),
    (128, 31, True, 0.0, 7), (129, 47, False, 0.0, 2), (244, 33, True, 1e-3, 9), (513, 64, False, 0.0, 50),
    (1025, 90, True, 0.0, 6)])
def test_random_lattices(nx, ny, paper_ports, decay, period):
    """Obstacles and every port kind; valve words that change before, at and after a
    launch's three steps; coupled steps in between (the scalar planes then join the
    fluid's)."""
    prob, init = W.random_case(nx + ny, nx, ny, paper_ports=paper_ports, decay=decay)
    r = np.random.default_rng(nx)
    u = {w: 0.05 * (r.random((2, ny, nx)) - 0.5) for w in (7, 5, 2)}
    chips = [lbm.Chip.from_problem(prob, scalar_variant=v) for v in (0, 1)]
    for c in chips:
        c.init_equilibrium(**init)
        c.set_valve_schedule(period, [7, 5, 2])
        for w, (ux, uy) in u.items():
            c.set_velocity_field(w, ux, uy)
    for n in (1, 3, 4, 9, 25):
        for c in chips:
            c.scalar_step(n, 0.7)
        _same(*chips)
    for c in chips:
        c.step(5)
        c.scalar_step(8)
        c.step(4)
    _same(*chips)
    assert chips[0].step_count() == chips[1].step_count()
    for c in chips:
        c.close()


@pytest.mark.parametrize("nx,ny", [(256, 128), (777, 401), (2100, 1000)])
def test_two_channel_chips(nx, ny):
    prob = W.config_large_chip(nx, ny)
    c_start = np.random.default_rng(3).random((ny, nx))
    chips = [lbm.Chip.from_problem(prob, scalar_variant=v) for v in (0, 1)]
    for c in chips:
        c.init_equilibrium(1.0, 0.0, 0.0, c_start)
        c.set_valve_schedule(17, prob["states"])
        for w, (ux, uy) in W.channel_flow_fields(prob).items():
            c.set_velocity_field(w, ux, uy)
        c.scalar_step(60)
    _same(*chips)
    for c in chips:
        c.close()


def test_store_velocity_under_capture():
    """A velocity field stored by a captured call (which may not wait for the stream, so
    the strips are not planned there): the scalar steps after its replay are those of a
    field stored directly."""
    s = torch.cuda.Stream()
    chips = [lbm.Chip.from_problem(W.config_small(), stream=s, torch_alloc=True) for _ in range(2)]
    for c in chips:
        c.set_valves(1)
        c.step(5)
        c.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        chips[0].store_velocity(1)
    graph.replay()
    torch.cuda.synchronize()
    chips[1].store_velocity(1)
    for c in chips:
        c.scalar_step(7)
    for a, b in zip(chips[0].populations(), chips[1].populations()):
        assert np.array_equal(a, b)
    for c in chips:
        c.close()
