"""lbm_step_diagnostics where a step stands by itself, whose last block forms the totals
(or a reduction after it), and where a call is cut into several runs of steps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1307_4703_gb300 import lbm, workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

STEP_PARTIALS = 32768  # block partials that one reduction launch adds up


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1307_4703_gb300 import build
    build.build()
    lbm.load()


def _two(prob, init, **opts):
    chips = [lbm.Chip.from_problem(prob, **opts) for _ in range(2)]
    for c in chips:
        c.init_equilibrium(**init)
        c.set_valve_schedule(4, [1, 2, 3, 0])
    return chips


def _compare(a, b, rows, want):
    """Rows and populations bit for bit; the last row is also what lbm_get_diagnostics
    gives."""
    a.synchronize()
    assert np.array_equal(rows.cpu().numpy(), np.array(want))
    assert np.array_equal(a.diagnostics(), want[-1])
    for x, y in zip(a.populations(), b.populations()):
        assert np.array_equal(x, y)
    a.close()
    b.close()


@pytest.mark.parametrize("paper_ports", [False, True])
@pytest.mark.parametrize("opts", [dict(), dict(variant=4), dict(precision="fp16"), dict(precision="bf16"),
                                  dict(precision="bf16", variant=1), dict(max_blocks=5), dict(max_blocks=17),
                                  dict(variant=4, block_threads=64), dict(variant=2), dict(wall_scheme=1)])
def test_steps_by_themselves(opts, paper_ports):
    """Calls of one step, again and again: each leaves the ticket count at zero."""
    prob, init = W.random_case(41, 300, 48, solid_frac=0.1, paper_ports=paper_ports)
    a, b = _two(prob, init, **opts)
    n = 9
    rows = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    want = []
    for k in range(n):
        a.step_diagnostics(1, rows[k].data_ptr())
        b.step(1)
        want.append(b.diagnostics())
    _compare(a, b, rows, want)


@pytest.mark.parametrize("block_threads,remainder", [(64, 1), (64, 2), (128, 1), (128, 0)])
def test_calls_of_several_runs(block_threads, remainder):
    """More steps than one reduction launch has room for: the partials' place is used
    again, a run ends before the call does, and a remainder of one step (which blocks of
    128 threads fold) or two follows."""
    prob, init = W.random_case(43, 512, 600, solid_frac=0.05)
    a, b = _two(prob, init, variant=1, block_threads=block_threads)
    n = 2 * (STEP_PARTIALS // a.info()["grid"]) + remainder
    assert 20 < n < 200
    rows = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    a.step_diagnostics(n, rows.data_ptr())
    want = []
    for _ in range(n):
        b.step(1)
        want.append(b.diagnostics())
    _compare(a, b, rows, want)
