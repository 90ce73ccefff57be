"""Totals after lbm_step calls whose last run of steps is one cooperative launch
(multi_step) and follows a run of a single step: those of the call's last step."""
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


def _check(plain, multi, calls):
    """After each call the totals of both handles: sums over another grouping of
    blocks, equal to round-off; each call moves them by far more than that."""
    before = np.zeros(4)
    for n in calls:
        for c in (plain, multi):
            c.step(n)
        d = plain.diagnostics()
        assert not np.allclose(d, before, rtol=1e-6, atol=1e-9)
        assert np.allclose(multi.diagnostics(), d, rtol=1e-6, atol=1e-9), n
        before = d
    plain.close()
    multi.close()


@pytest.mark.parametrize("calls", [(33,), (24, 9), (49, 5, 60)])
def test_single_step_before_the_last_run(calls):
    """Runs of at most eight steps, valves that switch every 25: the first calls leave a
    run of one step before a switch, the later ones start one step before it."""
    prob, init = W.random_case(12, 300, 20)
    chips = [lbm.Chip.from_problem(prob, **kw) for kw in ({}, dict(multi_step=8))]
    for c in chips:
        c.init_equilibrium(**init)
        c.set_valve_schedule(25, [7, 5, 2])
    _check(*chips, calls)


def test_batch_of_chips_that_switch_one_step_apart():
    probs = W.config_batch(2, seed=6)
    chips = [lbm.Chip.batch(probs, **kw) for kw in ({}, dict(multi_step=50))]
    for c in chips:
        for k, p in enumerate(probs):
            c.set_instance_schedule(k, 30 + k, p["states"])
    _check(*chips, (40, 25))
