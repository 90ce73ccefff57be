"""The paper's wall values are computed a thread a link from the list made with
the chip: lattices whose links see two, one and no fluid nodes ahead of them
(sparse to dense random obstacles, lists of no whole number of blocks) against
the FP64 oracle.  An FP32 step rounds some thirty operations of O(1) terms, 30
2^-24 a step, which the extrapolation 2 rho1 - rho2 can treble: 4 steps x 30 x 3
x 2^-24 = 2.2e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1307_4703_gb300 import lbm, workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

STEPS = 4


@pytest.mark.parametrize("precision,u", [("fp32", 0.0), ("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("nx,ny,solid_frac", [(5, 8, 0.0), (17, 9, 0.2), (131, 12, 0.02), (259, 33, 0.5)])
def test_wall_links_match_oracle(nx, ny, solid_frac, precision, u):
    prob, init = W.random_case(11, nx, ny, solid_frac=solid_frac)
    prob["wall_scheme"] = 1
    chip = lbm.Chip.from_problem(prob, precision=precision)
    ref = oracle.from_problem(prob)
    chip.init_equilibrium(**init)
    ref.init_equilibrium(**init)
    chip.set_valve_schedule(1, prob["states"])
    for t in range(STEPS):
        chip.step(1)
        ref.step(prob["states"][t])
    f, g = chip.populations()
    fp, gp = ref.post_collision()
    fl = ~ref.solid
    tol = STEPS * 90 * 2.0 ** -24 + 3 * STEPS * u / 4
    assert np.abs(f - np.moveaxis(fp, -1, 0))[:, fl].max() <= tol
    assert np.abs(g - np.moveaxis(gp, -1, 0))[:, fl].max() <= tol
    chip.close()
