"""The reverse step runs on 64-node tiles: widths around their edges, random
obstacles (bounce-back links inside tiles, across their edges and at the rim),
every port kind, against the FP64 oracle adjoint.  n forward and n reverse steps
of some thirty FP32 roundings each are off by 2 n 30 2^-24 of the largest terms
(2.2e-5 at n = 6); five times that for cancellation in the sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1307_4703_gb300 import lbm, workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

N = 6
TOL = 5 * 2 * N * 30 * 2.0 ** -24


@pytest.mark.parametrize("ckpt,multi", [(1, 0), (4, 0), (4, 3)])
@pytest.mark.parametrize("nx,ny,solid_frac", [(7, 9, 0.1), (63, 12, 0.3), (64, 8, 0.0), (66, 17, 0.3), (129, 33, 0.1)])
def test_reverse_steps_at_tile_edges(nx, ny, solid_frac, ckpt, multi):
    prob, init = W.random_case(9, nx, ny, solid_frac=solid_frac)
    fy, fx = np.nonzero(prob["solid"] == 0)
    ox, oy = fx[::3], fy[::3]
    tg = np.linspace(0.2, 0.8, len(ox))
    words = [7, 3, 7, 5, 7, 6, 7]
    L = oracle.from_problem(prob)
    L.init_equilibrium(**init)
    J, dt, du, dc = L.adjoint(N, words[:N], ox, oy, tg, np.ones(len(ox)))
    chip = lbm.Chip.from_problem(prob, multi_step=multi)
    chip.init_equilibrium(**init)
    chip.set_valve_schedule(1, words)
    gJ, gt, gu, gc = chip.adjoint(N, ox, oy, tg, ckpt_every=ckpt)
    assert abs(gJ - J) <= TOL * J
    assert abs(gt - dt) <= TOL * abs(dt)
    for got, ref in ((gu, du), (gc, dc)):
        assert np.linalg.norm(np.ravel(got) - np.ravel(ref)) <= TOL * np.linalg.norm(np.ravel(ref))
    chip.close()
