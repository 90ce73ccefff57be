"""The list of the paper's wall links where several host threads make it: the values of
the FP64 oracle (bound as in test_wall_links_gpu.py), in eight bytes a link."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1307_4703_gb300 import lbm, workloads as W  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

STEPS = 4


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1307_4703_gb300 import build
    build.build()
    lbm.load()


def _links(solid):
    """Neighbours of fluid nodes that are not fluid."""
    ny, nx = solid.shape
    pad = np.ones((ny + 2, nx + 2), bool)
    pad[1:-1, 1:-1] = solid != 0
    n = 0
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            n += np.count_nonzero((solid == 0) & pad[1 + dy:ny + 1 + dy, 1 + dx:nx + 1 + dx])
    return n


@pytest.mark.parametrize("nx,ny,solid_frac", [(900, 600, 0.2), (701, 777, 0.5), (20, 30000, 0.05)])
def test_large_lattices(nx, ny, solid_frac):
    prob, init = W.random_case(11, nx, ny, solid_frac=solid_frac)
    chip = lbm.Chip.from_problem(prob, wall_scheme=1)
    plain = lbm.Chip.from_problem(prob, variant=1)
    pitch = (nx + 127) // 128 * 128
    extra = chip.info()["device_bytes"] - plain.info()["device_bytes"]
    assert extra <= 8 * 4 * ny * pitch + 8 * _links(np.asarray(prob["solid"])) + 512
    plain.close()
    prob["wall_scheme"] = 1
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
    tol = STEPS * 90 * 2.0 ** -24
    assert np.abs(f - np.moveaxis(fp, -1, 0))[:, fl].max() <= tol
    assert np.abs(g - np.moveaxis(gp, -1, 0))[:, fl].max() <= tol
    chip.close()
