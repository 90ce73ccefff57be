"""The device read-out of the fields at the widths where its blocks change shape, with
arrays that 128-bit stores suit and ones they do not."""
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


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("nx,ny", [(5, 9), (60, 4001), (124, 33), (128, 34), (129, 35), (132, 2600), (256, 30), (257, 31),
                                   (513, 40), (1030, 29)])
def test_against_the_populations(nx, ny, precision):
    """The moments of the populations in FP64.  The kernel adds nine (five) FP32 values of
    magnitude below one, as deviations from rest, and divides by the density: a few units
    of 2^-24, and as much again from the populations read out in FP32."""
    prob, init = W.random_case(nx + ny, nx, ny)
    chip = lbm.Chip.from_problem(prob, precision=precision)
    chip.init_equilibrium(**init)
    f, g = (a.astype(np.float64) for a in chip.populations())
    e = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)], float)
    rho = f.sum(0)
    want = [rho, np.einsum("i,iyx->yx", e[:, 0], f) / rho, np.einsum("i,iyx->yx", e[:, 1], f) / rho, g.sum(0)]
    fluid = ~chip.solid
    for shift in (0, 1):  # an array one float past a 16-byte boundary
        out = [torch.full((ny * nx + 4,), np.nan, device="cuda") for _ in range(4)]
        chip.fields_device(*[o[shift:] for o in out])
        torch.cuda.synchronize()
        for o, w in zip(out, want):
            o = o.cpu().numpy()
            a = o[shift:shift + ny * nx].reshape(ny, nx)
            assert np.abs(a - w)[fluid].max() < 2e-6
            assert not np.any(a[~fluid])
            assert np.all(np.isnan(o[:shift])) and np.all(np.isnan(o[shift + ny * nx:]))
    only = torch.full((ny, nx), np.nan, device="cuda")
    chip.fields_device(C=only)
    torch.cuda.synchronize()
    assert np.array_equal(only.cpu().numpy(), a)  # (a: C of the loop above)
    chip.close()
