"""Few saddles on a large grid: the v-paths followed cell by cell, with walks
that join others, and left to the bricks where they are too long.  The pairs of
the single-field path, which chooses so by size and density, against those of a
batch of that one field, which always goes by the bricks; at the least number of
vertices and above it, with the last run of landmarks short, and on either side
of the density line; and dense saddles in grids so thin that bricks are mostly outside."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2505_21266_gb300 as dms
from paper_2505_21266_gb300 import batch as dms_batch
from paper_2505_21266_gb300 import fields


def _winding(shape):
    """A valley that winds down between walls, row by row, along all of the
    lowest layer, and pits in the walls of its upper end, from whose rims it is
    entered: paths of nearly a quarter of the layer's cells, which one walk has
    to go and the others join."""
    nz, ny, nx = shape
    y, x = torch.meshgrid(torch.arange(ny, device="cuda"), torch.arange(nx, device="cuda"), indexing="ij")
    step = (y // 4) * nx + torch.where((y // 4) % 2 == 0, x, nx - 1 - x)
    f = step.double() / (ny * nx)
    # walls between the rows, higher away from the gap that each has at one end
    f = torch.where(y % 4 == 0, f, 2.5 - 0.5 * (step % nx) / nx)
    f = torch.where((y % 4 != 0) & (x == torch.where((y // 4) % 2 == 0, nx - 1, 0)),
                    (step + (y % 4) / 4).double() / (ny * nx), f)
    f = f - torch.where((y > ny - 150) & (y % 16 == 2) & (x % 31 == 15), 0.9 + step.double() / (8 * ny * nx),
                        0.0)  # the pits
    z = torch.arange(nz, device="cuda").double().view(-1, 1, 1)
    return (f.view(1, ny, nx) + 4.0 * z).float().contiguous()


CASES = {
    "smooth": ((256, 512, 256), 0.0, True),            # 2^25 vertices
    "a little noise": ((301, 333, 351), 1e-4, True),   # no multiple of a run
    "slabs": ((9, 1999, 2003), 1e-5, True),
    "dense": ((257, 512, 256), 1e-2, False),           # above the line
    "small": ((255, 512, 256), 0.0, False),            # one slab below 2^25
}


def _same(f, few, pairing="rounds"):
    res = dms.diagram(f, pairing)
    n, c = f.numel(), [int(x.numel()) for x in res.crit]
    if few is not None:
        assert (n >= 1 << 25 and max(c[1], c[2]) <= n // 32) == few, (n, c)
    b = dms_batch.Batch([tuple(f.shape)], "cuda")
    b.set_fields([f])
    b.fit()
    d0, d2, _ = b.results()[0]
    assert np.array_equal(res.diagrams.numpy("d0"), d0)
    assert np.array_equal(res.diagrams.numpy("d2"), d2)
    assert len(d0) > 0
    return c


@pytest.mark.parametrize("case", CASES)
def test_by_cells_and_by_bricks(case):
    shape, noise, few = CASES[case]
    _same(fields.gaussian_mixture(shape, 64, (0.02, 0.1), noise, 7, "cuda"), few)


def test_self_correcting_pairing():
    _same(fields.gaussian_mixture((301, 333, 351), 64, (0.02, 0.1), 1e-4, 8, "cuda"), True, "selfcorrecting")


def test_winding_paths():
    _same(_winding((16, 1501, 1409)), True)


@pytest.mark.parametrize("shape", [(1201, 1001, 2), (4, 3, 180001), (1449, 2, 1511), (2, 1447, 1451),
                                   (180001, 3, 4), (1025, 1024, 2)])
@pytest.mark.parametrize("kind", ["noise", "ties"])
def test_thin_grids(shape, kind):
    f = fields.uniform01(shape, 5, "cuda") if kind == "noise" else fields.quantized_noise(shape, 4, 5, "cuda")
    _same(f, None)
