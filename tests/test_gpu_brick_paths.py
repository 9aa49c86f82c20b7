"""v-paths resolved by bricks (16^3 vertices for the descending paths, 16 x 8 x
8 for the dual ones, 32 x 32 on images): grids that end at, one short of and
one past a brick, where a step leaves the grid from a brick that does not touch
its last vertex, and smooth fields and combs whose paths cross many bricks,
turn and come back -- every pair against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_2d import _check as check2d
from test_gpu_parity import _check_all


def _fields(shape):
    rng = np.random.default_rng(sum(shape))
    grids = np.meshgrid(*[np.linspace(0, 1, n) for n in shape], indexing="ij")
    smooth = sum(np.sin(7.0 * g + i) for i, g in enumerate(grids))
    # a winding valley: one low row after the other, joined at alternating ends
    comb = rng.random(shape) * 0.5 + 4.0
    rows = comb.reshape(-1, shape[-2], shape[-1])[0]
    at = 0.0
    for y in range(0, shape[-2], 2):
        xs = range(shape[-1]) if (y // 2) % 2 == 0 else range(shape[-1] - 1, -1, -1)
        for x in xs:
            rows[y, x] = at = at + 1e-4
        if y + 1 < shape[-2]:
            rows[y + 1, xs[-1]] = at = at + 1e-4
    return {"noise": rng.random(shape), "smooth": smooth + 1e-3 * rng.random(shape), "comb": comb}


@pytest.mark.parametrize("kind", ["noise", "smooth", "comb"])
@pytest.mark.parametrize("shape", [(8, 16, 16), (9, 17, 17), (7, 15, 33), (17, 9, 18), (16, 8, 32), (25, 18, 49)])
def test_volume_paths_at_brick_edges(shape, kind):
    _check_all(_fields(shape)[kind].astype(np.float32))


@pytest.mark.parametrize("kind", ["noise", "smooth", "comb"])
@pytest.mark.parametrize("shape", [(32, 32), (33, 34), (31, 65), (97, 64)])
def test_image_paths_at_brick_edges(shape, kind):
    check2d(_fields(shape)[kind].astype(np.float32))
