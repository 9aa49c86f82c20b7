"""The lower stars of an image by tiles of 64 x 16 anchors: grids that end at,
one short of and one past a tile, on fields whose links have one, two and three
lower arcs, are wholly lower (maxima, their critical triangle at every place),
and are tied -- every vector, critical simplex and pair against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_2d import _check


def _field(kind, shape):
    rng = np.random.default_rng(sum(shape))
    y, x = np.indices(shape)
    return {
        "noise": lambda: rng.random(shape),
        "ties": lambda: rng.integers(0, 3, shape),
        # every third vertex of a row above its six neighbours, in random order
        "maxima": lambda: rng.random(shape) + 2.0 * ((x - y) % 3 == 0),
        "minima": lambda: rng.random(shape) - 2.0 * ((x - y) % 3 == 0),
    }[kind]().astype(np.float32)


@pytest.mark.parametrize("kind", ["noise", "ties", "maxima", "minima"])
@pytest.mark.parametrize("shape", [(16, 64), (15, 63), (17, 65), (33, 129), (2, 128), (48, 2)])
def test_lower_stars_at_tile_edges(shape, kind):
    _check(_field(kind, shape))
