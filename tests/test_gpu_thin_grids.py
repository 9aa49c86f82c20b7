"""Grids thin in one axis, whose tiles reach far outside, and the choices that
the gradient kernel's launch makes for them: tiles of 8 rows for grids of up to
8 rows at any size, one wave of CTAs where a second would be nearly empty;
partial tiles in both axes of a grid above the small ones -- records and desc of
every vertex against the vertex-by-vertex pass on the CPU."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import test_gpu_gradient_tiles as tiles
from test_gpu_gradient_tiles import host_lib  # noqa: F401


@pytest.mark.parametrize("shape", [
    (600, 8, 220), (700, 2, 760), (520, 9, 225), (900, 600, 2), (2, 1100, 480), (300, 300, 16),
    (44, 193, 129), (131, 25, 321), (9, 2, 300), (300, 9, 2), (2, 300, 9)])
@pytest.mark.parametrize("kind", ["noise", "ties"])
def test_thin_and_partial_tiles(host_lib, shape, kind):  # noqa: F811
    tiles.test_tilings_match_the_vertex_by_vertex_pass(host_lib, shape, kind)
