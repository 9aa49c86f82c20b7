"""The vertex order by tiles of 4096 keys that look back at the tiles before
them: fields of one tile, one short of it and just past it, of many tiles, and
of more than 2^25 vertices (the inverse permutation by slices); values that are
all different, tied (digits that are skipped), of both zeros, one value -- equal
to numpy's stable sort."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2505_21266_gb300 as dms


def _check(f):
    want = np.empty(f.size, np.uint32)
    want[np.argsort(f.reshape(-1), kind="stable")] = np.arange(f.size, dtype=np.uint32)
    got = dms.order(torch.from_numpy(f).cuda()).cpu().numpy().reshape(-1)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("shape", [(2, 2, 2), (13, 15, 21), (16, 16, 16), (10, 10, 41),
                                   (64, 64, 33), (96, 101, 97)])
def test_order_at_tile_edges(shape):
    rng = np.random.default_rng(sum(shape))
    n = int(np.prod(shape))
    for f in (rng.standard_normal(n), rng.integers(0, 4, n), np.full(n, 2.5), -np.arange(n),
              rng.choice([-0.0, 0.0, 1.0, -1.0, np.inf, -np.inf], n)):
        _check(f.astype(np.float32).reshape(shape))


@pytest.mark.parametrize("levels", [0, 5])
def test_order_by_slices(levels):
    rng = np.random.default_rng(levels)
    shape = (323, 322, 323)  # 2^25 + 39,506 vertices
    f = rng.integers(0, levels, shape) if levels else rng.random(shape)
    _check(f.astype(np.float32))
