"""The pairing rounds by number of saddles: one CTA (up to 4096), a grid that
meets at barriers and hands over to one CTA, one launch per phase handing over
to the grid (above 3 * 2^20), with few and with many nodes -- the pairs against
those of the self-correcting pairing (Alg. 4), which shares none of the rounds;
and a chain that merges one saddle per round at each of these sizes, which
must end in the sorted finish."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle
import oracle_jobs
import paper_2505_21266_gb300 as dms
from paper_2505_21266_gb300 import fields
from test_gpu_configs import _same_pairs, chain_field


def _same(f):
    o = dms.order(f)
    g = dms.gradient(o)
    c = dms.critical(g)
    a = dms.diagram_d0d2(f, o, g, c)
    b = dms.diagram_d0d2(f, o, g, c, pairing="selfcorrecting")
    assert torch.equal(a.d0, b.d0) and torch.equal(a.d2, b.d2)
    assert torch.equal(a.d0_essential, b.d0_essential)
    return c


@pytest.mark.parametrize("shape,lo,hi", [((3, 4, 5), 0, 64), ((25, 25, 25), 3500, 4096),
                                         ((28, 28, 27), 4097, 8192), ((70, 70, 70), 1 << 16, 1 << 18),
                                         ((236, 240, 244), (3 << 20) + 1, 1 << 23)])
def test_rounds_by_size(shape, lo, hi):
    c = _same(fields.uniform01(shape, 11, "cuda"))
    assert lo <= int(c[1].numel()) <= hi, c[1].numel()


@pytest.mark.parametrize("n", [60, 70, 4090, 4100, 9000])
def test_chain_of_wells(n):
    _same(torch.from_numpy(np.ascontiguousarray(chain_field(n))).cuda())


@pytest.mark.parametrize("n", [1024, 1025, 1026, 32 * 1024 + 1, 33 * 1024 + 2])
def test_pair_lists_at_tile_edges(n):
    """n - 1 saddles, all paired: the pair writer's tiles of 1024 full, one
    short and one over, and more tiles than one warp looks back over at once."""
    f_np = np.ascontiguousarray(chain_field(n, deeper_right=False))
    r = oracle.run(f_np)
    res = dms.diagram(torch.from_numpy(f_np).cuda())
    assert int(res.crit[1].numel()) == n - 1
    d0, d2, _ = oracle_jobs.sorted_pairs(r)
    _same_pairs(res.diagrams.numpy("d0"), d0)
    _same_pairs(res.diagrams.numpy("d2"), d2)
