"""The gradient kernel's tilings at the sizes where they can go wrong: one
slab per CTA, tiles ending one column, row or slab past or short of a border,
grids on both sides of the line between the small and the large tiling
(2^20 vertices), with rows that TMA can stage and rows it cannot -- records
and desc of every vertex against the same lower-star rule and correction run
vertex by vertex on the CPU (which test_lowerstar_host.py pins to the oracle)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2505_21266_gb300 as dms

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2505_21266_gb300", "csrc")


@pytest.fixture(scope="module")
def host_lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    so = str(tmp_path_factory.mktemp("ls") / "host_lowerstar.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "host_lowerstar.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _field(kind, shape):
    rng = np.random.default_rng(sum(shape))
    if kind == "noise":
        return rng.random(shape)
    if kind == "ties":
        return rng.integers(0, 3, shape).astype(np.float64)
    z, y, x = np.indices(shape)  # every second vertex an extremum of its neighbours
    return ((x + y + z) % 2) * 4.0 + rng.random(shape)


@pytest.mark.parametrize("shape", [
    (2, 2, 2), (3, 7, 31), (2, 8, 32), (5, 9, 33), (4, 10, 34), (9, 25, 64), (1 + 16, 24, 65),
    (3, 49, 36), (101, 103, 100), (102, 103, 100), (101, 103, 101), (33, 71, 450)])
@pytest.mark.parametrize("kind", ["noise", "ties", "checker"])
def test_tilings_match_the_vertex_by_vertex_pass(host_lib, shape, kind):
    f = _field(kind, shape)
    order = np.empty(f.size, np.uint32)
    order[np.argsort(f.reshape(-1), kind="stable")] = np.arange(f.size, dtype=np.uint32)
    nz, ny, nx = shape
    desc, rec = np.zeros(f.size, np.uint8), np.zeros(f.size, np.uint64)
    vp = ctypes.c_void_p
    assert host_lib.host_gradient(order.ctypes.data_as(vp), nx, ny, nz, desc.ctypes.data_as(vp),
                                  rec.ctypes.data_as(vp)) == 0
    o = torch.from_numpy(order.view(np.int32)).cuda().view(torch.uint32).reshape(shape)
    g = dms.gradient(o)
    assert np.array_equal(g.desc.cpu().numpy().reshape(-1), desc)
    assert np.array_equal(g.rec.cpu().numpy().reshape(-1).view(np.uint64), rec)
    assert int(g.counts[0]) == int((desc == 15).sum())
