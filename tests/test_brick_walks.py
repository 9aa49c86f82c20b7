"""The v-path words and walks of the kernels (csrc/dms_bricks.cuh, built for
the host) on the CPU: on the oracle's gradients of grids that span several
bricks, every saddle's two walks end where the oracle's triplets say, over the
bricks' words and cell by cell; and a walk
over words that loop from brick to brick (no gradient gives them, inconsistent
arrays of a caller may) ends as a loop after about the hops that the loop has,
not after as many as the grid has cells, while a valid walk of any length
reaches its end.  (A loop that is not recognised keeps a GPU busy for as long as
it is allowed to: it is shown here and not there.)"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from test_walk_schedule import OUTSIDE, _check, _d0_instance, _d2_instance

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2505_21266_gb300", "csrc")
END, LOOP = 0x80000000, 0xFFFFFFFE


def _ends(fn, src, shape, nodes, cells, turns):
    """The end words of the walks from cells; turns: cell by cell, in that
    order (None: over the bricks)."""
    nz, ny, nx = shape
    out = np.zeros(len(cells), np.uint32)
    assert fn(ctypes.c_void_p(src.ctypes.data), *(ctypes.c_int64(v) for v in (nx, ny, nz)),
              ctypes.c_void_p(nodes.ctypes.data), ctypes.c_int64(len(nodes)),
              ctypes.c_void_p(cells.ctypes.data), ctypes.c_int64(len(cells) // 2),
              ctypes.c_void_p(None if turns is None else turns.ctypes.data),
              ctypes.c_void_p(out.ctypes.data)) == 0
    return out


def _build(d, name):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    so = str(d / (name + ".so"))
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, name + ".cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lib = _build(tmp_path_factory.mktemp("bricks"), "host_bricks")
    lib.host_long_walk.restype = ctypes.c_int64
    lib.host_long_walk.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_void_p]
    return lib


@pytest.fixture(scope="module")
def gradient(tmp_path_factory):
    lib = _build(tmp_path_factory.mktemp("lowerstar"), "host_lowerstar")

    def run(f):
        nz, ny, nx = f.shape
        order = oracle.run(f, diagrams=False).order.astype(np.uint32)
        desc, rec = np.zeros(f.size, np.uint8), np.zeros(f.size, np.uint64)
        assert lib.host_gradient(order.ctypes.data, nx, ny, nz, desc.ctypes.data, rec.ctypes.data) == 0
        return desc, rec

    return run


def _fields():
    rng = np.random.default_rng(8)
    for shape in ((9, 10, 20), (5, 18, 17), (17, 9, 6), (3, 16, 33)):
        yield rng.random(shape).astype(np.float32)
    z, y, x = np.meshgrid(np.arange(10), np.arange(17), np.arange(19), indexing="ij")
    yield (np.sin(x * 0.5) * np.cos(y * 0.4) + 0.3 * np.sin(z * 0.9)).astype(np.float32)


@pytest.mark.parametrize("k", range(5))
@pytest.mark.parametrize("kind", ["d0", "d2"])
@pytest.mark.parametrize("how", ["bricks", "cells", "cells reversed", "cells shuffled"])
def test_walks_reach_the_oracle_ends(lib, gradient, how, kind, k):
    f = list(_fields())[k]
    desc, rec = gradient(f)
    saddles, starts, _, nodes, trip = (_d0_instance if kind == "d0" else _d2_instance)(f)
    assert saddles
    nodes = np.array(sorted(nodes), np.int64)
    cells = np.array([-1 if isinstance(s, tuple) else s for s in starts], np.int64)
    turns = np.arange(len(cells), dtype=np.int64)
    if how == "cells reversed":
        turns = turns[::-1].copy()
    if how == "cells shuffled":
        np.random.default_rng(k).shuffle(turns)
    fn, src = (lib.host_desc_ends, desc) if kind == "d0" else (lib.host_dual_ends, rec)
    out = _ends(fn, src, f.shape, nodes, cells, None if how == "bricks" else turns)
    node = out.astype(np.int64) - END
    assert (node >= 0).all()
    if kind == "d0":
        ends = [int(nodes[i]) for i in node]
    else:
        ends = [OUTSIDE if i == 0 else int(nodes[i - 1]) for i in node]
    _check(saddles, ends, trip)


@pytest.mark.parametrize("rows,half", [(0, 1), (0, 32), (2, 3), (4, 31), (30, 1), (30, 32), (60, 20)])
def test_a_loop_ends(lib, rows, half):
    end = np.zeros(1, np.uint32)
    reads = lib.host_long_walk(rows, half, end.ctypes.data)
    assert int(end[0]) == LOOP
    # to the loop and once round, both up to doubled by where it is noticed,
    # behind the hops that are not looked at
    assert 0 <= reads <= 130 + 4 * (32 * rows + 2 * half), reads


@pytest.mark.parametrize("rows", [0, 1, 3, 4, 5, 31, 62])
def test_a_long_walk_reaches_its_end(lib, rows):
    end = np.zeros(1, np.uint32)
    assert lib.host_long_walk(rows, 0, end.ctypes.data) == 32 * rows + 1
    assert int(end[0]) == END + 7


@pytest.mark.parametrize("turns,done", [([0, 1, 2, 3], [3]), ([3, 2, 1, 0], [0, 1, 2, 3]),
                                        ([1, 3, 0, 2], [3])])
def test_long_paths_wait_for_the_bricks(lib, turns, done):
    """A slope of 6000 vertices: cell by cell a walk from its top is too long,
    and so is any that joins it (from 4000, behind one that got down to 1900,
    too); from the top behind a walk that reached the end it is not.  Over the
    bricks all reach it.  Round a ring (no gradient) a walk ends as too long."""
    shape, n = (2, 2, 6000), 24000
    desc = np.full(n, 7, np.uint8)  # to x - 1
    desc[0] = 15
    for row in (6000, 12000, 18000):
        desc[row] = 11 if row == 18000 else (8 if row == 6000 else 9)  # -y-z, -y, -z
    nodes = np.zeros(1, np.int64)
    cells = np.array([5990, 5999, 4000, 70], np.int64)
    turns = np.array(turns, np.int64)
    assert (_ends(lib.host_desc_ends, desc, shape, nodes, cells, None) == END).all()
    out = _ends(lib.host_desc_ends, desc, shape, nodes, cells, turns)
    assert [j for j in range(4) if out[j] == END] == done and all(out[j] in (0, END) for j in range(4))
    desc[3000:3002] = 0, 7  # 3000 -> 3001 -> 3000
    out = _ends(lib.host_desc_ends, desc, shape, nodes, np.array([3000, 3500], np.int64), np.arange(2))
    assert (out == 0).all()
    assert (_ends(lib.host_desc_ends, desc, shape, nodes, np.array([3000, 3500], np.int64), None) == LOOP).all()
