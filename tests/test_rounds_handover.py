"""The pairing rounds' hand-over from the grid to CTA 0 (csrc/dms_pairs.cu,
pair_rounds), restated with CTAs that run in any order between their barriers,
on the kernel's own choice of count words (csrc/dms_rounds.cuh, built for the
host): a CTA that reads the count of the grid's last round late, however far
CTA 0 has gone on alone by then, reads that count and leaves.  With the words
shared between the grid's rounds and those of CTA 0 alone it may read a later
count, stay and work beside CTA 0: the simulation shows that too.  (A race on
memory: it is not run on a GPU without its mend.)  Needs no GPU."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2505_21266_gb300", "csrc")
CTAS = 3


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    so = str(tmp_path_factory.mktemp("rounds") / "host_rounds.so")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "host_rounds.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.host_goes_solo.argtypes = [ctypes.c_uint, ctypes.c_longlong, ctypes.c_int]
    return lib


class Sim:
    """One launch of CTAS CTAs.  forest: the live saddles before each forest
    round, then 0; exact: the forest's saddles, then those left after each
    exact round, then 0."""

    def __init__(self, lib, count_word, goes_solo, nn, forest, exact):
        self.lib, self.count_word, self.goes_solo, self.nn = lib, count_word, goes_solo, nn
        self.plan = {"forest": forest, "exact": exact}
        self.ctr = [0] * lib.host_words()
        self.ctr[lib.host_forest_word()] = exact[0]
        self.arrived = 0
        self.worked = []  # (CTA, solo, phase, round, n)

    def cta(self, b):
        """Yields before every access that other CTAs can see."""
        ctr, solo, forest, rnd, epoch = self.ctr, False, True, 1, 0
        n, at = self.plan["forest"][0], 0
        while True:
            if not solo and self.goes_solo(n, self.nn, forest):
                if b != 0:
                    return
                solo = True
            if n == 0:
                if not forest:
                    return
                forest, rnd, at = False, 1, 0
                yield
                n = ctr[self.lib.host_forest_word()]
                if b == 0:
                    for k in range(3):
                        ctr[self.count_word(k, solo)] = 0
                if not solo:
                    epoch += 1
                    self.arrived += 1
                    while self.arrived < epoch * CTAS:
                        yield "wait"
                continue
            phase = "forest" if forest else "exact"
            self.worked.append((b, solo, phase, rnd, n))
            if not solo:  # behind the search for the roots
                epoch += 1
                self.arrived += 1
                while self.arrived < epoch * CTAS:
                    yield "wait"
            word = self.count_word(rnd, solo)
            if b == 0:
                yield
                ctr[self.count_word(rnd + 1, solo)] = 0
            at += 1
            left = self.plan[phase][at] if at < len(self.plan[phase]) else 0
            share = left if solo else left // CTAS + (left % CTAS if b == 0 else 0)
            yield
            ctr[word] += share
            if not solo:
                epoch += 1
                self.arrived += 1
                while self.arrived < epoch * CTAS:
                    yield "wait"
            yield
            n = ctr[word]
            rnd += 1

    def run(self, order):
        """order(live) picks the next CTA among those that can go on."""
        live = {b: self.cta(b) for b in range(CTAS)}
        waiting = set()
        for _ in range(100_000):
            if not live:
                return True
            ready = [b for b in live if b not in waiting] or list(live)
            b = order(ready)
            arrived = self.arrived
            try:
                said = next(live[b])
            except StopIteration:
                del live[b]
                waiting.clear()
                continue
            if self.arrived != arrived:
                waiting.clear()
            if said == "wait":
                waiting.add(b)
                if len(waiting) == len(live):
                    return False  # everyone waits at a barrier nobody joins
            else:
                waiting.clear()
        return False


PLANS = [
    # (nodes, forest rounds, exact rounds): handed over in the forest phase, in
    # the exact rounds, and at the start of those
    (60_001, [90_000, 20_000, 4_000, 900, 100, 0], [60_000, 30_000, 11_000, 5_000, 4_500, 700, 0]),
    (4_001, [9_000, 2_000, 300, 0], [4_000, 1_500, 800, 100, 0]),
    (70_001, [90_000, 20_000, 4_000, 0], [70_000, 30_000, 4_000, 900, 20, 0]),
    (200_001, [300_000, 1_000, 0], [4_000, 900, 20, 0]),
]


def _orders():
    yield max  # CTA 0 runs last wherever it can: the others never late
    yield min  # CTA 0 goes on as far as it can: the others as late as can be
    for seed in range(120):  # CTA 0 ahead of the others by more and more
        rng = random.Random(seed)
        ahead = (0.0, 0.8, 0.95)[seed % 3]
        yield lambda ready: 0 if 0 in ready and rng.random() < ahead else rng.choice(ready)


def _ok(lib, count_word, goes_solo):
    for nn, forest, exact in PLANS:
        for order in _orders():
            s = Sim(lib, count_word, goes_solo, nn, forest, exact)
            if not s.run(order):
                return False
            alone = [i for i, w in enumerate(s.worked) if w[1]]
            if not alone or any(w[0] != 0 for w in s.worked[alone[0]:]):
                return False
            # CTA 0 saw every round's count
            mine = [(w[2], w[4]) for w in s.worked if w[0] == 0]
            if mine != [("forest", n) for n in forest[:-1]] + [("exact", n) for n in exact[:-1]]:
                return False
    return True


def _many_after_few(n, nn, forest):
    """A hand-over that lets CTA 0 meet up to 65,536 saddles alone."""
    return n <= 4096 and (not forest or nn <= 65_536)


def test_late_readers_leave(lib):
    for goes_solo in (lib.host_goes_solo, _many_after_few):
        assert _ok(lib, lambda r, solo: lib.host_count_word(r, int(solo)), goes_solo)


def test_shared_words_are_caught(lib):
    assert not _ok(lib, lambda r, solo: lib.host_first_round_word() + r % 3, _many_after_few)


def test_few_saddles_alone(lib):
    """CTA 0 alone never meets more than kSolo saddles: neither those live at
    the hand-over, nor, from the forest's rounds, the forest's (nodes - 1)."""
    few = lib.host_solo()
    for nn in (2, few, few + 1, few + 2, 2 * few, 60_000, 65_536, 65_537, 1 << 20):
        for n in (1, few - 1, few, few + 1, 1 << 20):
            for forest in (False, True):
                alone = lib.host_goes_solo(n, nn, int(forest))
                assert bool(alone) == (n <= few and (not forest or nn - 1 <= few)), (n, nn, forest)


def test_words_do_not_overlap(lib):
    grid = {lib.host_count_word(r, 0) for r in range(6)}
    alone = {lib.host_count_word(r, 1) for r in range(6)}
    assert len(grid) == len(alone) == 3 and not grid & alone
    assert all(0 <= w < lib.host_words() for w in grid | alone)
    # both are among the words cleared with those of the rounds
    assert min(grid | alone) >= lib.host_first_round_word()
