"""Calls from several host threads at once, each on a stream of its own: the
first ones of a process (what the launchers look up once is looked up by all of
them together), and sizes whose pairing rounds run in one CTA, in a grid that
meets at barriers, and in launches per phase.  Every result is what the call
gives alone, bit for bit."""
import subprocess
import sys
import os

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# in a process of its own, so that its threads make the first calls
CHILD = r"""
import sys, threading
sys.path.insert(0, sys.argv[1])
import torch
import paper_2505_21266_gb300 as dms
from paper_2505_21266_gb300 import fields

def volume(shape, seed):
    f = fields.uniform01(shape, seed, "cuda")
    def call():
        r = dms.diagram(f)
        return [r.order.view(torch.int32), r.grad.desc, r.grad.rec, *r.crit, r.diagrams.d0, r.diagrams.d2]
    return call

def image(shape, seed):
    f = fields.uniform01((1,) + shape, seed, "cuda")[0].contiguous()
    def call():
        r = dms.diagram2d(f)
        return [r.order.view(torch.int32), r.grad.desc, r.grad.rec, *r.crit, r.diagrams.d0, r.diagrams.d1]
    return call

calls = [volume((9, 11, 13), 1), volume((64, 60, 56), 2), volume((101, 90, 77), 3),
         volume((236, 240, 244), 4), image((700, 501), 5), volume((40, 44, 48), 6)]
REPS = 4
torch.cuda.synchronize()
got = [[] for _ in calls]
gate = threading.Barrier(len(calls))
wrong = []

def work(k):
    try:
        s = torch.cuda.Stream()
        gate.wait()
        with torch.cuda.stream(s):
            for _ in range(REPS):
                got[k].append(calls[k]())
        s.synchronize()
    except Exception as e:
        wrong.append((k, repr(e)))

threads = [threading.Thread(target=work, args=(k,)) for k in range(len(calls))]
for t in threads:
    t.start()
for t in threads:
    t.join()
assert not wrong, wrong
for k, call in enumerate(calls):
    alone = call()
    for many in got[k]:
        assert len(many) == len(alone)
        for a, b in zip(many, alone):
            assert torch.equal(a, b), k
print("SAME")
"""


def test_threads_on_their_own_streams():
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("SAME"), r.stdout + r.stderr
