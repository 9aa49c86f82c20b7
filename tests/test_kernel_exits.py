"""Launches and early exits, read off their source.  A word that
other CTAs of the same launch may write is no ground for a thread to leave
ahead of a barrier by itself, since the threads of one CTA may see different
values.  (What such a kernel does after a disagreement is an access out of
range, so it is not run: the source is the evidence.)  Needs no GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_21266_gb300", "csrc")


def _body(name, kernel):
    s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    at = s.index("{", s.index(") " + kernel + "("))
    depth, i = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(s[i], 0)
        i += 1
        if depth == 0:
            return s[at:i]


def test_sort_pass_leaves_as_a_whole():
    """onesweep_kernel: `failed` is set by any CTA whose wait runs out.  Up to
    the barrier behind the ticket only thread 0 reads it, and what it saw
    reaches the CTA through the ticket's word, tested before its first use."""
    body = _body("dms_order.cu", "onesweep_kernel")
    entry, rest = body.split("__syncthreads();", 1)
    reads = [st for st in entry.split(";") if "failed" in st]
    assert len(reads) == 1 and re.search(r"if \(threadIdx\.x == 0\)\s+sm\.tile = ", reads[0]), reads
    assert all("failed" not in cond for cond in re.findall(r"if \(([^;]*)\) return", entry))
    assert rest.index("if (sm.tile == kNoTile) return") < rest.index("tile = sm.tile")
    # further on it is only ever set
    assert set(re.findall(r"failed[^;]*", rest)) == {"failed = 1"}


def test_cooperative_grid_is_kept_per_device():
    """launch_rounds: what it keeps between calls (how many of its CTAs a
    device holds at once) is kept by device and may be read and written by
    several threads; a grid that is too large for the current device is
    refused at its launch, one from a race is anything."""
    s = open(os.path.join(CSRC, "dms_pairs.cu")).read()
    at = s.index("int launch_rounds(")
    body = s[at:s.index("\n}\n", at)]
    kept = re.findall(r"static (?!constexpr|const )[^;]*;", body)
    assert all(re.match(r"static std::atomic<int> \w+\[kDevices\];", k) for k in kept), kept
    assert body.index("cudaGetDevice(&dev)") < body.index("resident[dev]")
