"""Workloads of the framework, each one pass through its public entry points.

A case is a dict of plain values: what is computed (``path``), the field's
shape and recipe, and the options of the call.  ``prepare`` makes what a
program holds before the call (device fields, or page-locked host fields, or a
captured batch), ``run`` makes the call and returns everything it computes.

Recipes, after the fields of the benchmark and the tests: ``mixture`` is a
smooth field (Gaussians) with a little noise, the shape of simulation and
imaging data; ``noise`` is U[0,1) per vertex, the densest set of critical
simplices; ``ties`` is noise quantised to a number of levels, as integer
valued scans are, which puts the tie-break to work.
"""
import math

import numpy as np
import torch

import paper_2505_21266_gb300 as dms
from paper_2505_21266_gb300 import batch as dms_batch
from paper_2505_21266_gb300 import fields

PERSISTENCE = 0.05  # threshold of the simplification loss


def _mixture(gauss, lo, hi, noise):
    return {"field": "mixture", "gauss": gauss, "sigma_lo": lo, "sigma_hi": hi, "noise": noise}


def listed():
    return [
        # the smallest call: a patch of a volume, or one field of a parameter
        # sweep; the launches and the reads of counts are what it costs
        {"name": "diagram_24", "path": "diagram", "nx": 24, "ny": 24, "nz": 24,
         **_mixture(16, 0.05, 0.2, 1e-3)},
        # a small volume, such as a crop that a user looks at interactively
        {"name": "diagram_64", "path": "diagram", "nx": 64, "ny": 64, "nz": 64,
         **_mixture(16, 0.05, 0.2, 1e-3)},
        # a cropped scan: odd extents in every axis, rows that are not a
        # multiple of 16 bytes, noise at every vertex
        {"name": "diagram_odd", "path": "diagram", "nx": 203, "ny": 131, "nz": 77,
         "field": "noise"},
        # an integer-valued volume at the size of the paper's datasets:
        # massive ties and the densest critical simplices
        {"name": "diagram_ties_512", "path": "diagram", "nx": 512, "ny": 512, "nz": 512,
         "field": "ties", "levels": 256},
        # a large simulation volume, the size the framework is benchmarked on
        {"name": "diagram_1024", "path": "diagram", "nx": 1024, "ny": 1024, "nz": 1024,
         **_mixture(256, 0.01, 0.1, 1e-2)},
        # one gradient-descent step of topological simplification on a patch
        # (the size of the finite-difference check) ...
        {"name": "step_24", "path": "step", "nx": 24, "ny": 24, "nz": 24,
         **_mixture(8, 0.05, 0.2, 1e-4)},
        # ... and on the volume that the differentiable path is meant for
        {"name": "step_128", "path": "step", "nx": 128, "ny": 128, "nz": 128,
         **_mixture(32, 0.05, 0.2, 1e-4)},
        # a dataset of many volumes of uneven sizes, one graph replay
        {"name": "batch_64", "path": "batch", "fields": 64, "axis_lo": 32, "axis_hi": 256,
         "shapes": 0},
        # fields streamed from host memory, pairs back on the host
        {"name": "stream_256", "path": "stream", "fields": 4, "nx": 256, "ny": 256, "nz": 256,
         **_mixture(64, 0.02, 0.1, 1e-3)},
        # an image of odd extents
        {"name": "image_1500", "path": "image", "nx": 1501, "ny": 999,
         **_mixture(64, 0.01, 0.1, 1e-2)},
        # a large scan or map
        {"name": "image_16384", "path": "image", "nx": 16384, "ny": 16384,
         **_mixture(64, 0.01, 0.1, 1e-2)},
        # the complete diagram of a small volume: D0, D1 and D2
        {"name": "complete_64", "path": "complete", "nx": 64, "ny": 64, "nz": 64,
         **_mixture(16, 0.05, 0.2, 1e-3)},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _axes(rng, n, lo, hi, k=3):
    """k extents in [lo, hi] whose product is about n, uneven by up to 2."""
    side = n ** (1.0 / k)
    return [max(lo, min(hi, int(round(side * math.exp(rng.uniform(-0.35, 0.35)))) + rng.randint(0, 3)))
            for _ in range(k)]


def _field(rng):
    kind = rng.choice(["mixture", "mixture", "noise", "ties"])
    if kind == "mixture":
        lo = rng.uniform(0.01, 0.05)
        return _mixture(_log_int(rng, 8, 128), round(lo, 4), round(lo * rng.uniform(2, 8), 4),
                        10.0 ** rng.uniform(-4, -2))
    if kind == "ties":
        return {"field": "ties", "levels": _log_int(rng, 16, 4096)}
    return {"field": "noise"}


def draw(rng):
    path = rng.choice(["diagram"] * 5 + ["image"] * 2 + ["step", "batch", "stream", "complete"])
    if path == "diagram":
        nx, ny, nz = _axes(rng, _log_int(rng, 1 << 13, 1 << 26), 4, 900)
        c = {"path": path, "nx": nx, "ny": ny, "nz": nz, **_field(rng)}
        if rng.random() < 0.2 and nx * ny * nz < 1 << 24:
            c["pairing"] = "selfcorrecting"
        return c
    if path == "image":
        nx, ny = _axes(rng, _log_int(rng, 1 << 16, 1 << 27), 64, 30000, 2)
        return {"path": path, "nx": nx, "ny": ny, **_field(rng)}
    if path == "step":
        nx, ny, nz = _axes(rng, _log_int(rng, 1 << 12, 1 << 23), 4, 400)
        return {"path": path, "nx": nx, "ny": ny, "nz": nz,
                **_mixture(rng.randint(8, 64), 0.05, 0.2, 10.0 ** rng.uniform(-5, -3))}
    if path == "batch":
        lo = rng.randint(8, 64)
        return {"path": path, "fields": rng.randint(2, 64), "axis_lo": lo,
                "axis_hi": rng.randint(lo + 8, 192), "shapes": rng.randint(1, 1 << 20)}
    if path == "stream":
        nx, ny, nz = _axes(rng, _log_int(rng, 1 << 17, 1 << 24), 16, 500)
        return {"path": path, "fields": rng.randint(2, 6), "nx": nx, "ny": ny, "nz": nz,
                **_field(rng)}
    nx, ny, nz = _axes(rng, _log_int(rng, 1 << 12, 1 << 18), 8, 128)
    return {"path": path, "nx": nx, "ny": ny, "nz": nz,
            **_mixture(rng.randint(8, 32), 0.05, 0.2, 10.0 ** rng.uniform(-4, -3))}


# ---------------------------------------------------------------- inputs --

def _make(case, seed, device="cuda"):
    """The case's field [nz, ny, nx] (an image: [ny, nx]) from the seed."""
    shape = (case.get("nz", 1), case["ny"], case["nx"])
    if case["field"] == "mixture":
        f = fields.gaussian_mixture(shape, case["gauss"], (case["sigma_lo"], case["sigma_hi"]),
                                    case["noise"], seed, device)
    elif case["field"] == "ties":
        f = fields.quantized_noise(shape, case["levels"], seed, device)
    else:
        f = fields.uniform01(shape, seed, device)
    return f if "nz" in case else f[0].contiguous()


# A program keeps results of varying length in arrays of its own: one buffer
# of 64-bit words per field for the lists of critical simplices and the pair
# records (four words each), this many words per vertex (white noise needs
# 1.1 on a volume, 1.8 on an image); what lies past the lists stays zero.
LIST_WORDS = {3: 1.5, 2: 2.2}
STREAM_PAIRS = 0.15  # pair records per vertex, a streamed field's host array


def _lists(n, dims):
    return torch.zeros(int(LIST_WORDS[dims] * n) + 4096, dtype=torch.int64, device="cuda")


def prepare(case, seed):
    path = case["path"]
    if path == "batch":
        shapes = fields.batch_shapes(case["fields"], case["axis_lo"], case["axis_hi"],
                                     case["shapes"])
        b = dms_batch.Batch(shapes, "cuda")
        b.set_fields([fields.batch_field(i, s, seed, "cuda") for i, s in enumerate(shapes)])
        b.fit()
        b.d0.zero_()  # rows past the pairs are never written
        b.d2.zero_()
        b.capture()
        return {"case": case, "batch": b}
    if path == "stream":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"case": case,
                "fields": [_make(case, seed * 64 + i).cpu().pin_memory()
                           for i in range(case["fields"])],
                "pairs": [np.zeros((int(STREAM_PAIRS * n) + 1024, dms.PAIR_DTYPE.itemsize), np.uint8)
                          for i in range(case["fields"])]}
    f = _make(case, seed)
    if path == "step":
        return {"case": case, "field": f.requires_grad_(True)}
    return {"case": case, "field": f, "lists": _lists(f.numel(), f.dim())}


# ------------------------------------------------------------------ pass --

def _all(r, buf, more=()):
    """Every array of a single-field result, its lists moved to buf."""
    d = r.diagrams
    pairs = [d.d0, d.d2 if isinstance(d, dms.Diagrams) else d.d1, d.d0_essential, *more]
    lists = [*r.crit, *(p.view(torch.int64).view(-1) for p in pairs)]
    n = [int(t.numel()) for t in lists]
    torch.cat(lists, out=buf[:sum(n)])
    out = {"order": r.order.view(torch.int32), "desc": r.grad.desc, "rec": r.grad.rec,
           "lists": buf, "lengths": n}
    if isinstance(d, dms.Diagrams):
        out["counts"] = r.grad.counts
    return out


def run(state):
    case = state["case"]
    path = case["path"]
    if path == "diagram":
        return _all(dms.diagram(state["field"], case.get("pairing", "rounds")), state["lists"])
    if path == "image":
        return _all(dms.diagram2d(state["field"]), state["lists"])
    if path == "step":
        x = state["field"]
        x.grad = None
        loss = dms.topological_loss(x, PERSISTENCE)
        loss.backward()
        return {"loss": loss.detach(), "grad": x.grad}
    if path == "batch":
        b = state["batch"]
        b.replay()
        return {"order": b.order.view(torch.int32), "desc": b.desc, "rec": b.rec,
                "counts": b.counts, "offsets": b.pair_offsets, "essential": b.essential,
                "pairs": [b.d0, b.d2], "status": b.status}
    if path == "stream":
        lengths = []
        for out, mine in zip(dms.diagrams_from_host(state["fields"]), state["pairs"]):
            at = 0
            for p in out:
                mine[at:at + len(p)] = p.view(np.uint8).reshape(len(p), -1)
                at += len(p)
                lengths.append(len(p))
        return {"pairs": state["pairs"], "lengths": lengths}
    f = state["field"]
    r = dms.diagram(f)
    d1 = dms.diagram_d1(f, r.order, r.grad, r.crit, r.diagrams)
    return _all(r, state["lists"], [d1])


def work(case):
    """Bytes of the inputs read once and of the per-vertex outputs written
    once; the lists of critical simplices and of pairs, whose lengths the
    data decides, are left out.  Nothing here multiplies."""
    if case["path"] == "batch":
        shapes = fields.batch_shapes(case["fields"], case["axis_lo"], case["axis_hi"],
                                     case["shapes"])
        return {"bytes": 17 * sum(a * b * c for a, b, c in shapes), "flops": 0}
    n = case["nx"] * case["ny"] * case.get("nz", 1) * case.get("fields", 1)
    # field 4 + order 4 + descending code 1 + record 8 (an image: 2); a step
    # reads the field and writes its gradient; a stream's records stay inside
    per = {"image": 11, "step": 8, "stream": 4}.get(case["path"], 17)
    return {"bytes": per * n, "flops": 0}


# ----------------------------------------------------------------- exact --

def _find(parent, a):
    while parent[a] != a:
        parent[a] = parent[parent[a]]
        a = parent[a]
    return a


def _extremum_pairs(ends, age, saddle_order):
    """Elder rule over a graph: for each saddle (in the given order) that
    joins two components, (saddle, the younger root).  A larger age is
    younger."""
    parent = list(range(len(age)))
    a_of, b_of = ends[0].tolist(), ends[1].tolist()
    out = []
    for s in saddle_order.tolist():
        a, b = _find(parent, a_of[s]), _find(parent, b_of[s])
        if a == b:
            continue
        if age[a] < age[b]:
            a, b = b, a  # a is the younger
        parent[a] = b
        out.append((s, a))
    return out


def _simplices(shape):
    """Vertices of every edge, triangle and tet of the Freudenthal split, as
    [count, 2 / 3 / 4] vertex offsets."""
    nz, ny, nx = shape
    v = np.arange(nz * ny * nx).reshape(shape)

    def corner(c, reach):
        d = [(c >> k) & 1 for k in range(3)]
        r = [(reach >> k) & 1 for k in range(3)]
        return v[d[2]:nz - r[2] + d[2], d[1]:ny - r[1] + d[1], d[0]:nx - r[0] + d[0]].reshape(-1)

    chains = {2: [], 3: [], 4: []}
    for p in range(1, 8):
        chains[2].append((0, p))
        for q in range(p + 1, 8):
            if p & q == p:
                chains[3].append((0, p, q))
                for t in range(q + 1, 8):
                    if q & t == q:
                        chains[4].append((0, p, q, t))
    return [np.concatenate([np.stack([corner(c, ch[-1]) for c in ch], 1) for ch in chains[k]])
            for k in (2, 3, 4)]


def _exact_step(f):
    """(loss, gradient) of the simplification loss in 64 bits: the elder rule
    over all edges (D0) and over all triangles of the dual graph (D2); pairs
    inside one lower star have persistence zero and add nothing."""
    flat = f.reshape(-1)
    n = flat.size
    order = np.empty(n, np.int64)
    order[np.argsort(flat, kind="stable")] = np.arange(n)
    edges, tris, tets = _simplices(f.shape)
    value = flat.astype(np.float64)

    def key(s):  # orders decreasing, as one lexicographic row
        return -np.sort(-order[s], axis=1)

    def top(s):
        return s[np.arange(len(s)), np.argmax(order[s], axis=1)]

    pairs = []
    ke = key(edges)
    for s, m in _extremum_pairs((edges[:, 0], edges[:, 1]), order.tolist(),
                                np.lexsort((ke[:, 1], ke[:, 0]))):
        pairs.append((m, s))
    birth = [np.array([m for m, _ in pairs], np.int64)]
    death = [top(edges)[np.array([s for _, s in pairs], np.int64)]]
    # dual graph: node 0 = outside, node t + 1 = tet t
    st = np.sort(tris, axis=1)
    code = (st[:, 0] * n + st[:, 1]) * n + st[:, 2]
    by = np.argsort(code)
    ends = np.zeros((2, len(tris)), np.int64)
    seen = np.zeros(len(tris), np.int64)
    ts = np.sort(tets, axis=1)
    for omit in range(4):
        cols = [c for c in range(4) if c != omit]
        fc = (ts[:, cols[0]] * n + ts[:, cols[1]]) * n + ts[:, cols[2]]
        at = by[np.searchsorted(code[by], fc)]
        first = np.zeros(len(tets), bool)
        first[np.unique(at, return_index=True)[1]] = True
        for part in (first, ~first):  # a facet may occur twice under one omission
            ends[seen[at[part]], at[part]] = np.nonzero(part)[0] + 1
            np.add.at(seen, at[part], 1)
    kq = key(tets)
    age = np.zeros(len(tets) + 1, np.int64)
    age[1 + np.lexsort((-kq[:, 3], -kq[:, 2], -kq[:, 1], -kq[:, 0]))] = np.arange(1, len(tets) + 1)
    kt = key(tris)
    got = _extremum_pairs((ends[0], ends[1]), age.tolist(),
                          np.lexsort((-kt[:, 2], -kt[:, 1], -kt[:, 0])))
    birth.append(top(tris)[np.array([s for s, _ in got], np.int64)])
    death.append(top(tets)[np.array([t - 1 for _, t in got], np.int64)])
    birth, death = np.concatenate(birth), np.concatenate(death)
    pers = value[death] - value[birth]
    keep = pers < PERSISTENCE
    grad = np.zeros(n)
    np.add.at(grad, death[keep], 2 * pers[keep])
    np.add.at(grad, birth[keep], -2 * pers[keep])
    return float((pers[keep] ** 2).sum()), grad.reshape(f.shape)


def exact(case, seed):
    """Only the differentiable step returns computed numbers (a loss and its
    gradient); every other output is a whole number or a copy of input bits."""
    if case["path"] != "step" or case["nx"] * case["ny"] * case["nz"] > 100_000:
        return None
    loss, grad = _exact_step(_make(case, seed).cpu().numpy())
    return {"loss": torch.tensor(loss, dtype=torch.float64), "grad": torch.from_numpy(grad)}
