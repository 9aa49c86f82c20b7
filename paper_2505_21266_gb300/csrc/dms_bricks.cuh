// The v-paths of the pairing: the words that say where a cell's path goes on,
// and the walks over them.  Host-compilable as well: the CPU tests run these
// on small grids.
#pragma once

#include <cstdint>

#include "dms_grid.cuh"

#ifdef __CUDACC__
#define DMS_OUTLINE __device__ __noinline__
#else
#define DMS_OUTLINE
#endif

namespace dms {

// One step of an ascending dual path, tabulated.  Tet type k (chain
// 0 < c1 < c2 < 7 of its anchor cube) paired with the facet that omits
// chain vertex code - 1 leaves through that facet into the other tet on it:
//  * code 1 omits the anchor: the next tet is anchored at anchor + c1, chain
//    (c2 ^ c1, 7 ^ c1);
//  * code 4 omits the top: anchored at anchor - (7 ^ c2), chain
//    (7 ^ c2, (7 ^ c2) | c1);
//  * code 2 / 3 omit c1 / c2: same anchor, chain (c2 ^ c1, c2) / (c1, c1 | (7 ^ c2)).
// entry(4k + code - 1): next type (bits 0-2), anchor step corner (3-5), step
// sign (6-7: 0 none, 1 plus, 2 minus).
namespace dual_step_detail {
constexpr int c1_of(int k) { return (0x442211 >> (4 * k)) & 15; }
constexpr int c2_of(int k) { return (0x656353 >> (4 * k)) & 15; }
constexpr int type_of(int c1, int c2) { return (c1 >> 1) * 2 + ((c2 ^ c1) > (7 ^ c2) ? 1 : 0); }
constexpr uint64_t entry(int e) {
  const int k = e / 4, code = e % 4 + 1, c1 = c1_of(k), c2 = c2_of(k);
  int stp = 0, sg = 0, n1 = 0, n2 = 0;
  if (code == 1) { stp = c1; sg = 1; n1 = c2 ^ c1; n2 = 7 ^ c1; }
  else if (code == 4) { stp = 7 ^ c2; sg = 2; n1 = stp; n2 = stp | c1; }
  else if (code == 2) { n1 = c2 ^ c1; n2 = c2; }
  else { n1 = c1; n2 = c1 | (7 ^ c2); }
  return (uint64_t)(type_of(n1, n2) | (stp << 3) | (sg << 6));
}
}  // namespace dual_step_detail

// ---------------------------------------------------------------------------
// v-paths by bricks.
//
// A path (vertex -> paired edge -> other vertex; tet -> paired facet -> other
// cofacet) is followed cell by cell only inside bricks of up to 8192 cells, in
// shared memory, for all cells of a brick at once: every cell then knows where
// its path ends or leaves the brick, and a walk hops from brick to brick.
// Every cell has one word:
//   bit 31 set    the end: bits 0..30 the node (0 for OUTSIDE in the dual)
//   bit 31 clear  where the path goes on: bits 13..18 the brick (two bits per
//                 axis: 0, 1, 2 for the one before, this one, the next), bits
//                 0..12 the cell in it
// mark_ends gives the cells at path ends (minima, critical tets) their nodes
// first; resolve_paths reads them there.
// Followed cell by cell through memory, one load and one claim by
// compare-and-swap per step, a walk was a chain of 3 (vertices) and 10 (tets)
// dependent steps on average on noise, up to 400 on smooth fields, 1 us each;
// hops are 1.3 to 2.7 on average, up to 27.  Resolving all cells costs about
// 100 instructions per tet and a word per cell written, which noise, whose
// paths are short, pays back in fewer random reads: D0/D2 stage 64^3 mixture
// 705 -> 356 us, 128^3 smooth 953 -> 368 us, 16384^2 37.8 -> 30.8 ms, 512^3
// ties 28.9 -> 25.3 ms, 1024^3 87.7 -> 73.5 ms (of it a dual step as a sum on
// the cell's word, in place of packed coordinates: 1.5, and the walks' loop
// without a count of the grid's cells: 2).  Following every cell to its
// end in turn instead of doubling took 147 ms there.
// ---------------------------------------------------------------------------
constexpr uint32_t kEnd = 0x80000000u;
constexpr uint32_t kNoMark = kEnd | 0x7FFFFFFFu;  // an end without a node, or bad data
constexpr uint32_t kLoop = kEnd | 0x7FFFFFFEu;    // a path that does not end (bad data)
constexpr uint32_t kFinal = 0x40000000u;          // (in shared memory) a way on, out of the brick

// one field for the whole call
struct OneField {
  Grid g;
  DMS_HD void get(int64_t, Grid& out, int64_t& off) const {
    out = g;
    off = 0;
  }
  // brick id of 2^lx x 2^ly x 2^lz vertices: its field, its place in it
  DMS_HD void brick(int64_t id, int lx, int ly, int lz, Grid& out, int64_t& off,
                                        int& bx, int& by, int& bz) const {
    get(0, out, off);
    const uint32_t tx = (uint32_t)((g.nx + (1 << lx) - 1) >> lx), ty = (uint32_t)((g.ny + (1 << ly) - 1) >> ly);
    const uint32_t i = (uint32_t)id, r = i / tx;
    bx = (int)(i - r * tx);
    bz = (int)(r / ty);
    by = (int)(r - (uint32_t)bz * ty);
    (void)lz;
  }
};

// A cell of a brick: its vertex's coordinates in one word, eight bits per
// axis, each offset by the brick's extent, so that after a step the bits above
// the coordinate's say which brick it is in: 0, 1 (this one) or 2.
template <class P>
DMS_HD uint32_t packed_coords(int lv) {
  return ((lv & ((1 << P::LX) - 1)) + (1 << P::LX)) |
         (((lv >> P::LX) & ((1 << P::LY) - 1)) + (1 << P::LY)) << 8 |
         ((lv >> (P::LX + P::LY)) + (1 << P::LZ)) << 16;
}
DMS_HD constexpr uint32_t packed_step(int dx, int dy, int dz) {
  return (uint32_t)(dx + dy * 256 + dz * 65536);
}
// cell k of the vertex at c as a word: a cell of the brick, or a way out of it
template <class P>
DMS_HD uint32_t brick_word(uint32_t c, int k) {
  const uint32_t lv = (c & ((1u << P::LX) - 1)) | (c >> 8 & ((1u << P::LY) - 1)) << P::LX |
                      (c >> 16 & ((1u << P::LZ) - 1)) << (P::LX + P::LY);
  const uint32_t dir = (c >> P::LX & 3u) | (c >> (8 + P::LY) & 3u) << 2 | (c >> (16 + P::LZ) & 3u) << 4;
  const uint32_t local = lv * P::K + k;
  return dir == 21u ? local : kFinal | dir << 13 | local;
}
// is the vertex at c inside [0, mx) x [0, my) x [0, mz) of the brick at (x0, y0, z0)
template <class P>
DMS_HD bool inside(uint32_t c, int x0, int y0, int z0, uint32_t mx, uint32_t my,
                                       uint32_t mz) {
  return (uint32_t)(x0 + (int)(c & 255u) - (1 << P::LX)) < mx &&
         (uint32_t)(y0 + (int)(c >> 8 & 255u) - (1 << P::LY)) < my &&
         (uint32_t)(z0 + (int)(c >> 16) - (1 << P::LZ)) < mz;
}
// (A policy's cells() replaces the words that are not kNoMark.)
// the word of the end of a path: the node that mark_ends gave the cell (ends
// that are not in the list have none: bad data)
DMS_HD uint32_t end_word(const uint32_t* path, int64_t cell, const int64_t* list,
                                             int64_t n, uint32_t node0) {
  const uint32_t w = path[cell];
  const int64_t i = (int64_t)(w & ~kEnd) - node0;
  return (w & kEnd) && i >= 0 && i < n && ro(list + i) == cell ? w : kNoMark;
}

// a cell that a path is followed to without words: its vertex, its number there,
// and 0 or, at the path's end, the end's word
struct Cell {
  uint32_t w;
  int x, y, z, k;
};
DMS_HD bool within(const Cell& c, int64_t mx, int64_t my, int64_t mz) {
  return (uint32_t)c.x < (uint32_t)mx && (uint32_t)c.y < (uint32_t)my && (uint32_t)c.z < (uint32_t)mz;
}

// D0: descending paths from vertex to vertex, to a minimum
template <class F>
struct DescPaths {
  static constexpr int K = 1, LX = 4, LY = 4, LZ = 4;
  F fields;
  const uint8_t* desc;
  const int64_t* ends;  // the path ends' cells, their number (n_dev or n)
  const int64_t* n_dev;
  int64_t n;
  DMS_HD void cells(const Grid& g, const uint32_t* path, int64_t v, int lv, int x0,
                                        int y0, int z0, bool border, uint32_t (&w)[K]) const {
    const int d = ro(desc + v);
    if (d >= 14) {
      if (d == 15) w[0] = end_word(path, v, ends, n_dev ? *n_dev : n, 0);
      return;
    }
    const int c = (0x7653421 >> (4 * (d < 7 ? d : d - 7))) & 15, s = d < 7 ? 1 : -1;
    const uint32_t to = packed_coords<DescPaths>(lv) +
                        s * packed_step(c & 1, (c >> 1) & 1, (c >> 2) & 1);
    const bool out = border && !inside<DescPaths>(to, x0, y0, z0, (uint32_t)g.nx, (uint32_t)g.ny, (uint32_t)g.nz);
    if (!out) w[0] = brick_word<DescPaths>(to, 0);  // (outside: bad data)
  }
  // the same for one cell
  DMS_HD void step(const Grid& g, const uint32_t* path, int64_t v, Cell& c) const {
    const int d = ro(desc + v);
    c.w = kNoMark;
    if (d >= 14) {
      if (d == 15) c.w = end_word(path, v, ends, n_dev ? *n_dev : n, 0);
      return;
    }
    const int o = (0x7653421 >> (4 * (d < 7 ? d : d - 7))) & 15, s = d < 7 ? 1 : -1;
    c.x += s * (o & 1);
    c.y += s * ((o >> 1) & 1);
    c.z += s * ((o >> 2) & 1);
    if (within(c, g.nx, g.ny, g.nz)) c.w = 0;  // (outside: bad data)
  }
};

// the steps of the dual paths from tet type k with code c, at 4 k + c - 1, and
// the type they lead to (codes 2 and 3 stay at the anchor)
struct DualSteps {
  uint32_t step[24];
  uint8_t type[24];
};
constexpr DualSteps make_dual_steps() {
  DualSteps t{};
  for (int e = 0; e < 24; ++e) {
    const uint64_t w = dual_step_detail::entry(e);
    const int c = (int)(w >> 3) & 7, sg = (int)(w >> 6) == 1 ? 1 : ((int)(w >> 6) == 2 ? -1 : 0);
    t.step[e] = (uint32_t)(sg * ((c & 1) + ((c >> 1) & 1) * 256 + ((c >> 2) & 1) * 65536));
    t.type[e] = (uint8_t)(w & 7);
  }
  return t;
}

// D2: ascending dual paths from tet to tet, to a critical one or out of the
// grid (node 0, OUTSIDE)
template <class F>
struct DualPaths {
  static constexpr int K = 6, LX = 4, LY = 3, LZ = 3;
  F fields;
  const uint64_t* rec;
  const int64_t* ends;
  const int64_t* n_dev;
  int64_t n;
  DMS_HD void cells(const Grid& g, const uint32_t* path, int64_t v, int lv, int x0,
                                        int y0, int z0, bool border, uint32_t (&w)[K]) const {
    constexpr DualSteps st = make_dual_steps();
    constexpr int L[3] = {LX, LY, LZ};
    const uint32_t hi = (uint32_t)(ro(rec + v) >> 32), at = packed_coords<DualPaths>(lv);
    // a step goes up or down one axis: what it adds to the cell's word, with
    // the wrap and the brick where it leaves this one
    uint32_t up[3], down[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int shift = a == 0 ? 0 : (a == 1 ? LX : LX + LY), last = (1 << L[a]) - 1;
      const int at_axis = (lv >> shift) & last, one = K << shift;
      up[a] = at_axis == last ? kFinal + ((21 + (1 << 2 * a)) << 13) - last * one : one;
      down[a] = at_axis == 0 ? kFinal + ((21 - (1 << 2 * a)) << 13) + last * one : 0u - one;
    }
    const uint32_t base = (uint32_t)lv * K;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const uint32_t code = (hi >> (1 + 3 * k)) & 7u;
      if (code == 7u) {
        w[k] = end_word(path, v * 6 + k, ends, n_dev ? *n_dev : n, 1);
      } else if (code >= 1u && code <= 4u) {  // (else no tet there, or bad data)
        const int u = dual_step_detail::c1_of(k) >> 1, d = (7 ^ dual_step_detail::c2_of(k)) >> 1;
        const uint32_t add = code == 1u ? up[u] + st.type[4 * k]
                             : (code == 2u ? st.type[4 * k + 1]
                                : (code == 3u ? st.type[4 * k + 2] : down[d] + st.type[4 * k + 3]));
        // (tet anchors lie below the last vertex in every axis)
        const bool out = border && !inside<DualPaths>(
                                       at + (code == 1u ? st.step[4 * k] : (code == 4u ? st.step[4 * k + 3] : 0u)),
                                       x0, y0, z0, (uint32_t)(g.nx - 1), (uint32_t)(g.ny - 1), (uint32_t)(g.nz - 1));
        w[k] = out ? kEnd : base + add;  // out: OUTSIDE
      }
    }
  }
  DMS_HD void step(const Grid& g, const uint32_t* path, int64_t v, Cell& c) const {
    const uint32_t code = (uint32_t)(ro(rec + v) >> (33 + 3 * c.k)) & 7u;
    c.w = kNoMark;
    if (code == 7u) c.w = end_word(path, v * 6 + c.k, ends, n_dev ? *n_dev : n, 1);
    if (code < 1u || code > 4u) return;
    const int c1 = dual_step_detail::c1_of(c.k), c2 = dual_step_detail::c2_of(c.k);
    const int o = code == 1u ? c1 : (code == 4u ? 7 ^ c2 : 0), s = code == 1u ? 1 : -1;
    const int n1 = code == 3u ? c1 : (code == 4u ? 7 ^ c2 : c2 ^ c1);
    const int n2 = code == 1u ? 7 ^ c1 : (code == 2u ? c2 : c1 | (7 ^ c2));
    c.k = dual_step_detail::type_of(n1, n2);
    c.x += s * (o & 1);
    c.y += s * ((o >> 1) & 1);
    c.z += s * ((o >> 2) & 1);
    c.w = within(c, g.nx - 1, g.ny - 1, g.nz - 1) ? 0 : kEnd;  // out: OUTSIDE
  }
};

// ---- images (Grid with nz = 1)
DMS_HD int corner2(int s) { return (s % 3) + 1; }  // {1,2,3}

// D0: down the vertex-edge pairs (desc) to a minimum
struct DescPaths2d {
  static constexpr int K = 1, LX = 5, LY = 5, LZ = 0;
  OneField fields;
  const uint8_t* desc;
  const int64_t* ends;
  int64_t n;
  DMS_HD void cells(const Grid& g, const uint32_t* path, int64_t v, int lv, int x0,
                                        int y0, int, bool, uint32_t (&w)[K]) const {
    const int d = ro(desc + v);
    if (d >= 6) {
      if (d == 15) w[0] = end_word(path, v, ends, n, 0);
      return;
    }
    const int c = corner2(d), s = d < 3 ? 1 : -1;
    const uint32_t to = packed_coords<DescPaths2d>(lv) + s * packed_step(c & 1, (c >> 1) & 1, 0);
    const bool in = inside<DescPaths2d>(to, x0, y0, 0, (uint32_t)g.nx, (uint32_t)g.ny, 1u);
    if (in) w[0] = brick_word<DescPaths2d>(to, 0);  // (outside: bad data)
  }
};

// D1: from a triangle through the edge it is paired with to that edge's other
// triangle, up to a maximum (node j + 1) or out of the grid (OUTSIDE, node 0)
struct DualPaths2d {
  static constexpr int K = 2, LX = 5, LY = 5, LZ = 0;
  OneField fields;
  const uint16_t* rec;
  const int64_t* ends;
  int64_t n;
  DMS_HD void cells(const Grid& g, const uint32_t* path, int64_t v, int lv, int x0,
                                        int y0, int, bool, uint32_t (&w)[K]) const {
    const uint32_t rw = ro(rec + v), at = packed_coords<DualPaths2d>(lv);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t code = (rw >> (9 + 3 * k)) & 7u;
      if (code == 7u) {
        w[k] = end_word(path, v * 2 + k, ends, n, 1);
      } else if (code >= 1u && code <= 3u) {  // (else no triangle there, or bad data)
        // across the facet that omits chain vertex code - 1: the diagonal
        // (code 2): the square's other triangle; type 0 (code 1 / 3): the
        // square to the right / below; type 1: above / to the left
        const uint32_t to = at + (code == 2u ? 0u : (code == 1u ? (k == 0 ? packed_step(1, 0, 0) : packed_step(0, 1, 0))
                                                          : (k == 0 ? packed_step(0, -1, 0) : packed_step(-1, 0, 0))));
        const bool in = inside<DualPaths2d>(to, x0, y0, 0, (uint32_t)(g.nx - 1), (uint32_t)(g.ny - 1), 1u);
        w[k] = in ? brick_word<DualPaths2d>(to, 1 - k) : kEnd;
      }
    }
  }
};

template <class P>
int64_t brick_count(int64_t nx, int64_t ny, int64_t nz) {
  return ((nx + (1 << P::LX) - 1) >> P::LX) * ((ny + (1 << P::LY) - 1) >> P::LY) *
         ((nz + (1 << P::LZ) - 1) >> P::LZ);
}

// a walk: the word of its cell and the brick of that cell (Path: the words,
// const uint32_t* on the device)
struct Walk {
  uint32_t w;
  int bx, by, bz;
};
template <class P, class Path>
DMS_HD Walk walk_from(Path path, const Grid& g, int64_t v, int x, int y, int z,
                                          int k) {
  return Walk{ro(path + v * P::K + k), x >> P::LX, y >> P::LY, z >> P::LZ};
}
template <class P, class Path>
DMS_HD void walk_hop(Path path, const Grid& g, int64_t off, Walk& a) {
  const uint32_t local = a.w & 8191u, lv = local / P::K;
  a.bx += (int)(a.w >> 13 & 3u) - 1;
  a.by += (int)(a.w >> 15 & 3u) - 1;
  a.bz += (int)(a.w >> 17 & 3u) - 1;
  const int x = (a.bx << P::LX) + (int)(lv & ((1 << P::LX) - 1));
  const int y = (a.by << P::LY) + (int)((lv >> P::LX) & ((1 << P::LY) - 1));
  const int z = (a.bz << P::LZ) + (int)(lv >> (P::LX + P::LY));
  a.w = ro(path + (off + x + g.nx * y + g.sxy * z) * P::K + (local - lv * P::K));
}
// The end of a walk from a: where it goes on is a function of its word and
// brick, so a walk that meets one it had before loops (bad data).  It keeps one
// and compares, keeping a new one after 1, 2, 4, ... hops (Brent's method): a
// loop ends after about three times the hops that lead to it and once round.
template <class P, class Path>
DMS_OUTLINE uint32_t walk_on(Path path, const Grid& g, int64_t off, Walk a) {
  for (uint64_t span = 1;; span *= 2) {
    const Walk was = a;
    for (uint64_t i = 0; i < span; ++i) {
      if (a.w & kEnd) return a.w;
      walk_hop<P>(path, g, off, a);
      if (a.w == was.w && a.bx == was.bx && a.by == was.by && a.bz == was.bz) return kLoop;
    }
  }
}
// both walks of a saddle to their ends, their loads in flight together, the
// rest of a long one by itself: valid paths took up to 27 hops
constexpr int kFewHops = 128;
template <class P, class Path>
DMS_HD void walk_both(Path path, const Grid& g, int64_t off, Walk& a, Walk& b) {
  for (int it = 0; it < kFewHops && !(a.w & b.w & kEnd); ++it) {
    if (!(a.w & kEnd)) walk_hop<P>(path, g, off, a);
    if (!(b.w & kEnd)) walk_hop<P>(path, g, off, b);
  }
  if (!(a.w & kEnd)) a.w = walk_on<P>(path, g, off, a);
  if (!(b.w & kEnd)) b.w = walk_on<P>(path, g, off, b);
}

// ---------------------------------------------------------------------------
// Few saddles on a large grid, or a thin one: paths cell by cell, no brick
// resolved.
//
// Walks that meet go on as one.  One vertex in eight is a landmark: the first
// walk at a cell of it claims the cell's word, a later one stops there with a
// link to the first.  So only the landmarks' words need clearing, and a walk
// goes only a few steps along a path that another has taken.  Words: kNoMark
// free, kEnd | node an end (mark_ends), kLink | walk claimed.  A walk's result:
// an end, a link, or 0: a path, or a chain of links, too long for this (a walk
// that loops, of bad data, among them), whose saddle waits for the bricks.
//
// Both bounds keep winding paths, one dependent load of 0.7 us per cell, from
// costing more than a few ms ahead of the bricks; smooth fields of 1024^3
// stay below.  Landmarks are 8 in a row of every 64, so that clearing writes
// whole sectors: D0/D2 stage of 1024^3 mixtures with noise 0, 1e-3 and 2e-3
// (2e-7, 2.3e-3 and 9e-3 saddles per vertex) 3.7, 7.3 and 17.8 ms; one in 16
// anywhere 7.9, 12.2 and 24.6; 4 of 64 3.3, 7.4 and 19.4; 16 of 64 4.7, 8.4
// and 18.6; without claims 1.5, 16.0 and 58.
// ---------------------------------------------------------------------------
constexpr uint32_t kLink = 0x40000000u;  // (with fewer than 2^30 walks)
constexpr int kFewSteps = 4096, kFewLinks = 4096;
constexpr int kRun = 64, kGroup = 8;
DMS_HD uint32_t landmarks_of(int64_t run) {  // place of a run's first landmark, by a hash
  return ((uint32_t)run * 2654435761u) / (uint32_t)(0x100000000ull * kGroup / kRun) * kGroup;
}
DMS_HD bool is_landmark(int64_t v) { return ((uint32_t)v % kRun) / kGroup * kGroup == landmarks_of(v / kRun); }
DMS_HD uint32_t claim(uint32_t* word, uint32_t me) {  // the word as it was
#ifdef __CUDA_ARCH__
  return atomicCAS(word, kNoMark, me);
#else
  const uint32_t w = *word;
  if (w == kNoMark) *word = me;
  return w;
#endif
}
// walk number j from cell c: its result
template <class P>
DMS_HD uint32_t follow(const P& p, const Grid& g, uint32_t* path, Cell c, uint32_t j) {
  for (int it = 0; it < kFewSteps && !(c.w & kEnd); ++it) {
    const int64_t v = c.x + g.nx * c.y + g.sxy * c.z;
    if (is_landmark(v)) {
      const uint32_t w = claim(path + v * P::K + c.k, kLink | j);
      if (!(w & kEnd)) return w;
    }
    p.step(g, path, v, c);
  }
  return c.w;
}
// walk j's end, or 0.  Its result becomes what it leads to at every link, for
// those that link here: chains shorten while they are followed.
DMS_HD uint32_t end_of(volatile uint32_t* results, int64_t j) {
  uint32_t w = results[j];
  for (int it = 0; it < kFewLinks && w & kLink && !(w & kEnd); ++it) results[j] = w = results[w & ~kLink];
  return w & kEnd ? w : 0;
}

}  // namespace dms
