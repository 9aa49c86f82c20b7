// Host build of the v-path words and walks (dms_bricks.cuh): the words of a
// field's cells as a brick's CTA forms them, every one followed to where it
// leaves its brick, and the walks over them.  For test_brick_walks.py.
#include <type_traits>
#include <vector>

#include "dms_bricks.cuh"

namespace dms {
// words whose reads are counted
struct Counted {
  const uint32_t* p;
  int64_t* reads;
  Counted operator+(int64_t i) const { return Counted{p + i, reads}; }
};
inline uint32_t ro(const Counted& c) {
  ++*c.reads;
  return *c.p;
}
}  // namespace dms

using namespace dms;

namespace {

// (what a brick's CTA does, a cell at a time)
template <class P>
void resolve(const P& p, const Grid& g, uint32_t* path) {
  constexpr int VERTS = 1 << (P::LX + P::LY + P::LZ), CELLS = VERTS * P::K;
  for (int64_t id = 0; id < brick_count<P>(g.nx, g.ny, g.nz); ++id) {
    Grid gg;
    int64_t off;
    int bx, by, bz;
    p.fields.brick(id, P::LX, P::LY, P::LZ, gg, off, bx, by, bz);
    const int x0 = bx << P::LX, y0 = by << P::LY, z0 = bz << P::LZ;
    const bool border = bx == 0 || by == 0 || bz == 0 || x0 + (1 << P::LX) >= g.nx - 1 ||
                        y0 + (1 << P::LY) >= g.ny - 1 || z0 + (1 << P::LZ) >= g.nz - 1;
    std::vector<uint32_t> s(CELLS, kNoMark);
    auto vertex = [&](int lv) -> int64_t {
      const int x = x0 + (lv & ((1 << P::LX) - 1)), y = y0 + ((lv >> P::LX) & ((1 << P::LY) - 1));
      const int z = z0 + (lv >> (P::LX + P::LY));
      return x < g.nx && y < g.ny && z < g.nz ? x + g.nx * y + g.sxy * z : -1;
    };
    for (int lv = 0; lv < VERTS; ++lv) {
      uint32_t w[P::K];
      for (int k = 0; k < P::K; ++k) w[k] = kNoMark;
      if (vertex(lv) >= 0) p.cells(gg, path, vertex(lv), lv, x0, y0, z0, border, w);
      for (int k = 0; k < P::K; ++k) s[lv * P::K + k] = w[k];
    }
    for (int c = 0; c < CELLS; ++c) {
      if (vertex(c / P::K) < 0) continue;
      uint32_t w = s[c];
      for (int it = 0; it < CELLS && !(w & (kEnd | kFinal)); ++it) w = s[w];
      if (!(w & (kEnd | kFinal))) w = kLoop;
      path[vertex(c / P::K) * P::K + c % P::K] = w & kEnd ? w : w & ~kFinal;
    }
  }
}

template <class P>
void ends_of(const Grid& g, const uint32_t* path, const int64_t* cells, int64_t n, uint32_t* out) {
  for (int64_t i = 0; i < n; ++i) {
    Walk w[2];
    for (int j = 0; j < 2; ++j) {
      const int64_t c = cells[2 * i + j], v = c / P::K;
      w[j] = c < 0 ? Walk{kEnd, 0, 0, 0}
                   : walk_from<P>(path, g, v, (int)(v % g.nx), (int)(v / g.nx % g.ny), (int)(v / g.sxy),
                                  (int)(c % P::K));
    }
    walk_both<P>(path, g, 0, w[0], w[1]);
    out[2 * i] = w[0].w;
    out[2 * i + 1] = w[1].w;
  }
}

// the same cell by cell, no brick resolved, the walks in the order given: as
// one after the other, then their links
template <class P>
void cell_ends_of(const P& p, const Grid& g, uint32_t* path, const int64_t* cells, int64_t n,
                  const int64_t* order, uint32_t* out) {
  for (int64_t i = 0; i < 2 * n; ++i) {
    const int64_t j = order[i], at = cells[j], v = at / P::K;
    const Cell c = at < 0 ? Cell{kEnd, 0, 0, 0, 0}
                          : Cell{0, (int)(v % g.nx), (int)(v / g.nx % g.ny), (int)(v / g.sxy), (int)(at % P::K)};
    out[j] = follow(p, g, path, c, (uint32_t)j);
  }
  for (int64_t j = 0; j < 2 * n; ++j) out[j] = end_of(out, j);
}
template <class P>
std::vector<uint32_t> marked(const Grid& g, const int64_t* ends, int64_t n, uint32_t node0) {
  // (what no one wrote: anything)
  std::vector<uint32_t> path(g.n * P::K);
  for (size_t c = 0; c < path.size(); ++c) path[c] = (uint32_t)(c * 2654435761u);
  for (int64_t v = 0; v < g.n; ++v)
    for (int k = 0; k < P::K && is_landmark(v); ++k) path[v * P::K + k] = kNoMark;
  for (int64_t i = 0; i < n; ++i) path[ends[i]] = kEnd | (uint32_t)(i + node0);
  return path;
}

Grid grid(int64_t nx, int64_t ny, int64_t nz) { return Grid{nx, ny, nz, nx * ny * nz, nx * ny}; }

}  // namespace

extern "C" {

// ends: the cells of the nodes.  starts: two cells per saddle (-1: outside).
// order: cell by cell, the walks in this order (null: over the bricks).  out:
// the words of their ends.
int host_desc_ends(const uint8_t* desc, int64_t nx, int64_t ny, int64_t nz, const int64_t* ends,
                   int64_t nends, const int64_t* starts, int64_t n, const int64_t* order, uint32_t* out) {
  const Grid g = grid(nx, ny, nz);
  std::vector<uint32_t> path = marked<DescPaths<OneField>>(g, ends, nends, 0);
  const DescPaths<OneField> p{OneField{g}, desc, ends, nullptr, nends};
  if (order) return cell_ends_of(p, g, path.data(), starts, n, order, out), 0;
  resolve(p, g, path.data());
  ends_of<std::decay_t<decltype(p)>>(g, path.data(), starts, n, out);
  return 0;
}
int host_dual_ends(const uint64_t* rec, int64_t nx, int64_t ny, int64_t nz, const int64_t* ends,
                   int64_t nends, const int64_t* starts, int64_t n, const int64_t* order, uint32_t* out) {
  const Grid g = grid(nx, ny, nz);
  std::vector<uint32_t> path = marked<DualPaths<OneField>>(g, ends, nends, 1);
  const DualPaths<OneField> p{OneField{g}, rec, ends, nullptr, nends};
  if (order) return cell_ends_of(p, g, path.data(), starts, n, order, out), 0;
  resolve(p, g, path.data());
  ends_of<std::decay_t<decltype(p)>>(g, path.data(), starts, n, out);
  return 0;
}

// A walk through `lead` bricks, row by row of 32, and then round a ring of 2 x
// `half` bricks (half 0: to an end, node 7), over words made for it.  Returns
// the words it read; *out is its end.
int64_t host_long_walk(int64_t rows, int64_t half, uint32_t* out) {
  const Grid g = grid(512, 1024, 16);
  std::vector<uint32_t> path(g.n, kNoMark);
  auto cell = [&](int x, int y) -> int64_t { return 16 * x + g.nx * 16 * y; };
  auto go = [&](int x, int y, int X, int Y) {
    path[cell(x, y)] = (uint32_t)((X - x + 1) | (Y - y + 1) << 2 | 1 << 4) << 13;
  };
  for (int y = 0; y < rows; ++y)
    for (int i = 0; i < 32; ++i) {
      const int x = y & 1 ? 31 - i : i;
      if (i < 31) go(x, y, y & 1 ? x - 1 : x + 1, y);
      else go(x, y, x, y + 1);
    }
  const int y = (int)rows;
  if (half == 0) path[cell(rows & 1 ? 31 : 0, y)] = kEnd | 7u;
  for (int x = 0; x < half; ++x) {
    if (x + 1 < half) go(x, y, x + 1, y);
    else go(x, y, x, y + 1);
    if (x > 0) go(x, y + 1, x - 1, y + 1);
    else go(x, y + 1, x, y);
  }
  int64_t reads = 0;
  const Counted c{path.data(), &reads};
  Walk a = walk_from<DescPaths<OneField>>(c, g, cell(0, 0), 0, 0, 0, 0), b{kEnd | 3u, 0, 0, 0};
  walk_both<DescPaths<OneField>>(c, g, 0, a, b);
  *out = a.w;
  return b.w == (kEnd | 3u) ? reads : -1;
}

}  // extern "C"
