// ProcessLowerStars (Robins et al., Sec. 2.3) as a rule per edge of the grid
// plus a correction per vertex.  Host-compilable as well: the CPU tests run
// the same tables, rule and correction through process_lower_star.
//
// The lower star L(x) is the cone over the lower link of x (the link of x, a
// triangulated sphere on the 14 neighbours, restricted to the neighbours that
// precede x).  ProcessLowerStars pairs the link's vertices, edges and
// triangles (the edges, triangles and tets of L(x)); what its queues do, in
// key order, has this closed form:
//   * the link's vertices and edges: every component of the lower link has its
//     minimum spanning tree under the key order (PQone's edges are Prim's
//     algorithm), rooted at the component's lowest vertex; a vertex is paired
//     with the tree edge towards the root.  The lowest root of all is paired
//     with x itself, every other root is critical;
//   * the link's triangles and the edges outside the trees: the dual graph,
//     whose nodes are the link triangles and one node R for everything outside
//     the lower link, joined across the edges outside the trees.  A triangle
//     with one unclassified edge is a leaf of that graph; popping leaves in
//     any order gives the same pairs, and when none is left PQzero makes the
//     smallest remaining edge critical, which removes the smallest edge of a
//     cycle.  What remains is the dual graph's maximum spanning tree, rooted
//     at R: a triangle is paired with its tree edge towards R.  When the lower
//     link is the whole sphere there is no R; the leaf of smallest key goes
//     first, so the triangle of largest key is left as the root: critical.
//
// Both trees are built as in 2D, by the lower stars of the link's vertices.
// Take a lower neighbour y of x: its link inside the link of x is the cycle
// of 4 or 6 vertices around the edge {x, y}, and the ones below y form arcs of
// that cycle.
//   * One proper arc (the usual case): y is paired with the arc's lowest
//     vertex w, the remaining edges of the arc with its triangles, each with
//     its edge farther from w.  All of this belongs to the one edge {x, y}, so
//     it is decided once per edge of the grid, from the 4 or 6 orders around
//     it, by a table (edge_entry): per vertex 7 edges, not 14 neighbours, 36
//     triangles and 24 tets.
//   * No arc: y is a local minimum of the link of x, a root of the first tree.
//   * Several arcs: each further arc has an edge {y, its lowest vertex} that
//     either joins two trees (Kruskal: the vertices from one end to the
//     younger root change their tree edge) or closes a cycle.
//   * The whole cycle: y is a local maximum of the link of x; one triangle of
//     its cycle stays unpaired, a root of the second forest.
// If every lower neighbour but one has one proper arc, nothing is left to do:
// the rules' pairs form the two trees.  Otherwise (correct_star) the edges of
// the further arcs are visited in increasing key order and join trees, then
// those that closed cycles in decreasing order and join dual trees, an older
// root (lower vertex, higher triangle, R oldest) absorbing the younger one by
// reversing the path to it; an edge that closes cycles in both is critical.
#pragma once

#include <cstdint>
#include <type_traits>

#include "dms_star.cuh"

#ifdef __CUDACC__
#define DMS_HD __host__ __device__ __forceinline__
#define DMS_ROLLED _Pragma("unroll 1")  // a loop kept rolled: its code has to stay in cache
#else
#define DMS_HD inline
#define DMS_ROLLED
#endif

namespace dms {
namespace lowerstar {

// compile-time loop: f(std::integral_constant<int, I>) for I in [B, E)
template <int B, int E, class F>
DMS_HD void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}

DMS_HD int ffs32(uint32_t m) {
#ifdef __CUDA_ARCH__
  return __ffs((int)m) - 1;
#else
  return m ? __builtin_ctz(m) : -1;
#endif
}
DMS_HD int ffs64(uint64_t m) {
#ifdef __CUDA_ARCH__
  return __ffsll((long long)m) - 1;
#else
  return m ? __builtin_ctzll(m) : -1;
#endif
}
DMS_HD uint32_t umax(uint32_t a, uint32_t b) { return a > b ? a : b; }
DMS_HD uint32_t umin(uint32_t a, uint32_t b) { return a < b ? a : b; }

// ------------------------------------------------------- the edge's cycle --
// The vertices around the edge from a vertex to its neighbour in slot s, in
// cyclic order, as slots of that vertex; the star tet between positions i and
// i + 1.  Slot s and slot s + 7 are the same edge seen from its two ends, and
// list the same vertices in the same order.
struct Cycles {
  int n[14];
  int v[14][6];    // slots
  int tet[14][6];  // star tets
};
constexpr int slot_of(I3 d) {
  for (int s = 0; s < 14; ++s)
    if (kStar.off[s][0] == d.x && kStar.off[s][1] == d.y && kStar.off[s][2] == d.z) return s;
  return -1;
}
constexpr bool slots_adjacent(int a, int b) {
  return star_detail::adjacent(I3{kStar.off[a][0], kStar.off[a][1], kStar.off[a][2]},
                               I3{kStar.off[b][0], kStar.off[b][1], kStar.off[b][2]});
}
constexpr int star_tet(int a, int b, int c) {
  for (int q = 0; q < 24; ++q) {
    const uint32_t m = (1u << kStar.tetA[q]) | (1u << kStar.tetB[q]) | (1u << kStar.tetC[q]);
    if (m == ((1u << a) | (1u << b) | (1u << c))) return q;
  }
  return -1;
}
constexpr Cycles make_cycles() {
  Cycles c{};
  for (int s = 0; s < 7; ++s) {
    int n = 0;
    bool used[14] = {};
    for (int t = 0; t < 14 && n == 0; ++t)
      if (slots_adjacent(s, t)) {
        c.v[s][n++] = t;
        used[t] = true;
      }
    for (bool more = true; more;) {
      more = false;
      for (int t = 0; t < 14 && !more; ++t)
        if (!used[t] && slots_adjacent(s, t) && slots_adjacent(t, c.v[s][n - 1])) {
          c.v[s][n++] = t;
          used[t] = more = true;
        }
    }
    c.n[s] = c.n[s + 7] = n;
    for (int i = 0; i < n; ++i) {
      const int t = c.v[s][i];
      c.v[s + 7][i] = slot_of(I3{kStar.off[t][0] - kStar.off[s][0], kStar.off[t][1] - kStar.off[s][1],
                                 kStar.off[t][2] - kStar.off[s][2]});
    }
  }
  for (int s = 0; s < 14; ++s)
    for (int i = 0; i < c.n[s]; ++i)
      c.tet[s][i] = star_tet(s, c.v[s][i], c.v[s][(i + 1) % c.n[s]]);
  return c;
}
constexpr Cycles kCyc = make_cycles();
constexpr bool cycles_ok() {
  for (int s = 0; s < 14; ++s) {
    if (kCyc.n[s] != (s % 7 >= 3 && s % 7 < 6 ? 4 : 6)) return false;
    for (int i = 0; i < kCyc.n[s]; ++i)
      if (kCyc.v[s][i] < 0 || kCyc.tet[s][i] < 0 || (s < 7 && kCyc.v[s][i] == 13)) return false;
  }
  return true;
}
static_assert(cycles_ok(), "cycles of 6 around axis and space diagonals, 4 around face diagonals");

// record code of star tet q paired with its facet that omits slot u
constexpr int code_omitting(int q, int u) {
  const int w = u == kStar.tetC[q] ? 0 : (u == kStar.tetB[q] ? 1 : 2);
  return kStar.facetCode[q][w];
}
// position of the triangle on slots (s, u) among the cofacets of the edge s
constexpr int cof_of(int s, int u) {
  for (int j = 0; j < 36; ++j) {
    if (kStar.triA[j] == s && kStar.triB[j] == u) return kStar.cofIdx[j][0];
    if (kStar.triB[j] == s && kStar.triA[j] == u) return kStar.cofIdx[j][1];
  }
  return -1;
}

// ------------------------------------------------------------- the rule --
// What the edge {x, y} (x the higher end, type t) decides, for the set L of
// cycle positions below y and the position w of the cycle's lowest vertex:
// bits 1 + 3k .. 3 + 3k the code of the tet of type k around the edge (every
// tet type occurs at most once around an edge, so the codes need no anchor),
// bits 27..28 the edge's kind, bits 29..31 its code.
enum : uint32_t { kPlain = 0, kEmpty = 1, kArcs = 2, kWhole = 3 };
constexpr int kTetBit = 1, kKindBit = 27, kEdgeBit = 29;

constexpr int entry_base(int t) { return t == 6 ? 1536 : (t < 3 ? 512 * t : 2048 + 64 * (t - 3)); }
constexpr int kEntries = 2560;  // (the last rows are filling, see edge_offset)

constexpr uint32_t edge_entry(int t, uint32_t L, int w) {
  const int n = kCyc.n[t];
  if (L == 0) return kEmpty << kKindBit;
  if (w >= n || !((L >> w) & 1)) return 0;  // not met: the lowest vertex is below y
  int arcs = 0;
  for (int i = 0; i < n; ++i) arcs += ((L >> i) & 1) && !((L >> ((i + 1) % n)) & 1);
  const bool whole = arcs == 0;
  uint32_t e = (whole ? kWhole : (arcs > 1 ? kArcs : kPlain)) << kKindBit;
  e |= (uint32_t)(cof_of(t, kCyc.v[t][w]) + 1) << kEdgeBit;
  // away from w in both directions (round the whole cycle: one direction,
  // the last triangle unpaired), each tet omits its vertex nearer to w
  auto put = [&](int i, int near) {
    const int q = kCyc.tet[t][i];
    e |= (uint32_t)code_omitting(q, kCyc.v[t][near]) << (kTetBit + 3 * kStar.qType[q]);
  };
  int steps = 0;
  for (int i = w; ((L >> ((i + 1) % n)) & 1) && steps < n - 1; i = (i + 1) % n, ++steps) put(i, i);
  if (!whole)
    for (int i = w; (L >> ((i + n - 1) % n)) & 1; i = (i + n - 1) % n) put((i + n - 1) % n, i);
  return e;
}

struct Entries {
  uint32_t e[kEntries];
};
constexpr Entries make_entries() {
  Entries r{};
  for (int t = 0; t < 7; ++t) {
    const int n = kCyc.n[t];
    for (uint32_t L = 0; L < (1u << n); ++L)
      for (int w = 0; w < (n == 6 ? 8 : 4); ++w) r.e[entry_base(t) + (w << n) + L] = edge_entry(t, L, w);
  }
  return r;
}

// c added to x where a < b (a == b): on the device as a multiply-add, which
// leaves the integer pipe, the busiest here, to the comparison (one: the
// number 1, which the compiler must not know)
template <uint32_t C>
DMS_HD void add_if_less(uint32_t& x, uint32_t a, uint32_t b, uint32_t one) {
#ifdef __CUDA_ARCH__
  asm("{\n .reg .pred p;\n setp.lt.u32 p, %1, %2;\n @p mad.lo.u32 %0, %3, %4, %0;\n}"
      : "+r"(x) : "r"(a), "r"(b), "r"(one), "n"(C));
#else
  if (a < b) x += one * C;
#endif
}
template <uint32_t C>
DMS_HD void add_if_equal(uint32_t& x, uint32_t a, uint32_t b, uint32_t one) {
#ifdef __CUDA_ARCH__
  asm("{\n .reg .pred p;\n setp.eq.u32 p, %1, %2;\n @p mad.lo.u32 %0, %3, %4, %0;\n}"
      : "+r"(x) : "r"(a), "r"(b), "r"(one), "n"(C));
#else
  if (a == b) x += one * C;
#endif
}

// Where the edge of type t at a vertex of order oa has its entry, from the
// orders o[s] of that vertex's slots 0..12 (0xFFFFFFFF outside the grid): 4 x
// (L + (w << n)), a byte offset behind entry_base(t).  Equal orders occur only
// outside the grid; an edge of the grid has a cycle vertex in the grid, so its
// w is one position, and what else the sums of positions reach (at most 15
// rows of 64 behind the last type's first row) stays inside the table.
template <int T>
DMS_HD uint32_t edge_offset(uint32_t oa, const uint32_t* o, uint32_t one) {
  constexpr int n = kCyc.n[T], v0 = kCyc.v[T][0];
  const uint32_t y = umin(oa, o[T]);
  uint32_t m = o[v0];
  static_for<1, n>([&](auto I) {
    constexpr int v = kCyc.v[T][decltype(I)::value];
    m = umin(m, o[v]);
  });
  uint32_t at = 0;
  static_for<0, n>([&](auto I) {
    constexpr int i = decltype(I)::value, v = kCyc.v[T][i];
    add_if_less<(4u << i)>(at, o[v], y, one);
    if constexpr (i > 0) add_if_equal<((uint32_t)i << (n + 2))>(at, o[v], m, one);
  });
  return at;
}

// ------------------------------------------------------- the correction --
// Tables indexed at run time.
struct Tables {
  uint32_t entry[kEntries];
  uint8_t cyc[14][8];         // the cycle of slot s ([6]: its length)
  uint8_t cycTet[14][8];      // its star tets
  uint8_t cycCode[14][8];     // the tet's code when it is paired with its edge to position i
                              // (low four bits) or to the next position (high four)
  uint8_t slotOfCode[14][8];  // edge code - 1 -> the paired triangle's other slot
  uint8_t cofOfSlots[14][16];  // the edge code for that slot, minus one
  uint8_t posOfSlots[14][16];  // that slot's position in the cycle
  uint8_t triOfSlots[14][16];  // star triangle on two slots
  // a tet's facets that hold x, numbered 1..3:
  uint8_t tetNext[24][4];     // the tet across
  uint8_t tetFacet[24][4];    // the facet, a star triangle
  uint8_t tetCode[24][4];     // the tet's code when paired with it ([0]: 0)
  uint8_t tetFacetNo[24][36];  // star triangle -> the facet's number
  uint8_t triTets[36][2];     // the two tets on a star triangle
  uint8_t tetAt[24];          // corner << 3 | type of the tet's record
  uint8_t edgeAt[16];         // corner << 3 | type of the edge's record
  uint8_t triAt[36];          // corner << 4 | type of the triangle's record
  uint16_t tetSlots[24];      // the tet's slots, as a mask
  // the arcs left when the one that holds position w is taken from L (several
  // arcs): one of up to three positions, or two of one each -- bits 0..2 the
  // first one's start, 3..4 its length, 5..7 the second one's position (7:
  // none); [L + 64 w] for cycles of 6, [512 + L + 16 w] for cycles of 4
  uint8_t arcs[512 + 64];
};
constexpr uint32_t further_arcs(int n, uint32_t L, int w) {
  const uint32_t none = 7u << 5;
  if (w >= n || !((L >> w) & 1)) return none;
  uint32_t keep = 1u << w;
  for (int k = 0; k < n; ++k)
    for (int i = 0; i < n; ++i)
      if (((L >> i) & 1) && (((keep >> ((i + 1) % n)) & 1) || ((keep >> ((i + n - 1) % n)) & 1)))
        keep |= 1u << i;
  const uint32_t rest = L & ~keep;
  uint32_t r = none;
  bool one = false;
  for (int i = 0; i < n; ++i) {
    if (!((rest >> i) & 1) || ((rest >> ((i + n - 1) % n)) & 1)) continue;  // not a start
    int len = 1;
    while (len < n && ((rest >> ((i + len) % n)) & 1)) ++len;
    if (!one) r = none | (uint32_t)i | (uint32_t)len << 3;
    else r = (r & 31u) | (uint32_t)i << 5;
    one = true;
  }
  return r;
}

constexpr Tables make_tables() {
  Tables t{};
  const Entries en = make_entries();
  for (int i = 0; i < kEntries; ++i) t.entry[i] = en.e[i];
  for (int s = 0; s < 14; ++s) {
    t.cyc[s][6] = (uint8_t)kCyc.n[s];
    for (int i = 0; i < kCyc.n[s]; ++i) {
      t.cyc[s][i] = (uint8_t)kCyc.v[s][i];
      const int q = kCyc.tet[s][i];
      t.cycTet[s][i] = (uint8_t)q;
      t.cycCode[s][i] = (uint8_t)(code_omitting(q, kCyc.v[s][(i + 1) % kCyc.n[s]]) |
                                  code_omitting(q, kCyc.v[s][i]) << 4);
      const int c = cof_of(s, kCyc.v[s][i]);
      t.slotOfCode[s][c] = (uint8_t)kCyc.v[s][i];
      t.cofOfSlots[s][kCyc.v[s][i]] = (uint8_t)c;
      t.posOfSlots[s][kCyc.v[s][i]] = (uint8_t)i;
    }
    t.edgeAt[s] = (uint8_t)(kStar.eCorner[s] << 3 | kStar.eType[s]);
  }
  for (uint32_t L = 0; L < 64; ++L)
    for (int w = 0; w < 8; ++w) t.arcs[L + 64 * w] = (uint8_t)further_arcs(6, L, w);
  for (uint32_t L = 0; L < 16; ++L)
    for (int w = 0; w < 4; ++w) t.arcs[512 + L + 16 * w] = (uint8_t)further_arcs(4, L, w);
  for (int q = 0; q < 24; ++q) {
    const int slots[3] = {kStar.tetA[q], kStar.tetB[q], kStar.tetC[q]};
    t.tetSlots[q] = (uint16_t)((1u << slots[0]) | (1u << slots[1]) | (1u << slots[2]));
    t.tetAt[q] = (uint8_t)(kStar.qCorner[q] << 3 | kStar.qType[q]);
    for (int w = 0; w < 3; ++w) {
      const int j = kStar.tetF[q][w];
      t.tetFacet[q][w + 1] = (uint8_t)j;
      t.tetCode[q][w + 1] = (uint8_t)kStar.facetCode[q][w];
      t.tetFacetNo[q][j] = (uint8_t)(w + 1);
      for (int p = 0; p < 24; ++p)
        if (p != q && ((kStar.triCof[j] >> p) & 1)) t.tetNext[q][w + 1] = (uint8_t)p;
    }
  }
  for (int j = 0; j < 36; ++j) {
    t.triOfSlots[kStar.triA[j]][kStar.triB[j]] = (uint8_t)j;
    t.triOfSlots[kStar.triB[j]][kStar.triA[j]] = (uint8_t)j;
    t.triAt[j] = (uint8_t)(kStar.tCorner[j] << 4 | kStar.tType[j]);
    int k = 0;
    for (int q = 0; q < 24; ++q)
      if ((kStar.triCof[j] >> q) & 1) t.triTets[j][k++] = (uint8_t)q;
  }
  return t;
}

// On the device the 32 lanes of a warp correct 32 vertices in step: every loop
// runs while any lane has work, so that the lanes stay together (a loop per
// lane, left to diverge, ran the lanes one after the other).
DMS_HD bool any_lane(bool p) {
#ifdef __CUDA_ARCH__
  return __any_sync(0xFFFFFFFFu, p);
#else
  return p;
#endif
}

// Corrects the lower star of x whose edges' rules have been applied.  A gives
// the orders o(s) of the slots, o(s, i) of position i of slot s's cycle, and
// the record codes of the simplices whose highest vertex is x: parents() is
// the slot that each slot's edge leads to, four bits each (15: unpaired),
// facets() the number of the facet that each star tet is paired with, two
// bits each (0: unpaired); set_edge(s, old, new) and set_tet(q, old, new)
// change a code, crit_tri(j) marks a triangle critical.
// on: the lane has a vertex.  lm = its lower slots (used only where whole is
// not empty in some lane); mins, arcs, whole = the slots whose edge is kEmpty
// / kArcs / kWhole.  Returns desc, the slot paired with x.  Both forests are
// kept in registers while they change; the codes that differ are written at
// the end.  Every loop is bounded (16 steps cover any path in a link of 14
// vertices, 24 any path of its triangles), also on inputs that are no order.
template <class A>
DMS_HD int correct_star(A& a, const Tables& tb, bool on, uint32_t lm, uint32_t mins, uint32_t arcs,
                        uint32_t whole) {
  if (!on) mins = arcs = whole = 0;
  // the lowest local minimum of the link is the lowest vertex of all
  int delta = 0;
  uint32_t od = 0xFFFFFFFFu;
  DMS_ROLLED
  for (uint32_t m = mins; any_lane(m != 0);) {
    if (m) {
      const int s = ffs32(m);
      const uint32_t os = a.o(s);
      if (os < od) {
        od = os;
        delta = s;
      }
      m &= m - 1;
    }
  }
  const bool trees = (mins & (mins - 1)) != 0;  // more than one
  uint64_t cycles = 0;  // edges that closed a cycle, (h << 4 | l) bytes, the highest lowest
  if (any_lane(arcs != 0)) {
    const uint64_t par0 = a.parents();
    uint64_t par = par0;
    auto up = [&](int s) -> int { return (int)(par >> (4 * s)) & 15; };
    // the edges to further arcs, (h << 4 | l) bytes in increasing key order
    // (the lowest byte first), at most 16
    uint64_t ev0 = 0, ev1 = 0;
    int nev = 0;
    DMS_ROLLED
    for (uint32_t left = arcs; any_lane(left != 0);) {
      // the lowest of the vertices with several arcs
      int h = 0;
      uint32_t oh = 0xFFFFFFFFu;
      const bool has = left != 0;
      DMS_ROLLED
      for (uint32_t m = left; any_lane(m != 0);) {
        if (m) {
          const int s = ffs32(m);
          const uint32_t os = a.o(s);
          if (os <= oh) {
            oh = os;
            h = s;
          }
          m &= m - 1;
        }
      }
      left &= ~(1u << h);
      // its arcs but that of its rule's vertex
      const int n = tb.cyc[h][6];
      uint32_t L = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
      for (int i = 0; i < 6; ++i) L |= (a.o(h, i) < oh ? 1u : 0u) << i;  // (position n on: none)
      const int w = tb.posOfSlots[h][up(h)];
      const uint32_t rest = has ? tb.arcs[n == 6 ? L + 64 * w : 512 + (L & 15u) + 16 * (w & 3)] : 224u;
      const int len = (int)(rest >> 3) & 3, p0 = (int)rest & 7;
      int at = p0;  // the first one's lowest position
      if (any_lane(len > 1)) {
        if (len > 1) {
          const int p1 = p0 + 1 < n ? p0 + 1 : 0, p2 = p1 + 1 < n ? p1 + 1 : 0;
          const uint32_t o0 = a.o(h, p0), o1 = a.o(h, p1), o2 = len > 2 ? a.o(h, p2) : 0xFFFFFFFFu;
          at = o1 < o0 ? (o2 < o1 ? p2 : p1) : (o2 < o0 ? p2 : p0);
          // its triangles, each with its edge farther from that position
          a.set_tet(tb.cycTet[h][p0], 0u, (tb.cycCode[h][p0] >> (at != p0 ? 0 : 4)) & 15u);
          if (len > 2) a.set_tet(tb.cycTet[h][p1], 0u, (tb.cycCode[h][p1] >> (at == p2 ? 0 : 4)) & 15u);
        }
      }
      int second = (int)(rest >> 5);
      if (len) {
        if (second != 7 && a.o(h, second) < a.o(h, at)) {
          const int t = at;
          at = second;
          second = t;
        }
        uint32_t e = (uint32_t)(h << 4 | tb.cyc[h][at]);
        int k = 1;
        if (second != 7) {
          e |= (uint32_t)(h << 4 | tb.cyc[h][second]) << 8;
          k = 2;
        }
        if (nev < 8) {
          ev0 |= (uint64_t)e << (8 * nev);
          if (nev == 7) ev1 = e >> 8;
        } else {
          ev1 |= (uint64_t)e << (8 * (nev - 8));
        }
        nev += k;
      }
    }
    DMS_ROLLED
    for (int k = 0; k < 16 && any_lane(k < nev); ++k) {
      const bool ev = k < nev;
      const uint32_t e = (uint32_t)ev0 & 255u;
      ev0 = ev0 >> 8 | ev1 << 56;
      ev1 >>= 8;
      const int h = (int)(e >> 4), l = (int)e & 15;
      // the roots of both ends (one tree: the same)
      int r0 = h, r1 = l;
      bool go = ev && trees;
      DMS_ROLLED
      for (int it = 0; it < 16 && any_lane(go); ++it) {
        if (go) {
          const int u0 = up(r0), u1 = up(r1);
          go = (u0 & u1) != 15;
          r0 = u0 != 15 ? u0 : r0;
          r1 = u1 != 15 ? u1 : r1;
        }
      }
      bool flip = ev && trees && r0 != r1;
      if (ev && !flip) {
        // closes a cycle; with one dual tree (no local maximum of the link)
        // it closes one there too and is critical
        if (whole) cycles = cycles << 8 | (uint64_t)e;
        else a.crit_tri(tb.triOfSlots[h][l]);
      }
      // the younger (higher) root's side hangs below the other end
      int cur = h, to = l;
      if (flip && a.o(r0) < a.o(r1)) {
        cur = l;
        to = h;
      }
      DMS_ROLLED
      for (int it = 0; it < 16 && any_lane(flip); ++it) {
        if (flip) {
          const int old = up(cur);
          par ^= (uint64_t)(old ^ to) << (4 * cur);
          to = cur;
          cur = old;
          flip = old != 15;
        }
      }
    }
    DMS_ROLLED
    for (uint64_t d = par ^ par0; any_lane(d != 0);) {
      if (d) {
        const int s = ffs64(d) >> 2;
        d &= ~(15ull << (4 * s));
        const int old = (int)(par0 >> (4 * s)) & 15;
        a.set_edge(s, old == 15 ? 0u : tb.cofOfSlots[s][old] + 1u, tb.cofOfSlots[s][up(s)] + 1u);
        mins &= ~(1u << s);  // (a local minimum joined to another tree is no root any more)
      }
    }
  }
  // the roots left over, but the lowest, are critical
  DMS_ROLLED
  for (uint32_t m = mins & ~(1u << delta); any_lane(m != 0);) {
    if (m) {
      a.set_edge(ffs32(m), 0u, 7u);
      m &= m - 1;
    }
  }
  if (!any_lane(whole != 0)) return delta;

  // dual trees: the edges that closed cycles, highest first
  const uint64_t fac0 = a.facets();
  uint64_t fac = fac0;
  uint32_t QL = 0;
  static_for<0, 24>([&](auto Q) {
    constexpr int q = decltype(Q)::value;
    constexpr uint32_t m = (1u << kStar.tetA[q]) | (1u << kStar.tetB[q]) | (1u << kStar.tetC[q]);
    if ((m & ~lm) == 0) QL |= 1u << q;
  });
  auto facet = [&](int q) -> int { return (int)(fac >> (2 * q)) & 3; };
  auto top_of = [&](int q) -> uint32_t {
    uint32_t t = 0;
    DMS_ROLLED
    for (uint32_t m = tb.tetSlots[q]; m; m &= m - 1) t = umax(t, a.o(ffs32(m)));
    return t;
  };
  // turns the path from q to its root round, q's facet becoming w
  auto reroot = [&](bool go, int q, int w) {
    DMS_ROLLED
    for (int it = 0; it < 24 && any_lane(go); ++it) {
      if (go) {
        const int old = facet(q);
        fac ^= (uint64_t)(old ^ w) << (2 * q);
        go = old != 0;
        const int j = tb.tetFacet[q][old];
        q = tb.tetNext[q][old];
        w = tb.tetFacetNo[q][j];
      }
    }
  };
  constexpr int R = 24;
  DMS_ROLLED
  for (; any_lane(cycles != 0); cycles >>= 8) {
    const bool ev = cycles != 0;
    const int h = (int)(cycles >> 4) & 15, l = (int)cycles & 15;
    const int j = ev ? tb.triOfSlots[h][l] : 0;
    const int q0 = tb.triTets[j][0], q1 = tb.triTets[j][1];
    // the unpaired triangles that the two sides lead to, or R
    int r0 = ev && ((QL >> q0) & 1) ? q0 : R, r1 = ev && ((QL >> q1) & 1) ? q1 : R;
    bool g0 = r0 != R, g1 = r1 != R;
    DMS_ROLLED
    for (int it = 0; it < 24 && any_lane(g0 || g1); ++it) {
      if (g0) {
        const int w = facet(r0), nx = tb.tetNext[r0][w];
        if (w) r0 = (QL >> nx) & 1 ? nx : R;
        g0 = w != 0 && r0 != R;
      }
      if (g1) {
        const int w = facet(r1), nx = tb.tetNext[r1][w];
        if (w) r1 = (QL >> nx) & 1 ? nx : R;
        g1 = w != 0 && r1 != R;
      }
    }
    if (ev && r0 == r1) a.crit_tri(j);
    const bool turn = ev && r0 != r1;
    bool first = r1 == R;  // the side that is turned round: the younger root's
    if (turn && r0 != R && r1 != R) first = top_of(r0) < top_of(r1);
    const int q = first ? q0 : q1;
    reroot(turn, q, tb.tetFacetNo[q][j]);
  }
  const bool sphere = lm == 0x3FFFu && whole != 0;
  int crit = R;
  if (any_lane(sphere)) {
    // the whole sphere: the triangle of largest key is the critical root, on
    // the highest vertex, its highest neighbour and the higher of the two
    // vertices next to both
    int h = 0;
    uint32_t oh = 0;
    DMS_ROLLED
    for (uint32_t m = sphere ? whole : 0u; any_lane(m != 0);) {
      if (m) {
        const int s = ffs32(m);
        const uint32_t os = a.o(s);
        if (os >= oh) {
          oh = os;
          h = s;
        }
        m &= m - 1;
      }
    }
    const int n = tb.cyc[h][6];
    int b = 0;
    uint32_t ob = a.o(h, 0);
    DMS_ROLLED
    for (int i = 1; i < 6; ++i) {
      const uint32_t oi = i < n ? a.o(h, i) : 0u;
      if (oi > ob) {
        ob = oi;
        b = i;
      }
    }
    const int up = b + 1 < n ? b + 1 : 0, dn = b ? b - 1 : n - 1;
    if (sphere) crit = tb.cycTet[h][a.o(h, up) > a.o(h, dn) ? b : dn];
    reroot(sphere, crit, 0);
  }
  DMS_ROLLED
  for (uint64_t d = fac ^ fac0; any_lane(d != 0);) {
    if (d) {
      const int q = ffs64(d) >> 1;
      d &= ~(3ull << (2 * q));
      a.set_tet(q, tb.tetCode[q][(int)(fac0 >> (2 * q)) & 3], tb.tetCode[q][facet(q)]);
    }
  }
  if (crit != R) a.set_tet(crit, 0u, 7u);
  return delta;
}

// ------------------------------------------------- one vertex by itself --
// The rule and the correction for one vertex, its records' words held in
// scratch: what the gradient kernel does per tile, for the CPU tests.
template <int NT>
struct Keys {
  uint64_t rec[8];
};

struct StarScratch {
  const uint32_t* od;
  uint64_t* rec;
  const Tables& tb;
  uint32_t o(int s) const { return od[s]; }
  uint32_t o(int s, int i) const { return i < tb.cyc[s][6] ? od[tb.cyc[s][i]] : 0xFFFFFFFFu; }
  uint64_t parents() const {
    uint64_t p = 0;
    for (int s = 0; s < 14; ++s) {
      const uint32_t c = (uint32_t)(rec[tb.edgeAt[s] >> 3] >> (3 * (tb.edgeAt[s] & 7))) & 7u;
      p |= (uint64_t)(c ? tb.slotOfCode[s][c - 1] : 15) << (4 * s);
    }
    return p;
  }
  uint64_t facets() const {
    uint64_t f = 0;
    for (int q = 0; q < 24; ++q) {
      const uint32_t c = (uint32_t)(rec[tb.tetAt[q] >> 3] >> (33 + 3 * (tb.tetAt[q] & 7))) & 7u;
      for (int w = 1; w < 4; ++w)
        if (c && c == tb.tetCode[q][w]) f |= (uint64_t)w << (2 * q);
    }
    return f;
  }
  void set_edge(int s, uint32_t old, uint32_t c) {
    rec[tb.edgeAt[s] >> 3] ^= (uint64_t)(old ^ c) << (3 * (tb.edgeAt[s] & 7));
  }
  void set_tet(int q, uint32_t old, uint32_t c) {
    rec[tb.tetAt[q] >> 3] ^= (uint64_t)(old ^ c) << (33 + 3 * (tb.tetAt[q] & 7));
  }
  void crit_tri(int j) { rec[tb.triAt[j] >> 4] |= 1ull << (21 + (tb.triAt[j] & 15)); }
};

// o[s] = order of neighbour s (0xFFFFFFFF outside the grid), lm = the slots
// below x.  Returns desc and fills acc[c], the record bits contributed to the
// anchor x - corner c.
template <int NT>
inline int process_lower_star(uint32_t lm, const uint32_t (&o)[14], const Tables& tb, Keys<NT>& keys,
                              int, uint64_t (&acc)[8]) {
  for (int c = 0; c < 8; ++c) keys.rec[c] = acc[c] = 0;
  if (!lm) return 15;
  uint32_t mins = 0, arcs = 0, whole = 0;
  StarScratch a{o, keys.rec, tb};
  for (int s = 0; s < 14; ++s) {
    if (!((lm >> s) & 1)) continue;
    const int n = kCyc.n[s], t = s % 7;
    uint32_t L = 0;
    int w = 0;
    for (int i = 0; i < n; ++i) {
      if (o[kCyc.v[s][i]] < o[s]) L |= 1u << i;
      if (o[kCyc.v[s][i]] < o[kCyc.v[s][w]]) w = i;
    }
    const uint32_t e = tb.entry[entry_base(t) + (w << n) + (int)L], kind = (e >> kKindBit) & 3u;
    mins |= (kind == kEmpty ? 1u : 0u) << s;
    arcs |= (kind == kArcs ? 1u : 0u) << s;
    whole |= (kind == kWhole ? 1u : 0u) << s;
    a.set_edge(s, 0, e >> kEdgeBit);
    for (int i = 0; i < n; ++i) {
      const int q = kCyc.tet[s][i];
      if (((L >> i) & 1) && ((L >> ((i + 1) % n)) & 1))
        a.set_tet(q, 0, (e >> (kTetBit + 3 * kStar.qType[q])) & 7u);
    }
  }
  const int d = correct_star(a, tb, true, lm, mins, arcs, whole);
  for (int c = 0; c < 8; ++c) acc[c] = keys.rec[c];
  return d;
}

}  // namespace lowerstar
}  // namespace dms
