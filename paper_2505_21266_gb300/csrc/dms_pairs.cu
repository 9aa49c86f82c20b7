// Extremum-saddle persistence pairs D0 and D2 (Sec. 2.5, Alg. 1; Sec. 4.1-4.2).
//
// 1. v-path tracing.  D0: from both vertices of a critical edge, follow desc[]
//    (vertex -> paired edge -> other vertex) to a minimum.  D2: from both
//    cofacets of a critical triangle follow the dual gradient (tet -> its
//    paired facet -> that facet's other cofacet) to a critical tetrahedron, or
//    to the virtual OUTSIDE node when the path leaves the grid.  The paths are
//    first resolved by bricks of the grid in shared memory (every cell learns
//    where its path leaves the brick, or its extremum), then each saddle hops
//    from brick to brick; few saddles on a large grid, and many on a thin one,
//    are followed cell by cell (follow_by_cells).  Triplets whose two ends
//    coincide are dropped.
// 2. Pairing rounds.  Alg. 1 visits the saddles in increasing order and, with
//    a union-find whose roots are the oldest extremum of each component,
//    pairs the saddle with the younger root when it joins two components.
//    Here every round takes, for each current component, its lightest live
//    saddle; a saddle that is the lightest of BOTH of its components is merged
//    at once.  Such a saddle meets exactly the components Alg. 1 would have
//    met at its turn (everything merged so far inside a component is lighter
//    than every live saddle touching it, and nothing lighter touches it), so
//    every merge -- and therefore every pair -- is the one Alg. 1 makes;
//    saddles whose ends already share a root are dropped, as in Alg. 1.
//    The lightest live saddle overall qualifies, so each round makes progress.
//    Per round: one phase finds both roots (path halving) and records, per
//    root, the lightest saddle with one 64-bit atomicMax of
//    (round << 44 | ~weight); the other merges the mutual ones and appends the
//    rest to the next live list.  A phase is a launch while very many saddles
//    are live, the later rounds are one cooperative launch.
// 3. Paired saddles are compacted in saddle-id order in one launch (a tile
//    looks back at the counts of the tiles before it) and written as dms_pair
//    records; birth/death values are copied from the field.
//
// Weights and ages are 44-bit integers ordered like the lexicographic keys
// of Sec. 2.1: (order of the top vertex) followed by the ranks, among the
// lower neighbours of that top vertex, of the other vertices.
#include <algorithm>
#include <atomic>
#include <cstdint>

#include "dms_bricks.cuh"
#include "dms_common.cuh"
#include "dms_radix.cuh"
#include "dms_rounds.cuh"
#include "dms_scan.cuh"

namespace dms {
namespace {

constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint64_t kMask44 = (1ull << 44) - 1;
constexpr int kCornerOfEdge[7] = {1, 2, 4, 3, 5, 6, 7};

// The type tables (corners of edge type k, triangle type k = (p, q), tet type
// k = chain (c1, c2)) as 4-bit fields of immediates: a lookup with an index
// that differs between lanes is a shift and a mask, not a serialised
// constant-memory access.
__device__ __forceinline__ int edge_corner(int k) { return (0x7653421u >> (4 * k)) & 15; }
__device__ __forceinline__ int tri_p(int k) { return (int)((0x653421424121ull >> (4 * k)) & 15); }
__device__ __forceinline__ int tri_q(int k) { return (int)((0x777777665533ull >> (4 * k)) & 15); }
__device__ __forceinline__ int tet_c1(int k) { return (0x442211u >> (4 * k)) & 15; }
__device__ __forceinline__ int tet_c2(int k) { return (0x656353u >> (4 * k)) & 15; }
// neighbour slots: +c for s < 7, -c for s >= 7, c = corner of edge type s % 7
__constant__ int cSlotCorner[14] = {1, 2, 4, 3, 5, 6, 7, 1, 2, 4, 3, 5, 6, 7};

// the union-find nodes (extrema), as separate arrays so that the parent
// array, which the root searches chase, stays small enough for L2: parent,
// the tag of the node's lightest live saddle in the current round, its age
// (a larger age is younger)
struct Nodes {
  uint32_t* parent;
  unsigned long long* best;
  uint64_t* age;
  // a node that never dies (OUTSIDE in D2, kNone in D0): it takes no tags --
  // a saddle to it merges by the downhill rule exactly when the mutual rule
  // would, and thousands of boundary saddles would otherwise contend for
  // its tag
  uint32_t immortal;
};

// one saddle of the pairing, in one 32-byte sector: its weight, its two
// end nodes, their roots in the current round and the extremum it kills
struct alignas(16) Sad {
  uint64_t w;
  uint32_t na, nb, ra, rb, res, pad;
};
struct Tri {
  Sad* s;
};

struct Dev {
  Grid g;
  int64_t slot_delta[14];
};

__device__ __forceinline__ int64_t corner_delta(const Grid& g, int c) {
  return (c & 1) + ((c >> 1) & 1) * g.nx + ((c >> 2) & 1) * g.sxy;
}
__device__ __forceinline__ void xyz(const Grid& g, int64_t v, int64_t& x, int64_t& y, int64_t& z) {
  // vertex offsets are below 2^32: 32-bit divisions are enough
  const uint32_t u = (uint32_t)v, sxy = (uint32_t)g.sxy, nx = (uint32_t)g.nx;
  const uint32_t zz = u / sxy, r = u - zz * sxy, yy = r / nx;
  z = zz;
  y = yy;
  x = r - yy * nx;
}
__device__ __forceinline__ void coords(const Grid& g, int64_t v, int& x, int& y, int& z) {
  int64_t x64, y64, z64;
  xyz(g, v, x64, y64, z64);
  x = (int)x64;
  y = (int)y64;
  z = (int)z64;
}
// is anchor + corner c inside the grid, for c in {0..7} with all of +c
__device__ __forceinline__ bool fits(const Grid& g, int64_t ax, int64_t ay, int64_t az, int c) {
  return ax >= 0 && ay >= 0 && az >= 0 && ax + (c & 1) < g.nx && ay + ((c >> 1) & 1) < g.ny &&
         az + ((c >> 2) & 1) < g.nz;
}

// rank of neighbour u among the lower neighbours of its top vertex t
__device__ __forceinline__ uint32_t local_rank(const Dev& D, const uint32_t* __restrict__ order,
                                               int64_t t, uint32_t ou) {
  int64_t x, y, z;
  xyz(D.g, t, x, y, z);
  uint32_t r = 0;
#pragma unroll
  for (int s = 0; s < 14; ++s) {
    int c = cSlotCorner[s];
    int sg = s < 7 ? 1 : -1;
    int64_t nx = x + sg * (c & 1), ny = y + sg * ((c >> 1) & 1), nz = z + sg * ((c >> 2) & 1);
    if (nx < 0 || ny < 0 || nz < 0 || nx >= D.g.nx || ny >= D.g.ny || nz >= D.g.nz) continue;
    r += __ldg(order + t + D.slot_delta[s]) < ou ? 1u : 0u;
  }
  return r;
}

// tet type of the chain 0 < c1 < c2 < 7 (c1 one corner bit, c2 two): the
// types are ordered by c1, then by whether the bit c2 adds is the larger of
// the two bits c1 leaves
__device__ __forceinline__ int tet_type(int c1, int c2) {
  return (c1 >> 1) * 2 + ((c2 ^ c1) > (7 ^ c2) ? 1 : 0);
}

__global__ void mark_ends(const int64_t* __restrict__ list, const int64_t* n_dev, int64_t n_host,
                          uint32_t node0, uint32_t* path) {
  const int64_t n = n_dev ? *n_dev : n_host;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    path[list[i]] = kEnd | (uint32_t)(i + node0);
}

// Appends of a whole CTA (256 threads) to two lists at once: one atomic per
// list per CTA and pass -- a counter that every warp of the grid hits
// serialises the appends of the first rounds, where almost every live
// saddle is appended to one list or the other.  Every thread of the CTA
// must call it.
struct CtaAppend {
  unsigned int off[2][8];
  unsigned int base[2];
};
__device__ __forceinline__ void cta_append2(CtaAppend& sh, bool w0, uint32_t* l0, unsigned int* c0,
                                            bool w1, uint32_t* l1, unsigned int* c1, uint32_t v) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned b0 = __ballot_sync(0xFFFFFFFFu, w0), b1 = __ballot_sync(0xFFFFFFFFu, w1);
  if (lane == 0) {
    sh.off[0][warp] = __popc(b0);
    sh.off[1][warp] = __popc(b1);
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    const int k = threadIdx.x;
    unsigned int t = 0;
    for (int w = 0; w < 8; ++w) {
      const unsigned int x = sh.off[k][w];
      sh.off[k][w] = t;
      t += x;
    }
    sh.base[k] = t ? atomicAdd(k ? c1 : c0, t) : 0u;
  }
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
  if (w0) l0[sh.base[0] + sh.off[0][warp] + __popc(b0 & lt)] = v;
  if (w1) l1[sh.base[1] + sh.off[1][warp] + __popc(b1 & lt)] = v;
  __syncthreads();
}


// The two cofacets of critical triangle id (anchor a, type k) in field g
// (anchor coordinates ax, ay, az); -1 where a cofacet leaves the grid.
__device__ __forceinline__ void tri_cofacets(const Grid& g, int64_t a, int k, int64_t ax,
                                             int64_t ay, int64_t az, int64_t cof[2]) {
  const int p = tri_p(k), q = tri_q(k);
  cof[0] = cof[1] = -1;
  if (q == 7) {
    const int e = (__popc(p) == 1) ? (7 ^ p) : p;
    const int e1 = e & -e, e2 = e ^ e1;
    if (fits(g, ax, ay, az, 7)) {
      if (__popc(p) == 1) {
        cof[0] = a * 6 + tet_type(p, p | e1);
        cof[1] = a * 6 + tet_type(p, p | e2);
      } else {
        cof[0] = a * 6 + tet_type(e1, p);
        cof[1] = a * 6 + tet_type(e2, p);
      }
    }
  } else {
    if (fits(g, ax, ay, az, 7)) cof[0] = a * 6 + tet_type(p, q);
    const int e = 7 ^ q;
    const int64_t bx = ax - (e & 1), by = ay - ((e >> 1) & 1), bz = az - ((e >> 2) & 1);
    if (fits(g, bx, by, bz, 7)) cof[1] = (a - corner_delta(g, e)) * 6 + tet_type(e, e | p);
  }
}

// a batch: the field that holds an anchor or a brick, by binary search
struct ManyFields {
  const dms_field_desc* fd;
  int n;
  const int64_t* brick0;  // nfields + 1: the fields' first bricks (see brick_table)
  __device__ __forceinline__ void set(const dms_field_desc& d, Grid& out, int64_t& off) const {
    out.nx = d.nx;
    out.ny = d.ny;
    out.nz = d.nz;
    out.sxy = (int64_t)d.nx * d.ny;
    out.n = out.sxy * d.nz;
    off = d.offset;
  }
  __device__ __forceinline__ void get(int64_t anchor, Grid& out, int64_t& off) const {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (fd[mid].offset <= anchor) lo = mid;
      else hi = mid;
    }
    set(fd[lo], out, off);
  }
  __device__ __forceinline__ void brick(int64_t id, int lx, int ly, int lz, Grid& out, int64_t& off,
                                        int& bx, int& by, int& bz) const {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(brick0 + mid) <= id) lo = mid;
      else hi = mid;
    }
    set(fd[lo], out, off);
    OneField{out}.brick(id - __ldg(brick0 + lo), lx, ly, lz, out, off, bx, by, bz);
    off = fd[lo].offset;
  }
};

__device__ __forceinline__ int64_t slot_delta_g(const Grid& g, int s) {
  const int c = (0x7653421 >> (4 * (s < 7 ? s : s - 7))) & 15;
  const int64_t d = (c & 1) + ((c >> 1) & 1) * g.nx + ((c >> 2) & 1) * g.sxy;
  return s < 7 ? d : -d;
}

// One CTA per brick: the words of all its cells, by pointer doubling.  A word
// is always a cell further along the path, so no barrier is needed between
// passes: every thread goes on until its own words are final.  (A path that
// loops, of bad data, is left as kLoop after as many passes as the brick has
// cells.)
constexpr int kBrickThreads = 256;
template <class P>
__global__ void __launch_bounds__(kBrickThreads) resolve_paths(const P p, uint32_t* path) {
  constexpr int VERTS = 1 << (P::LX + P::LY + P::LZ), CELLS = VERTS * P::K;
  static_assert(CELLS <= 8192, "a cell of a brick has 13 bits");
  __shared__ uint32_t s[CELLS];
  volatile uint32_t* const vs = s;
  Grid g;
  int64_t off;
  int bx, by, bz;
  p.fields.brick(blockIdx.x, P::LX, P::LY, P::LZ, g, off, bx, by, bz);
  const int x0 = bx << P::LX, y0 = by << P::LY, z0 = bz << P::LZ;
  const int wx = min((int64_t)1 << P::LX, g.nx - x0), wy = min((int64_t)1 << P::LY, g.ny - y0);
  const int wz = min((int64_t)1 << P::LZ, g.nz - z0);
  // a step from this brick may leave the grid (or reach its last vertices,
  // which anchor no tets)
  const bool border = bx == 0 || by == 0 || bz == 0 || x0 + (1 << P::LX) >= g.nx - 1 ||
                      y0 + (1 << P::LY) >= g.ny - 1 || z0 + (1 << P::LZ) >= g.nz - 1;
  const int64_t first = off + x0 + g.nx * y0 + g.sxy * z0;
  // a thread's words stay in registers, too
  constexpr int VPT = VERTS / kBrickThreads;
  uint32_t w[VPT][P::K];
#pragma unroll
  for (int j = 0; j < VPT; ++j) {
    const int lv = j * kBrickThreads + threadIdx.x;
    const int lx = lv & ((1 << P::LX) - 1), ly = (lv >> P::LX) & ((1 << P::LY) - 1), lz = lv >> (P::LX + P::LY);
#pragma unroll
    for (int k = 0; k < P::K; ++k) w[j][k] = kNoMark;
    if (lx < wx && ly < wy && lz < wz)
      p.cells(g, path, first + lx + g.nx * ly + g.sxy * lz, lv, x0, y0, z0, border, w[j]);
#pragma unroll
    for (int k = 0; k < P::K; ++k) vs[lv * P::K + k] = w[j][k];
  }
  __syncthreads();
  bool again = true;
  for (int pass = 0; again && pass < CELLS; ++pass) {
    again = false;
#pragma unroll
    for (int j = 0; j < VPT; ++j)
#pragma unroll
      for (int k = 0; k < P::K; ++k) {
        if (w[j][k] & (kEnd | kFinal)) continue;
        w[j][k] = vs[w[j][k]];
        vs[(j * kBrickThreads + threadIdx.x) * P::K + k] = w[j][k];
        again = true;
      }
  }
  if (again) {  // bad data: a path that loops
#pragma unroll
    for (int j = 0; j < VPT; ++j)
#pragma unroll
      for (int k = 0; k < P::K; ++k)
        if (!(w[j][k] & (kEnd | kFinal))) vs[(j * kBrickThreads + threadIdx.x) * P::K + k] = kLoop;
  }
  __syncthreads();
  // rows of vertices, whose cells are consecutive here and in memory, to warps
  constexpr int ROW = P::K << P::LX, ROWS = VERTS >> P::LX;
  for (int row = threadIdx.x >> 5; row < ROWS; row += kBrickThreads / 32) {
    const int ly = row & ((1 << P::LY) - 1), lz = row >> P::LY;
    if (ly >= wy || lz >= wz) continue;
    uint32_t* out = path + (first + g.nx * ly + g.sxy * lz) * P::K;
#pragma unroll
    for (int c = threadIdx.x & 31; c < ROW; c += 32) {
      const uint32_t w = s[row * ROW + c];
      if (c < wx * P::K) out[c] = w & kEnd ? w : w & ~kFinal;
    }
  }
}

// the node at a path's end, from its word
__device__ __forceinline__ uint32_t walk_end(uint32_t w, int32_t* dstatus) {
  if (w < kLoop) return w & ~kEnd;
  set_status(dstatus, w == kLoop ? DMS_ERR_TIMEOUT : DMS_ERR_ARG);  // bad data
  return 0;
}
// the saddle's record with its weight and ends, live where they differ.  With
// tag set it also does the first round's search of the pairing rounds (every
// node is still its own root): both ends are the roots and are tagged with the
// saddle, so that the rounds start at their merge step.
__device__ __forceinline__ bool store_saddle(Tri T, int64_t i, uint64_t w, uint32_t n0, uint32_t n1,
                                             bool tag, const Nodes& nd) {
  Sad sd;
  sd.w = w;
  sd.na = sd.ra = n0;
  sd.nb = sd.rb = n1;
  sd.res = kNone;
  sd.pad = 0;
  T.s[i] = sd;
  if (n0 == n1) return false;
  if (tag) {
    const unsigned long long tv = (1ull << 44) | (kMask44 - w);
    if (n0 != nd.immortal) atomicMax(nd.best + n0, tv);
    if (n1 != nd.immortal) atomicMax(nd.best + n1, tv);
  }
  return true;
}

// ranks of two neighbours u1, u2 (orders o1, o2) of vertex t = (x, y, z) of a
// field among the neighbours of t below
__device__ __forceinline__ void star_ranks(const Grid& g, const uint32_t* __restrict__ order, int64_t t,
                                           int x, int y, int z, uint32_t o1, uint32_t o2,
                                           uint32_t& r1, uint32_t& r2) {
  const int mx = (int)g.nx, my = (int)g.ny, mz = (int)g.nz;
  r1 = r2 = 0;
#pragma unroll
  for (int s = 0; s < 14; ++s) {
    const int c = (0x7653421 >> (4 * (s < 7 ? s : s - 7))) & 15;
    const int sg = s < 7 ? 1 : -1;
    const int nx = x + sg * (c & 1), ny = y + sg * ((c >> 1) & 1), nz = z + sg * ((c >> 2) & 1);
    if ((uint32_t)nx >= (uint32_t)mx || (uint32_t)ny >= (uint32_t)my || (uint32_t)nz >= (uint32_t)mz) continue;
    const uint32_t on = __ldg(order + t + slot_delta_g(g, s));
    r1 += on < o1 ? 1u : 0u;
    r2 += on < o2 ? 1u : 0u;
  }
}

// Paths cell by cell (see follow_by_cells): the words of the landmarks
// free, then one walk per thread
template <class P>
__global__ void clear_landmarks(int64_t n, uint32_t* path) {
  constexpr int WORDS = kGroup * P::K;  // of a run, consecutive
  const int64_t words = (n + kRun - 1) / kRun * WORDS;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < words;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t / WORDS, c = (r * kRun + landmarks_of(r)) * P::K + (t - r * WORDS);
    if (c < n * P::K) path[c] = kNoMark;
  }
}
template <class P, class S>
__global__ void __launch_bounds__(256, 8) follow_cells(const P paths, const S starts, int64_t nwalk,
                                                       uint32_t* path, uint32_t* results) {
  const Grid g = paths.fields.g;
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j < nwalk) results[j] = follow(paths, g, path, starts.at(g, j), (uint32_t)j);
}
// walk j's first cell: an end of critical edge j / 2, a cofacet of critical
// triangle j / 2
struct EdgeEnds {
  const int64_t* crit1;
  __device__ __forceinline__ Cell at(const Grid& g, int64_t j) const {
    const int64_t id = __ldg(crit1 + (j >> 1)), a = id / 7;
    const int c = j & 1 ? edge_corner((int)(id - a * 7)) : 0;
    int x, y, z;
    coords(g, a, x, y, z);
    return Cell{0, x + (c & 1), y + ((c >> 1) & 1), z + ((c >> 2) & 1), 0};
  }
};
struct TriCofacets {
  const int64_t* crit2;
  __device__ __forceinline__ Cell at(const Grid& g, int64_t j) const {
    const int64_t id = __ldg(crit2 + (j >> 1)), a = id / 12;
    int x, y, z;
    int64_t cof[2];
    coords(g, a, x, y, z);
    tri_cofacets(g, a, (int)(id - a * 12), x, y, z, cof);
    const int64_t t = j & 1 ? cof[1] : cof[0];
    if (t < 0) return Cell{kEnd, 0, 0, 0, 0};  // OUTSIDE
    const int64_t v = t / 6;
    coords(g, v, x, y, z);
    return Cell{0, x, y, z, (int)(t - v * 6)};
  }
};

// Where a saddle's two ends come from:
//   kBricks  walks over the words of the resolved bricks;
//   kCells   the results of follow_cells; saddles with a long path go to the
//            list far[0..*far_n);
//   kFar     as kBricks, the saddles of that list.
enum Follow { kBricks, kCells, kFar };

// D0: each critical edge's weight (its lexicographic key), its two descending
// paths.  (Bound by random reads of orders and path words: 32 registers for 64
// warps an SM; the D0/D2 stage of 1024^3 takes 80.3 ms with 54, 76.6 with 32.)
template <Follow HOW, class P>
__global__ void __launch_bounds__(256, 8) link_d0(
    const P paths, const uint32_t* __restrict__ order, const int64_t* __restrict__ crit1,
    const int64_t* n_dev, int64_t n_host, const uint32_t* __restrict__ path, Tri T, uint32_t* live,
    unsigned int* live_n, uint32_t* results, uint32_t* far, unsigned int* far_n, int32_t* dstatus,
    bool tag, Nodes nd) {
  __shared__ CtaAppend sh;
  const int64_t ne = n_dev ? *n_dev : n_host;
  // CTA-uniform passes: every thread reaches the appends
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < ne;
       base += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = base + threadIdx.x;
    bool keep = false, longer = false;
    if (i < ne) {
      if constexpr (HOW == kFar) i = far[i];
      const int64_t id = crit1[i], a = id / 7;
      const int c = edge_corner((int)(id - a * 7));
      Grid g;
      int64_t off;
      paths.fields.get(a, g, off);
      int x, y, z;
      coords(g, a - off, x, y, z);
      const int cx = c & 1, cy = (c >> 1) & 1, cz = (c >> 2) & 1;
      const int64_t b = a + corner_delta(g, c);
      Walk wa, wb;
      if constexpr (HOW == kCells) {
        wa.w = end_of(results, 2 * i);
        wb.w = end_of(results, 2 * i + 1);
        longer = !(wa.w & wb.w & kEnd);
      } else {
        wa = walk_from<P>(path, g, a, x, y, z, 0);
        wb = walk_from<P>(path, g, b, x + cx, y + cy, z + cz, 0);
      }
      const uint32_t oa = __ldg(order + a), ob = __ldg(order + b);
      const bool up = ob > oa;
      uint32_t r, r2;
      star_ranks(g, order, up ? b : a, up ? x + cx : x, up ? y + cy : y, up ? z + cz : z, min(oa, ob),
                 min(oa, ob), r, r2);
      if constexpr (HOW != kCells) walk_both<P>(path, g, off, wa, wb);
      if (!longer)
        keep = store_saddle(T, i, ((uint64_t)(oa > ob ? oa : ob) << 4) | r, walk_end(wa.w, dstatus),
                            walk_end(wb.w, dstatus), tag, nd);
    }
    if constexpr (HOW == kCells) cta_append2(sh, keep, live, live_n, longer, far, far_n, (uint32_t)i);
    else cta_append2(sh, keep, live, live_n, false, live, live_n, (uint32_t)i);
  }
}

// D2: each critical triangle's weight (decreasing triangle key), the two dual
// paths from its cofacets
template <Follow HOW, class P>
__global__ void __launch_bounds__(256, 8) link_d2(
    const P paths, const uint32_t* __restrict__ order, const int64_t* __restrict__ crit2,
    const int64_t* n_dev, int64_t n_host, const uint32_t* __restrict__ path, Tri T, uint32_t* live,
    unsigned int* live_n, uint32_t* results, uint32_t* far, unsigned int* far_n, int32_t* dstatus,
    bool tag, Nodes nd) {
  __shared__ CtaAppend sh;
  const int64_t nt = n_dev ? *n_dev : n_host;
  // CTA-uniform passes: every thread reaches the appends
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < nt;
       base += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = base + threadIdx.x;
    bool keep = false, longer = false;
    if (i < nt) {
      if constexpr (HOW == kFar) i = far[i];
      const int64_t id = crit2[i], a = id / 12;
      const int k = (int)(id - a * 12);
      Grid g;
      int64_t off;
      paths.fields.get(a, g, off);
      int x, y, z;
      coords(g, a - off, x, y, z);
      Walk wk[2];
      if constexpr (HOW == kCells) {
        wk[0].w = end_of(results, 2 * i);
        wk[1].w = end_of(results, 2 * i + 1);
        longer = !(wk[0].w & wk[1].w & kEnd);
      } else {
        int64_t cof[2];
        tri_cofacets(g, a, k, x, y, z, cof);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (cof[j] < 0) {
            wk[j] = Walk{kEnd, 0, 0, 0};  // no cofacet on that side: OUTSIDE
          } else {
            const int64_t v = cof[j] / 6;
            int vx, vy, vz;
            coords(g, v - off, vx, vy, vz);
            wk[j] = walk_from<P>(path, g, v, vx, vy, vz, (int)(cof[j] - v * 6));
          }
        }
      }
      // the key: the order of the highest vertex, the ranks of the others
      // among its neighbours
      const int c[3] = {0, tri_p(k), tri_q(k)};
      uint32_t o[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) o[j] = __ldg(order + a + corner_delta(g, c[j]));
      int it = 0;
      if (o[1] > o[it]) it = 1;
      if (o[2] > o[it]) it = 2;
      uint32_t om = 0, ol = 0xFFFFFFFFu;
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (j != it) {
          om = max(om, o[j]);
          ol = min(ol, o[j]);
        }
      const int ct = it == 0 ? 0 : (it == 1 ? c[1] : c[2]);
      uint32_t rm, rl;
      star_ranks(g, order, a + corner_delta(g, ct), x + (ct & 1), y + ((ct >> 1) & 1),
                 z + ((ct >> 2) & 1), om, ol, rm, rl);
      const uint64_t key = ((uint64_t)max(o[0], max(o[1], o[2])) << 8) | (rm << 4) | rl;
      if constexpr (HOW != kCells) walk_both<P>(path, g, off, wk[0], wk[1]);
      if (!longer)
        keep = store_saddle(T, i, kMask44 - key, walk_end(wk[0].w, dstatus), walk_end(wk[1].w, dstatus),
                            tag, nd);
    }
    if constexpr (HOW == kCells) cta_append2(sh, keep, live, live_n, longer, far, far_n, (uint32_t)i);
    else cta_append2(sh, keep, live, live_n, false, live, live_n, (uint32_t)i);
  }
}

__global__ void init_nodes_d0(const uint32_t* __restrict__ order, const int64_t* __restrict__ crit0,
                              int64_t nmin, Nodes nd) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nmin) return;
  nd.parent[i] = (uint32_t)i;
  nd.best[i] = 0ull;
  nd.age[i] = __ldg(order + crit0[i]);
}

__global__ void init_nodes_d2(Dev D, const uint32_t* __restrict__ order,
                              const int64_t* __restrict__ crit3, int64_t nmax, Nodes nd) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i > nmax) return;
  nd.parent[i] = (uint32_t)i;
  nd.best[i] = 0ull;
  if (i == 0) {
    nd.age[0] = 0;  // OUTSIDE is older than every maximum
    return;
  }
  int64_t id = crit3[i - 1];
  int64_t a = id / 6;
  int k = (int)(id - a * 6);
  int cs[4] = {0, tet_c1(k), tet_c2(k), 7};
  int64_t v[4];
  uint32_t o[4];
  int it = 0;
  for (int j = 0; j < 4; ++j) {
    v[j] = a + corner_delta(D.g, cs[j]);
    o[j] = __ldg(order + v[j]);
    if (o[j] > o[it]) it = j;
  }
  uint32_t r[3];
  int n = 0;
  for (int j = 0; j < 4; ++j)
    if (j != it) r[n++] = local_rank(D, order, v[it], o[j]);
  // sort the three ranks decreasingly
  uint32_t h = max(r[0], max(r[1], r[2])), l = min(r[0], min(r[1], r[2]));
  uint32_t m = r[0] + r[1] + r[2] - h - l;
  uint64_t key = ((uint64_t)o[it] << 12) | (h << 8) | (m << 4) | l;
  nd.age[i] = (kMask44 - key) + 1;  // a higher maximum is older
}

__device__ __forceinline__ uint32_t find_root(Nodes nd, uint32_t x) {
  uint32_t p = nd.parent[x];
  while (p != x) {
    uint32_t gp = nd.parent[p];
    if (gp != p) nd.parent[x] = gp;  // path halving: only ever points further up
    x = gp;
    p = nd.parent[x];
  }
  return x;
}

// ---------------------------------------------------------------------------
// The pairing rounds.
//
// Merge rules of the exact rounds (see the header comment):
//  * mutual: the saddle is the lightest live saddle of both components -> the
//    younger root dies;
//  * downhill: the saddle is the lightest live saddle of component a and the
//    other component b is older -> a's root dies.  At the saddle's turn in
//    Alg. 1 a's component is exactly a (nothing lighter touches it, and every
//    merge that built a used a lighter saddle), while b's side already holds
//    b's root, which is older than a's, so a's root is the younger one.
// A root dies through its own lightest saddle only, so it dies at most once
// per round, and the links never form a cycle (each points to an older root).
//
// The minimum spanning forest first (Borůvka), then the pairing on its edges:
// Alg. 1 pairs nothing at a saddle whose ends are already joined by lighter
// saddles, and such a saddle changes no component: these are exactly the
// saddles outside the minimum spanning forest of the extremum graph
// (weights are distinct), so the pairing over the forest's edges alone is
// the pairing over all saddles.  Borůvka rounds find the forest fast: every
// component joins its neighbour across its lightest live saddle (that
// saddle is a forest edge by the cut property), with no regard to ages, so
// components at least halve per round and the saddles inside a component
// drop out as loops.  The exact rounds then run on the forest's edges only.
// ---------------------------------------------------------------------------

// both roots of a live saddle, and the saddle as the lightest of each so far
__device__ __forceinline__ void find_saddle(const Tri& T, const Nodes& nd, uint32_t i,
                                            unsigned int round) {
  // roots only ever gain parents: search from last round's roots
  const uint32_t a = find_root(nd, round == 1 ? T.s[i].na : T.s[i].ra);
  const uint32_t b = find_root(nd, round == 1 ? T.s[i].nb : T.s[i].rb);
  T.s[i].ra = a;
  T.s[i].rb = b;
  if (a == b) return;
  const unsigned long long tv = ((unsigned long long)round << 44) | (kMask44 - T.s[i].w);
  if (a != nd.immortal) atomicMax(nd.best + a, tv);
  if (b != nd.immortal) atomicMax(nd.best + b, tv);
}

// whether a live saddle is the lightest of its roots (la, lb); false where
// they are one (inside a component: no forest edge, no pair).  ONE: within one
// launch, the tags are read from L2, where the atomics put them
template <bool ONE>
__device__ __forceinline__ bool lightest(const Tri& T, const Nodes& nd, uint32_t i, unsigned int round,
                                         uint32_t& a, uint32_t& b, bool& la, bool& lb) {
  a = T.s[i].ra;
  b = T.s[i].rb;
  if (a == b) return false;
  const unsigned long long tv = ((unsigned long long)round << 44) | (kMask44 - T.s[i].w);
  la = a != nd.immortal && (ONE ? __ldcg(nd.best + a) : nd.best[a]) == tv;
  lb = b != nd.immortal && (ONE ? __ldcg(nd.best + b) : nd.best[b]) == tv;
  return true;
}

// Borůvka: the saddle is a forest edge (tree), stays live (wait), or neither
template <bool ONE>
__device__ __forceinline__ void hook_saddle(const Tri& T, const Nodes& nd, uint32_t i,
                                            unsigned int round, bool& wait, bool& tree) {
  uint32_t a, b;
  bool la, lb;
  if (!lightest<ONE>(T, nd, i, round, a, b, la, lb)) return;
  tree = la || lb;
  wait = !tree;
  // each component hooks under the other end of its own lightest saddle; two
  // components that chose the same saddle hook one way only
  if (la && lb) nd.parent[min(a, b)] = max(a, b);
  else if (la) nd.parent[a] = b;
  else if (lb) nd.parent[b] = a;
}

// exact round: the saddle kills a root, stays live (wait), or neither
template <bool ONE>
__device__ __forceinline__ void merge_saddle(const Tri& T, const Nodes& nd, uint32_t i,
                                             unsigned int round, bool& wait) {
  uint32_t a, b;
  bool la, lb;
  if (!lightest<ONE>(T, nd, i, round, a, b, la, lb)) return;
  uint32_t young = kNone, old = kNone;
  if (la || lb) {
    const uint64_t ga = nd.age[a], gb = nd.age[b];
    if (la && (lb || ga > gb)) {
      young = ga > gb ? a : b;
      old = ga > gb ? b : a;
    } else if (lb && gb > ga) {
      young = b;
      old = a;
    }
  }
  wait = young == kNone;  // the lightest of neither side, or uphill: wait
  if (!wait) {
    nd.parent[young] = old;
    T.s[i].res = young;
  }
}

// ---- one launch per phase: rounds of many saddles
__global__ void round_find(const uint32_t* __restrict__ live, const unsigned int* __restrict__ live_n,
                           Tri T, Nodes nd, unsigned int round) {
  const unsigned int n = *live_n;
  for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    find_saddle(T, nd, live[j], round);
}

__global__ void __launch_bounds__(256) round_merge(const uint32_t* __restrict__ live,
                                                   const unsigned int* __restrict__ live_n, Tri T,
                                                   Nodes nd, unsigned int round, uint32_t* next,
                                                   unsigned int* next_n) {
  __shared__ CtaAppend sh;
  const unsigned int n = *live_n;
  // CTA-uniform passes: every thread reaches the appends
  for (unsigned int base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
    const unsigned int j = base + threadIdx.x;
    bool wait = false;
    const uint32_t i = j < n ? live[j] : 0;
    if (j < n) merge_saddle<false>(T, nd, i, round, wait);
    cta_append2(sh, wait, next, next_n, false, next, next_n, i);
  }
}

__global__ void __launch_bounds__(256) boruvka_hook(const uint32_t* __restrict__ live,
                                                    const unsigned int* __restrict__ live_n, Tri T,
                                                    Nodes nd, unsigned int round, uint32_t* next,
                                                    unsigned int* next_n, uint32_t* forest,
                                                    unsigned int* forest_n) {
  __shared__ CtaAppend sh;
  const unsigned int n = *live_n;
  // CTA-uniform passes: every thread reaches the appends
  for (unsigned int base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
    const unsigned int j = base + threadIdx.x;
    bool wait = false, tree = false;
    const uint32_t i = j < n ? live[j] : 0;
    if (j < n) hook_saddle<false>(T, nd, i, round, wait, tree);
    cta_append2(sh, wait, next, next_n, tree, forest, forest_n, i);
  }
}

// node arrays back to singletons: *n_dev + n nodes (n_dev may be null)
__global__ void reset_nodes(Nodes nd, const int64_t* __restrict__ n_dev, int64_t n) {
  if (n_dev) n += *n_dev;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    nd.parent[i] = (uint32_t)i;
    nd.best[i] = 0ull;
  }
}

// ---- all rounds in one launch: fewer saddles
// A cooperative grid (all its CTAs resident) takes its counts from device
// memory and meets at a barrier after each phase, so that no round costs a
// launch or a read of a count on the host; when few saddles are live, CTA 0
// goes on alone.  A round cost 25-30 us with one launch per phase and a
// synchronising read, 4 us with the grid barrier, 3 us in the lone CTA: the
// D0/D2 stage of 24^3 and 64^3 mixtures 733 -> 446 and 1119 -> 765 us, of 2 M
// vertices of noise 2.5 -> 1.4 ms, of a 1501 x 999 image 3.8 -> 1.1 ms (its
// last 4096 saddles used to go to the one-thread finish).  Many saddles hide
// the launches, and the grid's static share per CTA costs more: with all
// rounds in here the stage took 92.4 instead of 89.4 ms on the 1024^3 mixture
// (117 M saddles) and 31.4 instead of 30.5 ms on 512^3 quantised noise; the
// line lies where both ways cost the same (512 K to 10 M: within 1 %).
constexpr int kRoundThreads = 512;
constexpr int64_t kOneLaunch = (int64_t)3 << 20;  // saddles up to which the rounds are one launch
constexpr unsigned int kMaxExactRounds = 256;  // then the sorted finish, whatever is left
constexpr unsigned int kMaxForestRounds = 64;  // components at least halve per round
constexpr uint32_t kBarrierPolls = 1u << 23;

struct Rounds {
  Tri T;
  Nodes nd;
  uint32_t *cur, *nxt;   // the live saddles, room for the next round's
  const unsigned int* n;  // their count
  unsigned int round;     // the first round's number
  // Borůvka rounds append the forest's saddles to `forest` (null: exact
  // rounds); then, unless forest_only, the exact rounds on them follow
  uint32_t* forest;
  bool forest_only;
  bool first_found;       // the first round's search is done (link_d0, link_d2)
  unsigned int* ctr;
  const int64_t* n_dev;   // node count: *n_dev + nnode, or nnode alone
  int64_t nnode;
  uint32_t* left;         // the saddles that the exact rounds leave live end here
};

// as cta_append2, for kRoundThreads
struct RoundAppend {
  unsigned int off[2][kRoundThreads / 32];
  unsigned int base[2];
};
__device__ __forceinline__ void round_append2(RoundAppend& sh, bool w0, uint32_t* l0, unsigned int* c0,
                                              bool w1, uint32_t* l1, unsigned int* c1, uint32_t v) {
  constexpr int NW = kRoundThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned b0 = __ballot_sync(0xFFFFFFFFu, w0), b1 = __ballot_sync(0xFFFFFFFFu, w1);
  if (lane == 0) {
    sh.off[0][warp] = __popc(b0);
    sh.off[1][warp] = __popc(b1);
  }
  __syncthreads();
  if (warp < 2) {
    const unsigned int x = lane < NW ? sh.off[warp][lane] : 0u;
    unsigned int t = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, t, o);
      if (lane >= o) t += y;
    }
    if (lane < NW) sh.off[warp][lane] = t - x;
    if (lane == 31) sh.base[warp] = t ? atomicAdd(warp ? c1 : c0, t) : 0u;
  }
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
  if (w0) l0[sh.base[0] + sh.off[0][warp] + __popc(b0 & lt)] = v;
  if (w1) l1[sh.base[1] + sh.off[1][warp] + __popc(b1 & lt)] = v;
  __syncthreads();
}

// all CTAs of the grid (CTA 0 alone once solo); false when the others did not
// arrive within kBarrierPolls polls or gave up themselves
__device__ __forceinline__ bool round_sync(unsigned int* ctr, unsigned int& epoch, bool solo) {
  __syncthreads();
  if (solo) return true;
  int ok = 1;
  ++epoch;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr + kCtrBarrier, 1u);
    volatile unsigned int* bar = ctr + kCtrBarrier;
    volatile unsigned int* stop = ctr + kCtrAbort;
    const unsigned int want = epoch * gridDim.x;
    uint32_t it = 0;
    while ((int)(*bar - want) < 0) {
      if (++it > kBarrierPolls || *stop) {
        *stop = 1;
        ok = 0;
        break;
      }
    }
    __threadfence();
  }
  return __syncthreads_and(ok) != 0;
}

// An exact round that removes under 1/64 of the live saddles (a chain of
// components merging one saddle per round, say), or the round limit, ends the
// rounds: what is left (ctr[kCtrLeft] saddles, in `left`) goes to the sorted
// finish, which continues Alg. 1 exactly for any number of saddles.
__global__ void __launch_bounds__(kRoundThreads, 4) pair_rounds(const Rounds R, int32_t* dstatus) {
  __shared__ RoundAppend sh;
  unsigned int* const ctr = R.ctr;
  const Tri T = R.T;
  const Nodes nd = R.nd;
  const int64_t nn = (R.n_dev ? *R.n_dev : 0) + R.nnode;
  unsigned int epoch = 0, round = R.round;
  unsigned int n = __ldcg(R.n);
  uint32_t *cur = R.cur, *nxt = R.nxt;
  bool solo = gridDim.x == 1, forest = R.forest != nullptr, found = R.first_found;
  for (;;) {
    if (!solo && goes_solo(n, nn, forest)) {
      if (blockIdx.x != 0) return;
      solo = true;
    }
    const unsigned int first = (solo ? 0 : blockIdx.x * kRoundThreads) + threadIdx.x;
    const unsigned int step = solo ? kRoundThreads : gridDim.x * kRoundThreads;
    if (n == 0) {
      if (!forest || R.forest_only) return;
      // the forest is complete: single components again, its saddles live
      forest = false;
      for (int64_t i = first; i < nn; i += step) {
        nd.parent[i] = (uint32_t)i;
        nd.best[i] = 0ull;
      }
      n = __ldcg(ctr + kCtrForest);
      if (first < 3) ctr[count_word(first, solo)] = 0;
      nxt = R.cur;
      cur = R.forest;
      round = 1;
      if (!round_sync(ctr, epoch, solo)) break;
      continue;
    }
    if (forest && round > kMaxForestRounds) break;
    if (!found) {
      for (unsigned int j = first; j < n; j += step) find_saddle(T, nd, cur[j], round);
      if (!round_sync(ctr, epoch, solo)) break;
    }
    found = false;
    // the next round's word was last read two rounds ago
    unsigned int* const nxt_n = ctr + count_word(round, solo);
    if (first == 0) ctr[count_word(round + 1, solo)] = 0;
    // CTA-uniform passes: every thread reaches the appends
    for (unsigned int base = first - threadIdx.x; base < n; base += step) {
      const unsigned int j = base + threadIdx.x;
      bool wait = false, tree = false;
      const uint32_t i = j < n ? cur[j] : 0;
      if (j < n) {
        if (forest) hook_saddle<true>(T, nd, i, round, wait, tree);
        else merge_saddle<true>(T, nd, i, round, wait);
      }
      round_append2(sh, wait, nxt, nxt_n, tree, R.forest, ctr + kCtrForest, i);
    }
    if (!round_sync(ctr, epoch, solo)) break;
    const unsigned int left = __ldcg(nxt_n);
    uint32_t* const t = cur;
    cur = nxt;
    nxt = t;
    ++round;
    if (!forest && left && ((uint64_t)left * 64 > (uint64_t)n * 63 || round > kMaxExactRounds)) {
      for (unsigned int j = first; j < left; j += step) R.left[j] = cur[j];
      if (first == 0) ctr[kCtrLeft] = left;
      return;
    }
    n = left;
  }
  // a barrier that ran out, or a forest that does not end
  if (threadIdx.x == 0) set_status(dstatus, DMS_ERR_TIMEOUT);
}

// launches pair_rounds for at most n live saddles (its own words of ctr are
// zero: all from kCtrRound on)
int launch_rounds(const Rounds& R, int64_t n, int32_t* dstatus, cudaStream_t s) {
  // the device's resident CTAs: asked once per device, by any thread (they find the same)
  constexpr int kDevices = 64;
  static std::atomic<int> resident[kDevices];
  int dev = 0, blocks = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return DMS_ERR_CUDA;
  if (dev < kDevices) blocks = resident[dev].load(std::memory_order_relaxed);
  if (blocks == 0) {
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pair_rounds, kRoundThreads, 0) !=
            cudaSuccess ||
        per_sm < 1)
      return DMS_ERR_CUDA;
    blocks = sms * per_sm;
    if (dev < kDevices) resident[dev].store(blocks, std::memory_order_relaxed);
  }
  const unsigned grid =
      n <= (int64_t)kSolo ? 1u
                          : (unsigned)std::min<int64_t>(blocks, (n + kRoundThreads - 1) / kRoundThreads);
  Rounds r = R;
  void* args[2] = {&r, &dstatus};
  if (cudaLaunchCooperativeKernel((const void*)pair_rounds, dim3(grid), dim3(kRoundThreads), args, 0,
                                  s) != cudaSuccess)
    return DMS_ERR_CUDA;
  count_launch();
  return DMS_OK;
}

// The last few live saddles, processed one by one in increasing weight: the
// lightest live saddle is always the lightest of both of its components, so
// this continues Alg. 1 exactly.
__global__ void gather_live(const uint32_t* __restrict__ live, const unsigned int* __restrict__ live_n,
                            const Tri T, unsigned long long* keys, uint32_t* vals) {
  unsigned int n = *live_n;
  for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    keys[j] = T.s[live[j]].w;
    vals[j] = live[j];
  }
}

__global__ void sequential_finish(const uint32_t* __restrict__ sorted, const unsigned int* __restrict__ live_n,
                                  Tri T, Nodes nd) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  unsigned int n = *live_n;
  for (unsigned int j = 0; j < n; ++j) {
    uint32_t i = sorted[j];
    uint32_t a = T.s[i].na, b = T.s[i].nb;
    while (nd.parent[a] != a) a = nd.parent[a] = nd.parent[nd.parent[a]];
    while (nd.parent[b] != b) b = nd.parent[b] = nd.parent[nd.parent[b]];
    if (a == b) continue;
    uint32_t young = nd.age[a] > nd.age[b] ? a : b;
    uint32_t old = young == a ? b : a;
    nd.parent[young] = old;
    T.s[i].res = young;
  }
}

// ---------------------------------------------------------------------------
// The paired saddles as records in saddle-id order: one launch.  A CTA takes a
// tile of PTILE saddles by ticket, counts its pairs, and learns how many lie
// before it by decoupled look-back: every tile publishes its own count, then,
// when it knows it, the count up to its end; a warp reads the tiles before its
// own back to the first that has the latter.  Tickets are drawn in order, so
// the tiles that a CTA waits for are running or done; the waits are bounded
// all the same.
// Bound by the gathers of the carriers' orders and values, so a thread has four
// independent saddles of a strided tile in flight (16 consecutive ones, one
// after the other, before): with the counting and scanning launches gone, 2D
// 16384^2 (76.6 M pairs) 10.8 -> 3 ms for both lists, the D0/D2 stage of 512^3
// ties 30.5 -> 28.9 ms, of a 24^3 mixture 444 -> 407 us.
// ---------------------------------------------------------------------------
constexpr int PNT = 256, PITEMS = 4, PTILE = PNT * PITEMS;
constexpr uint32_t kLookPolls = 1u << 22;

// words of the look-back: a ticket counter, the tiles' states (2 bits: 1 the
// tile's count, 2 the count up to its end; 62 bits: that count), zero at first
inline int64_t look_words(int64_t nsad) { return 1 + (nsad + PTILE - 1) / PTILE; }

struct PairSmem {
  unsigned int cnt[PITEMS][PNT / 32];
  unsigned int total;
  long long before;
  long long tile;
};

// the tile of this CTA (every thread calls)
__device__ __forceinline__ int64_t take_tile(PairSmem& sm, unsigned long long* look) {
  if (threadIdx.x == 0) sm.tile = (long long)atomicAdd(look, 1ull);
  __syncthreads();
  return sm.tile;
}

// places of the tile's pairs: at[k] for the saddle tile * PTILE + k * PNT +
// threadIdx.x where paired[k]; *total (last tile only) all pairs
__device__ __forceinline__ void place_pairs(PairSmem& sm, unsigned long long* look, int64_t tile,
                                            const bool (&paired)[PITEMS], int64_t (&at)[PITEMS],
                                            int32_t* dstatus) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = PNT / 32;
  static_assert(PITEMS * NW == 32, "one warp scans the warps' counts");
  unsigned bal[PITEMS];
#pragma unroll
  for (int k = 0; k < PITEMS; ++k) {
    bal[k] = __ballot_sync(0xFFFFFFFFu, paired[k]);
    if (lane == 0) sm.cnt[k][warp] = __popc(bal[k]);
  }
  __syncthreads();
  if (warp == 0) {
    unsigned int* c = &sm.cnt[0][0];
    const unsigned int x = c[lane];
    unsigned int t = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xFFFFFFFFu, t, o);
      if (lane >= o) t += y;
    }
    c[lane] = t - x;
    const unsigned long long total = __shfl_sync(0xFFFFFFFFu, t, 31);
    volatile unsigned long long* st = look + 1;
    constexpr unsigned long long kOwn = 1ull << 62, kUpTo = 2ull << 62, kVal = kOwn - 1;
    if (lane == 0) st[tile] = (tile == 0 ? kUpTo : kOwn) | total;
    unsigned long long before = 0;
    for (int64_t j = tile - 1; j >= 0; j -= 32) {  // the 32 tiles up to j
      const int64_t i = j - lane;
      unsigned long long v = kUpTo;  // (before the first tile: nothing)
      if (i >= 0) {
        uint32_t it = 0;
        do {
          v = st[i];
        } while ((v >> 62) == 0 && ++it < kLookPolls);
        if ((v >> 62) == 0) {
          set_status(dstatus, DMS_ERR_TIMEOUT);
          v = kUpTo;
        }
      }
      const unsigned full = __ballot_sync(0xFFFFFFFFu, (v >> 62) == 2);
      unsigned long long s = (!full || lane <= __ffs(full) - 1) ? v & kVal : 0ull;
#pragma unroll
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
      before += s;
      if (full) break;
    }
    if (lane == 0) {
      if (tile > 0) st[tile] = kUpTo | (before + total);
      sm.before = (long long)before;
      sm.total = (unsigned int)total;
    }
  }
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int k = 0; k < PITEMS; ++k) at[k] = sm.before + sm.cnt[k][warp] + __popc(bal[k] & lt);
}

__device__ __forceinline__ int64_t top_of(const Dev& D, const uint32_t* order, const int64_t* v,
                                          int m) {
  int64_t best = v[0];
  uint32_t ob = __ldg(order + v[0]);
  for (int j = 1; j < m; ++j) {
    uint32_t o = __ldg(order + v[j]);
    if (o > ob) {
      ob = o;
      best = v[j];
    }
  }
  return best;
}

__device__ __forceinline__ void write_one_d0(const Dev& D, const float* f, const uint32_t* order,
                                            const int64_t* crit0, const int64_t* crit1,
                                            const Tri& T, int64_t i, dms_pair* out) {
  int64_t m = crit0[T.s[i].res];
  int64_t id = crit1[i];
  int64_t a = id / 7;
  int k = (int)(id - a * 7);
  int64_t v[2] = {a, a + corner_delta(D.g, edge_corner(k))};
  int64_t top = top_of(D, order, v, 2);
  dms_pair p;
  p.birth_id = m;
  p.death_id = id;
  p.birth = __ldg(f + m);
  p.death = __ldg(f + top);
  p.birth_vtx = (uint32_t)m;
  p.death_vtx = (uint32_t)top;
  *out = p;
}

__device__ __forceinline__ void write_one_d2(const Dev& D, const float* f, const uint32_t* order,
                                            const int64_t* crit2, const int64_t* crit3,
                                            const Tri& T, int64_t i, dms_pair* out) {
  int64_t tet = crit3[T.s[i].res - 1];  // node 0 (OUTSIDE) never dies
  int64_t tri = crit2[i];
  int64_t a = tri / 12;
  int k = (int)(tri - a * 12);
  int64_t tv[3] = {a, a + corner_delta(D.g, tri_p(k)), a + corner_delta(D.g, tri_q(k))};
  int64_t b = tet / 6;
  int kk = (int)(tet - b * 6);
  int64_t qv[4] = {b, b + corner_delta(D.g, tet_c1(kk)), b + corner_delta(D.g, tet_c2(kk)),
                   b + corner_delta(D.g, 7)};
  int64_t st = top_of(D, order, tv, 3), qt = top_of(D, order, qv, 4);
  dms_pair p;
  p.birth_id = tri;
  p.death_id = tet;
  p.birth = __ldg(f + st);
  p.death = __ldg(f + qt);
  p.birth_vtx = (uint32_t)st;
  p.death_vtx = (uint32_t)qt;
  *out = p;
}

// dim 0 -> D0 records, dim 2 -> D2 records, in saddle-id order
__global__ void __launch_bounds__(PNT) write_pairs(int dim, Dev D, const float* __restrict__ f,
                                                   const uint32_t* __restrict__ order,
                                                   const int64_t* __restrict__ critA,
                                                   const int64_t* __restrict__ critB, const Tri T,
                                                   int64_t nsad, unsigned long long* look,
                                                   dms_pair* out, int64_t cap, int64_t* n_out,
                                                   int32_t* dstatus) {
  __shared__ PairSmem sm;
  const int64_t tile = take_tile(sm, look), base = tile * PTILE + threadIdx.x;
  bool paired[PITEMS];
  int64_t at[PITEMS];
#pragma unroll
  for (int k = 0; k < PITEMS; ++k)
    paired[k] = base + k * PNT < nsad && T.s[base + k * PNT].res != kNone;
  place_pairs(sm, look, tile, paired, at, dstatus);
  if (tile == gridDim.x - 1 && threadIdx.x == 0) {
    const int64_t total = sm.before + sm.total;
    *n_out = total;
    if (total > cap) set_status(dstatus, DMS_ERR_CAPACITY);
  }
#pragma unroll
  for (int k = 0; k < PITEMS; ++k) {
    if (!paired[k] || at[k] >= cap) continue;
    if (dim == 0) write_one_d0(D, f, order, critA, critB, T, base + k * PNT, out + at[k]);
    else write_one_d2(D, f, order, critA, critB, T, base + k * PNT, out + at[k]);
  }
}

__global__ void write_essential(const float* __restrict__ f, const uint32_t* __restrict__ order,
                                const int64_t* __restrict__ crit0, int64_t nmin, dms_pair* ess) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= nmin) return;
  int64_t m = crit0[i];
  if (__ldg(order + m) != 0u) return;  // the global minimum never dies
  dms_pair p;
  p.birth_id = m;
  p.death_id = -1;
  p.birth = __ldg(f + m);
  p.death = __int_as_float(0x7F800000);
  p.birth_vtx = (uint32_t)m;
  p.death_vtx = 0;
  *ess = p;
}

struct DiagWs {
  Tri T0, T2;
  uint32_t *live0, *live1;
  uint32_t* forest;  // the spanning-forest saddles found by the Borůvka rounds
  unsigned int* ctr;  // counts (kCtr...)
  Nodes nd;  // union-find nodes: parent, best live saddle, age
  // the self-correcting pairing's next links (the current ones live in
  // nd.parent and nd.best)
  uint32_t* sc_parent;
  unsigned long long* sc_w;
  uint32_t* path;  // one word per cell (vertex / tet id): where its path goes on or ends
  radix64::Buffers rb;
  size_t bytes;
};

// nc: counts of the node and saddle lists as for 3D (minima, edges, triangles,
// tets); npath: path words, one per vertex / tet id the walks may visit
DiagWs carve_diag(void* base, const int64_t* nc, int64_t npath) {
  WsCarver c(base);
  DiagWs w;
  const int64_t nsad = std::max<int64_t>(std::max<int64_t>(nc[1], nc[2]), 1);
  const int64_t nnode = std::max<int64_t>(nc[0], nc[3] + 1);
  static_assert(sizeof(Sad) == 32, "one sector per saddle");
  w.T0.s = c.take<Sad>(nsad);
  w.T2 = w.T0;  // D0 and D2 run one after the other and share the arrays
  w.live0 = c.take<uint32_t>(nsad);
  w.live1 = c.take<uint32_t>(nsad);
  w.forest = c.take<uint32_t>(nsad);
  w.ctr = c.take<unsigned int>(kCtrWords);
  w.nd.parent = c.take<uint32_t>(nnode);
  w.nd.best = c.take<unsigned long long>(nnode);
  w.nd.age = c.take<uint64_t>(nnode);
  w.nd.immortal = kNone;
  w.sc_parent = c.take<uint32_t>(nnode);
  w.sc_w = c.take<unsigned long long>(nnode);
  w.path = c.take<uint32_t>(npath);
  w.rb = radix64::carve(c, std::max<int64_t>(nsad, 4096));
  w.bytes = c.used;
  return w;
}

// Whether the paths of nsad saddles are followed cell by cell.  The bricks cost
// the same however few the saddles are, 21 ns per 1000 vertices; the walks
// break even at 0.03 saddles per vertex on every grid that is large enough for
// the depth of their chains to be hidden.  D0/D2 stage by bricks and by cells:
// 1024^3 mixtures of 2e-7, 2.3e-3, 9e-3, 3.0e-2 and 5.6e-2 saddles per vertex
// 23.2 / 3.7, 25.4 / 7.4, 30.5 / 17.8, 41.4 / 41.9 and 50.9 / 63.3 ms; 512^3,
// 1.3e-6, 4e-3, 1.6e-2, 3.2e-2 and 5.9e-2: 3.28 / 1.64, 3.82 / 2.06, 4.64 / 3.61,
// 5.86 / 5.87 and 8.18 / 9.65; 384^3, 8e-6 and 2.8e-2: 1.60 / 1.42 and 2.86 /
// 2.84; 256^3, 1e-5 and 2.3e-2: 0.72 / 0.99 and 1.25 / 1.31.
//
// Bricks that reach far outside a thin grid cost nearly what full ones do, so
// there the walks win at any density that keeps them short.  By bricks and by
// cells, (z, y, x): 4096 x 4096 x 2 noise 8.7 / 3.4 ms, 4096 x 2 x 4096 6.1 /
// 3.5, 4096 x 2048 x 4 (bricks four times the grid) 7.0 / 4.8, 2048 x 1024 x 2
// 1.6 / 0.95; 1024 x 1024 x 2 1.1 / 0.8, 512 x 512 x 2 0.60 / 0.55; 2048 x 2048
// x 6 (not four times) 5.0 / 4.2; smooth fields, whose walks are long: 2 x 2048
// x 2048 0.71 / 1.24, 20,000 x 9 x 9 1.2 / 5.6.
constexpr int64_t kFewGrid = 1 << 25, kFewPer = 32, kThinGrid = 1 << 21, kThinBricks = 4, kThinPer = 64;
template <class P>
bool follow_by_cells(int64_t nsad, const Grid& g) {
  if (2 * nsad >= (int64_t)kLink) return false;
  const int64_t bricks = brick_count<P>(g.nx, g.ny, g.nz) << (P::LX + P::LY + P::LZ);
  return (g.n >= kFewGrid && nsad <= g.n / kFewPer) ||
         (g.n >= kThinGrid && bricks >= kThinBricks * g.n && nsad >= g.n / kThinPer);
}

// the saddles' weights and ends: link(kernel, n) launches one of the three
template <class P, class S, class L, class K>
int link_saddles(DiagWs& w, const P& paths, const S& starts, uint32_t node0, int64_t nsad, const L& link,
                 K* bricks, K* cells, K* far, cudaStream_t s) {
  const Grid& g = paths.fields.g;
  const bool cells_first = follow_by_cells<P>(nsad, g);
  if (cells_first) {
    const int64_t nb = (g.n / kRun + 1) * kGroup * P::K / 256 + 1;
    clear_landmarks<P><<<(unsigned)std::min<int64_t>(nb, 1 << 16), 256, 0, s>>>(g.n, w.path); count_launch();
  }
  if (paths.n > 0) {
    mark_ends<<<(unsigned)((paths.n + 255) / 256), 256, 0, s>>>(paths.ends, nullptr, paths.n, node0, w.path); count_launch();
  }
  if (cells_first) {
    follow_cells<<<(unsigned)((2 * nsad + 255) / 256), 256, 0, s>>>(
        paths, starts, 2 * nsad, w.path, reinterpret_cast<uint32_t*>(w.rb.ka)); count_launch();
    link(cells, nsad);
    unsigned int h = 0;
    DMS_CUDA_OK(cudaMemcpyAsync(&h, w.ctr + kCtrFar, sizeof(h), cudaMemcpyDeviceToHost, s));
    DMS_CUDA_OK(cudaStreamSynchronize(s));
    if (h == 0) return launch_status();
    bricks = far;
    nsad = h;
  }
  resolve_paths<<<(unsigned)brick_count<P>(g.nx, g.ny, g.nz), kBrickThreads, 0, s>>>(paths, w.path); count_launch();
  link(bricks, nsad);
  return launch_status();
}

// the saddles that the rounds left live, if any, in sorted order
int finish_sorted(DiagWs& w, Tri T, cudaStream_t s) {
  unsigned int h = 0;
  DMS_CUDA_OK(cudaMemcpyAsync(&h, w.ctr + kCtrLeft, sizeof(h), cudaMemcpyDeviceToHost, s));
  DMS_CUDA_OK(cudaStreamSynchronize(s));
  if (h == 0) return DMS_OK;
  gather_live<<<(h + 255) / 256, 256, 0, s>>>(w.live1, w.ctr + kCtrLeft, T, w.rb.ka, w.rb.va); count_launch();
  const bool in_a = radix64::sort(w.rb, h, 44, s);
  sequential_finish<<<1, 32, 0, s>>>(in_a ? w.rb.va : w.rb.vb, w.ctr + kCtrLeft, T, w.nd); count_launch();
  return launch_status();
}

// rounds of one launch per phase while more than kOneLaunch saddles are live:
// cur/nxt with the counts cur_n/nxt_n in turn, from `round` on; forest: the
// Borůvka rounds
int run_large(DiagWs& w, Tri T, uint32_t*& cur, unsigned int*& cur_n, uint32_t*& nxt,
              unsigned int*& nxt_n, unsigned int& round, unsigned int h, bool forest, bool found,
              cudaStream_t s) {
  while ((int64_t)h > kOneLaunch) {
    if (round > kMaxForestRounds) return forest ? DMS_ERR_TIMEOUT : DMS_OK;
    const unsigned int prev = h;
    const unsigned int blocks = std::min((h + 255) / 256, 1u << 16);
    DMS_CUDA_OK(cudaMemsetAsync(nxt_n, 0, sizeof(unsigned int), s));
    if (!found) {
      round_find<<<blocks, 256, 0, s>>>(cur, cur_n, T, w.nd, round); count_launch();
    }
    found = false;
    if (forest) {
      boruvka_hook<<<blocks, 256, 0, s>>>(cur, cur_n, T, w.nd, round, nxt, nxt_n, w.forest,
                                          w.ctr + kCtrForest); count_launch();
    } else {
      round_merge<<<blocks, 256, 0, s>>>(cur, cur_n, T, w.nd, round, nxt, nxt_n); count_launch();
    }
    std::swap(cur, nxt);
    std::swap(cur_n, nxt_n);
    ++round;
    DMS_CUDA_OK(cudaMemcpyAsync(&h, cur_n, sizeof(h), cudaMemcpyDeviceToHost, s));
    DMS_CUDA_OK(cudaStreamSynchronize(s));
    if (!forest && (uint64_t)h * 64 > (uint64_t)prev * 63) break;  // pair_rounds will end, too
  }
  return DMS_OK;
}

// pairs the live saddles in w.live0 (ctr[kCtrLive], of nsad) over nnode nodes:
// Borůvka rounds collect the spanning forest's saddles, the exact rounds pair
// them (forest false: the exact rounds on all live saddles)
int run_pairing(DiagWs& w, Tri T, int64_t nsad, int64_t nnode, cudaStream_t s, int32_t* dstatus,
                bool forest) {
  Rounds r;
  r.T = T;
  r.nd = w.nd;
  r.cur = w.live0;
  r.nxt = forest ? w.live1 : w.forest;
  r.n = w.ctr + kCtrLive;
  r.round = 1;
  r.forest = forest ? w.forest : nullptr;
  r.forest_only = false;
  r.first_found = forest;
  r.left = w.live1;
  r.ctr = w.ctr;
  r.n_dev = nullptr;
  r.nnode = nnode;
  if (nsad > kOneLaunch) {
    uint32_t *cur = r.cur, *nxt = r.nxt;
    unsigned int *cur_n = w.ctr + kCtrLive, *nxt_n = w.ctr + kCtrNext, h = 0;
    DMS_CUDA_OK(cudaMemcpyAsync(&h, cur_n, sizeof(h), cudaMemcpyDeviceToHost, s));
    DMS_CUDA_OK(cudaStreamSynchronize(s));
    if (forest) {
      const bool more = (int64_t)h > kOneLaunch;
      DMS_TRY(run_large(w, T, cur, cur_n, nxt, nxt_n, r.round, h, true, true, s));
      r.cur = cur;
      r.nxt = nxt;
      r.n = cur_n;
      r.forest_only = true;
      r.first_found = !more;
      DMS_TRY(launch_rounds(r, kOneLaunch, dstatus, s));
      const unsigned int nb = (unsigned int)std::min<int64_t>((nnode + 255) / 256, 1 << 16);
      reset_nodes<<<std::max(nb, 1u), 256, 0, s>>>(w.nd, nullptr, nnode); count_launch();
      DMS_CUDA_OK(cudaMemcpyAsync(&h, w.ctr + kCtrForest, sizeof(h), cudaMemcpyDeviceToHost, s));
      DMS_CUDA_OK(cudaMemsetAsync(w.ctr + kCtrRound, 0, (kCtrWords - kCtrRound) * sizeof(unsigned int), s));
      DMS_CUDA_OK(cudaStreamSynchronize(s));
      cur = w.forest;
      cur_n = w.ctr + kCtrForest;
      nxt = w.live0;
      nxt_n = w.ctr + kCtrLive;
      r.round = 1;
      r.forest = nullptr;
      r.forest_only = r.first_found = false;
    }
    DMS_TRY(run_large(w, T, cur, cur_n, nxt, nxt_n, r.round, h, false, false, s));
    r.cur = cur;
    r.nxt = nxt;
    r.n = cur_n;
  }
  DMS_TRY(launch_rounds(r, nsad, dstatus, s));
  return finish_sorted(w, T, s);
}

// ---------------------------------------------------------------------------
// The paper's self-correcting pairing (Sec. 4.3, Alg. 4) as a GPU fixpoint,
// an alternative to the Borůvka forest + exact rounds above.
//
// Every extremum e holds a link (parent, saddle): the root it was merged
// into and the saddle that merged it -- the representative of Alg. 4 that
// also records the saddle which assigned it.  Every round, every live
// saddle sigma (all of them at once, as Alg. 4 runs all its triplets)
// computes the representatives of its two ends by following only links
// set by saddles that come before sigma in Alg. 1's order (earlier links
// exist at sigma's turn, later ones would not), with no path compression;
// if they differ, the younger one dies at sigma, and of several saddles
// that kill the same extremum the earliest wins (atomicMin of the weight).
// The links of the next round are exactly those winning claims.  A saddle
// whose representatives were computed from wrong links is recomputed in the
// next round -- the self-correction of Alg. 4 -- and by induction on the
// saddle order the k earliest saddles are right after k rounds, so the
// rounds stop, when no link changes, at Alg. 1's pairs.  The node arrays
// hold the current links: nd.parent (the parent, the node itself if none)
// and nd.best (the linking saddle's weight, kNoLink if none).
// ---------------------------------------------------------------------------
constexpr unsigned long long kNoLink = ~0ull;

__device__ __forceinline__ uint32_t sc_find(const Nodes& nd, uint32_t t, uint64_t w,
                                            uint32_t limit, int32_t* dstatus) {
  for (uint32_t it = 0; it <= limit; ++it) {
    if (nd.best[t] >= w) return t;  // no link, or one set by a later saddle
    t = nd.parent[t];
  }
  set_status(dstatus, DMS_ERR_TIMEOUT);  // links form no cycle: not reached
  return t;
}

__global__ void sc_reset(Nodes nd, unsigned long long* nw, int64_t nnode) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nnode;
       i += (int64_t)gridDim.x * blockDim.x) {
    nd.parent[i] = (uint32_t)i;
    nd.best[i] = kNoLink;
    nw[i] = kNoLink;
  }
}

// representatives of both ends as of each saddle's turn; claim the younger
__global__ void sc_claim(const uint32_t* __restrict__ live, const unsigned int* __restrict__ live_n,
                         Tri T, Nodes nd, unsigned long long* nw, uint32_t nnode, int32_t* dstatus) {
  const unsigned int n = *live_n;
  for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    const uint32_t i = live[j];
    const uint64_t w = T.s[i].w;
    const uint32_t a = sc_find(nd, T.s[i].na, w, nnode, dstatus);
    const uint32_t b = sc_find(nd, T.s[i].nb, w, nnode, dstatus);
    if (a == b) {  // both ends already joined at this saddle's turn: no pair
      T.s[i].ra = kNone;
      continue;
    }
    const uint32_t young = nd.age[a] > nd.age[b] ? a : b;
    T.s[i].ra = young;
    T.s[i].rb = young == a ? b : a;
    atomicMin(nw + young, (unsigned long long)w);
  }
}

// the winning claims become the next round's links
__global__ void sc_link(const uint32_t* __restrict__ live, const unsigned int* __restrict__ live_n,
                        Tri T, uint32_t* np, const unsigned long long* __restrict__ nw) {
  const unsigned int n = *live_n;
  for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    const uint32_t i = live[j];
    const uint32_t young = T.s[i].ra;
    if (young != kNone && nw[young] == T.s[i].w) np[young] = T.s[i].rb;
  }
}

// current <- next; counts the nodes whose link changed
__global__ void sc_commit(Nodes nd, uint32_t* np, unsigned long long* nw, int64_t nnode,
                          unsigned int* changed) {
  unsigned int c = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nnode;
       i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long w = nw[i];
    const uint32_t p = w == kNoLink ? (uint32_t)i : np[i];
    if (w != nd.best[i] || p != nd.parent[i]) ++c;
    nd.best[i] = w;
    nd.parent[i] = p;
    nw[i] = kNoLink;
  }
  c = __reduce_add_sync(0xFFFFFFFFu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(changed, c);
}

// the pair of each live saddle from the final links
__global__ void sc_result(const uint32_t* __restrict__ live, const unsigned int* __restrict__ live_n,
                          Tri T, Nodes nd) {
  const unsigned int n = *live_n;
  for (unsigned int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    const uint32_t i = live[j];
    const uint32_t young = T.s[i].ra;
    T.s[i].res = (young != kNone && nd.best[young] == T.s[i].w) ? young : kNone;
  }
}

constexpr int kMaxSelfCorrectingRounds = 1 << 16;

int run_selfcorrecting(DiagWs& w, Tri T, int64_t nnode, cudaStream_t s, int32_t* dstatus) {
  unsigned int* live_n = w.ctr + kCtrLive;
  unsigned int* changed = w.ctr + kCtrChanged;
  unsigned int h = 0;
  DMS_CUDA_OK(cudaMemcpyAsync(&h, live_n, sizeof(h), cudaMemcpyDeviceToHost, s));
  DMS_CUDA_OK(cudaStreamSynchronize(s));
  const unsigned int nb = (unsigned int)std::min<int64_t>((nnode + 255) / 256, 1 << 16);
  sc_reset<<<std::max(nb, 1u), 256, 0, s>>>(w.nd, w.sc_w, nnode); count_launch();
  if (h == 0) return launch_status();
  const unsigned int blocks = (unsigned int)std::min<int64_t>((h + 255) / 256, 1 << 16);
  for (int round = 1;; ++round) {
    if (round > kMaxSelfCorrectingRounds) return DMS_ERR_TIMEOUT;
    DMS_CUDA_OK(cudaMemsetAsync(changed, 0, sizeof(unsigned int), s));
    sc_claim<<<blocks, 256, 0, s>>>(w.live0, live_n, T, w.nd, w.sc_w, (uint32_t)nnode, dstatus); count_launch();
    sc_link<<<blocks, 256, 0, s>>>(w.live0, live_n, T, w.sc_parent, w.sc_w); count_launch();
    sc_commit<<<std::max(nb, 1u), 256, 0, s>>>(w.nd, w.sc_parent, w.sc_w, nnode, changed); count_launch();
    unsigned int c = 0;
    DMS_CUDA_OK(cudaMemcpyAsync(&c, changed, sizeof(c), cudaMemcpyDeviceToHost, s));
    DMS_CUDA_OK(cudaStreamSynchronize(s));
    if (c == 0) break;
  }
  sc_result<<<blocks, 256, 0, s>>>(w.live0, live_n, T, w.nd); count_launch();
  return launch_status();
}

int write_diagram(int dim, DiagWs& w, const Dev& D, const float* f, const uint32_t* order,
                  const int64_t* critA, const int64_t* critB, int64_t nsad, dms_pair* out,
                  int64_t cap, int64_t* n_out, int32_t* dstatus, cudaStream_t s) {
  if (nsad <= 0) {
    DMS_CUDA_OK(cudaMemsetAsync(n_out, 0, sizeof(int64_t), s));
    return DMS_OK;
  }
  unsigned long long* look = w.rb.ka;
  DMS_CUDA_OK(cudaMemsetAsync(look, 0, look_words(nsad) * sizeof(*look), s));
  write_pairs<<<(unsigned)(look_words(nsad) - 1), PNT, 0, s>>>(dim, D, f, order, critA, critB, w.T0, nsad,
                                                               look, out, cap, n_out, dstatus); count_launch();
  return launch_status();
}

}  // namespace

size_t diagram_workspace_bytes(const Grid& g, const int64_t* n_crit) {
  return carve_diag(nullptr, n_crit, 6 * g.n).bytes;
}

int launch_diagram(const float* f, const uint32_t* order, const uint8_t* desc, const uint64_t* rec,
                   const Grid& g, const int64_t* crit0, const int64_t* crit1, const int64_t* crit2,
                   const int64_t* crit3, const int64_t* nc, dms_pair* d0, int64_t cap0,
                   dms_pair* d2, int64_t cap2, dms_pair* ess, int64_t* n_out, void* ws,
                   int32_t* dstatus, cudaStream_t s, int pairing) {
  DiagWs w = carve_diag(ws, nc, 6 * g.n);
  Dev D;
  D.g = g;
  for (int sl = 0; sl < 14; ++sl) {
    int c = kCornerOfEdge[sl % 7];
    int64_t d = (c & 1) + ((c >> 1) & 1) * g.nx + ((c >> 2) & 1) * g.sxy;
    D.slot_delta[sl] = sl < 7 ? d : -d;
  }
  const int TB = 256;
  auto nb = [&](int64_t n) { return (unsigned)std::max<int64_t>(1, (n + TB - 1) / TB); };
  uint32_t* const results = reinterpret_cast<uint32_t*>(w.rb.ka);  // (two words per saddle)

  // ---- D0
  DMS_CUDA_OK(cudaMemsetAsync(w.ctr, 0, kCtrWords * sizeof(unsigned int), s));
  if (nc[0] > 0) {
    init_nodes_d0<<<nb(nc[0]), TB, 0, s>>>(order, crit0, nc[0], w.nd); count_launch();
    write_essential<<<nb(nc[0]), TB, 0, s>>>(f, order, crit0, nc[0], ess); count_launch();
  }
  w.nd.immortal = kNone;  // every minimum but the global one can die
  if (nc[1] > 0) {
    using Paths = DescPaths<OneField>;
    const Paths paths{OneField{g}, desc, crit0, nullptr, nc[0]};
    auto link = [&](auto kernel, int64_t n) {
      kernel<<<nb(n), TB, 0, s>>>(paths, order, crit1, nullptr, n, w.path, w.T0, w.live0, w.ctr + kCtrLive,
                                  results, w.live1, w.ctr + kCtrFar, dstatus, pairing == 0, w.nd); count_launch();
    };
    DMS_TRY(link_saddles(w, paths, EdgeEnds{crit1}, 0u, nc[1], link, link_d0<kBricks, Paths>, link_d0<kCells, Paths>,
                         link_d0<kFar, Paths>, s));
  }
  int st = pairing == 1 ? run_selfcorrecting(w, w.T0, std::max<int64_t>(nc[0], 1), s, dstatus)
                        : run_pairing(w, w.T0, nc[1], std::max<int64_t>(nc[0], 1), s, dstatus, true);
  if (st) return st;
  st = write_diagram(0, w, D, f, order, crit0, crit1, nc[1], d0, cap0, n_out + 0, dstatus, s);
  if (st) return st;

  // ---- D2
  DMS_CUDA_OK(cudaMemsetAsync(w.ctr, 0, kCtrWords * sizeof(unsigned int), s));
  init_nodes_d2<<<nb(nc[3] + 1), TB, 0, s>>>(D, order, crit3, nc[3], w.nd); count_launch();
  w.nd.immortal = 0;  // OUTSIDE
  if (nc[2] > 0) {
    using Paths = DualPaths<OneField>;
    const Paths paths{OneField{g}, rec, crit3, nullptr, nc[3]};
    auto link = [&](auto kernel, int64_t n) {
      kernel<<<nb(n), TB, 0, s>>>(paths, order, crit2, nullptr, n, w.path, w.T2, w.live0, w.ctr + kCtrLive,
                                  results, w.live1, w.ctr + kCtrFar, dstatus, pairing == 0, w.nd); count_launch();
    };
    DMS_TRY(link_saddles(w, paths, TriCofacets{crit2}, 1u, nc[2], link, link_d2<kBricks, Paths>, link_d2<kCells, Paths>,
                         link_d2<kFar, Paths>, s));
  }
  st = pairing == 1 ? run_selfcorrecting(w, w.T2, nc[3] + 1, s, dstatus)
                    : run_pairing(w, w.T2, nc[2], nc[3] + 1, s, dstatus, true);
  if (st) return st;
  st = write_diagram(2, w, D, f, order, crit2, crit3, nc[2], d2, cap2, n_out + 1, dstatus, s);
  if (st) return st;
  return launch_status();
}

}  // namespace dms

// ===========================================================================
// Batched form: many fields in one pass, nothing synchronising the host.
// The critical lists hold GLOBAL ids (anchors in the concatenated arrays);
// every field is traced with its own dims; the pairing's rounds run on the
// device, which reads the counts, until they end (pair_rounds), and what they
// leave is finished in sorted order.  D0 graphs of different
// fields are disjoint; the D2 graphs share the OUTSIDE node, which is older
// than every maximum, so each field's pairs are those it has alone.
// ===========================================================================
namespace dms {
namespace {

struct FieldTab {
  const dms_field_desc* fd;
  int n;
};

__device__ __forceinline__ int field_of_vertex(const FieldTab& ft, int64_t v) {
  int lo = 0, hi = ft.n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (ft.fd[mid].offset <= v) lo = mid;
    else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ Grid grid_of(const dms_field_desc& d) {
  Grid g;
  g.nx = d.nx;
  g.ny = d.ny;
  g.nz = d.nz;
  g.sxy = (int64_t)d.nx * d.ny;
  g.n = g.sxy * d.nz;
  return g;
}

__device__ __forceinline__ int64_t slot_delta_of(const Grid& g, int s) {
  const int k = s < 7 ? s : s - 7;
  const int c = (0x7653421 >> (4 * k)) & 15;
  const int64_t d = (c & 1) + ((c >> 1) & 1) * g.nx + ((c >> 2) & 1) * g.sxy;
  return s < 7 ? d : -d;
}

// rank of u among the lower neighbours of t (global index, field offset off)
__device__ __forceinline__ uint32_t local_rank_f(const Grid& g, int64_t off,
                                                 const uint32_t* __restrict__ order, int64_t t,
                                                 uint32_t ou) {
  int64_t x, y, z;
  xyz(g, t - off, x, y, z);
  uint32_t r = 0;
#pragma unroll
  for (int s = 0; s < 14; ++s) {
    const int c = (0x7653421 >> (4 * (s < 7 ? s : s - 7))) & 15;
    const int sg = s < 7 ? 1 : -1;
    const int64_t nx = x + sg * (c & 1), ny = y + sg * ((c >> 1) & 1), nz = z + sg * ((c >> 2) & 1);
    if (nx < 0 || ny < 0 || nz < 0 || nx >= g.nx || ny >= g.ny || nz >= g.nz) continue;
    r += __ldg(order + t + slot_delta_of(g, s)) < ou ? 1u : 0u;
  }
  return r;
}

__global__ void b_init_nodes_d0(const uint32_t* __restrict__ order, const int64_t* __restrict__ crit0,
                                const int64_t* __restrict__ cnt, Nodes nd) {
  const int64_t n = cnt[0];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    nd.parent[i] = (uint32_t)i;
    nd.best[i] = 0ull;
    nd.age[i] = __ldg(order + crit0[i]);
  }
}

__global__ void b_essential(const FieldTab ft, const float* __restrict__ f,
                            const uint32_t* __restrict__ order, const int64_t* __restrict__ crit0,
                            const int64_t* __restrict__ cnt, dms_pair* ess) {
  const int64_t n = cnt[0];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = crit0[i];
    if (__ldg(order + m) != 0u) continue;  // each field's global minimum
    const int fi = field_of_vertex(ft, m);
    const int64_t lm = m - ft.fd[fi].offset;
    dms_pair p;
    p.birth_id = lm;
    p.death_id = -1;
    p.birth = __ldg(f + m);
    p.death = __int_as_float(0x7F800000);
    p.birth_vtx = (uint32_t)lm;
    p.death_vtx = 0;
    ess[fi] = p;
  }
}

__global__ void b_init_nodes_d2(const FieldTab ft, const uint32_t* __restrict__ order,
                                const int64_t* __restrict__ crit3, const int64_t* __restrict__ cnt,
                                Nodes nd) {
  const int64_t nmax = cnt[3];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= nmax;
       i += (int64_t)gridDim.x * blockDim.x) {
    nd.parent[i] = (uint32_t)i;
    nd.best[i] = 0ull;
    if (i == 0) {
      nd.age[0] = 0;  // OUTSIDE is older than every maximum of every field
      continue;
    }
    const int64_t id = crit3[i - 1];
    const int64_t a = id / 6;
    const int k = (int)(id - a * 6);
    const dms_field_desc fd = ft.fd[field_of_vertex(ft, a)];
    const Grid g = grid_of(fd);
    const int cs[4] = {0, tet_c1(k), tet_c2(k), 7};
    int64_t v[4];
    uint32_t o[4];
    int it = 0;
    for (int j = 0; j < 4; ++j) {
      v[j] = a + corner_delta(g, cs[j]);
      o[j] = __ldg(order + v[j]);
      if (o[j] > o[it]) it = j;
    }
    uint32_t r[3];
    int n = 0;
    for (int j = 0; j < 4; ++j)
      if (j != it) r[n++] = local_rank_f(g, fd.offset, order, v[it], o[j]);
    const uint32_t h = max(r[0], max(r[1], r[2])), l = min(r[0], min(r[1], r[2]));
    const uint32_t m = r[0] + r[1] + r[2] - h - l;
    const uint64_t key = ((uint64_t)o[it] << 12) | (h << 8) | (m << 4) | l;
    nd.age[i] = (kMask44 - key) + 1;
  }
}

// the fields' first bricks (one small CTA): fields in turn, a few hundred
__global__ void brick_table(const FieldTab ft, int lx, int ly, int lz, int64_t* brick0) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  int64_t acc = 0;
  for (int f = 0; f < ft.n; ++f) {
    brick0[f] = acc;
    const dms_field_desc d = ft.fd[f];
    acc += (int64_t)((d.nx + (1 << lx) - 1) >> lx) * ((d.ny + (1 << ly) - 1) >> ly) *
           ((d.nz + (1 << lz) - 1) >> lz);
  }
  brick0[ft.n] = acc;
}

// the saddles still live after the rounds, finished in increasing weight in
// one CTA: bitonic sort in shared memory, then one thread runs Alg. 1
constexpr int kFinishMax = 4096;
__global__ void __launch_bounds__(1024) b_finish(const uint32_t* __restrict__ live,
                                                 const unsigned int* __restrict__ live_n, Tri T,
                                                 Nodes nd,
                                                 int32_t* dstatus) {
  __shared__ unsigned long long key[kFinishMax];
  __shared__ uint32_t idx[kFinishMax];
  const unsigned int n = *live_n;
  if (n == 0 || n > (unsigned)kFinishMax) return;  // more: the sorted finish below
  (void)dstatus;
  for (int i = threadIdx.x; i < kFinishMax; i += blockDim.x) {
    key[i] = i < (int)n ? T.s[live[i]].w : ~0ull;
    idx[i] = i < (int)n ? live[i] : kNone;
  }
  __syncthreads();
  for (int size = 2; size <= kFinishMax; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < kFinishMax; i += blockDim.x) {
        const int j = i ^ stride;
        if (j > i) {
          const bool up = (i & size) == 0;
          if ((key[i] > key[j]) == up) {
            const unsigned long long tk = key[i];
            key[i] = key[j];
            key[j] = tk;
            const uint32_t ti = idx[i];
            idx[i] = idx[j];
            idx[j] = ti;
          }
        }
      }
      __syncthreads();
    }
  if (threadIdx.x != 0) return;
  for (unsigned int j = 0; j < n; ++j) {
    const uint32_t i = idx[j];
    uint32_t a = T.s[i].na, b = T.s[i].nb;
    while (nd.parent[a] != a) a = nd.parent[a] = nd.parent[nd.parent[a]];
    while (nd.parent[b] != b) b = nd.parent[b] = nd.parent[nd.parent[b]];
    if (a == b) continue;
    const uint32_t young = nd.age[a] > nd.age[b] ? a : b;
    nd.parent[young] = young == a ? b : a;
    T.s[i].res = young;
  }
}

// the count of live saddles left to the device-wide sorted finish (those
// the one-CTA finish does not take), for the kernels that read it
__global__ void b_big_count(const unsigned int* __restrict__ live_n, unsigned int* big_n) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const unsigned int n = *live_n;
    *big_n = n > (unsigned)kFinishMax ? n : 0u;
  }
}

// per-field pair counts, then offsets (one CTA; fields are few)
__global__ void b_count_fields(const FieldTab ft, const Tri T, const int64_t* __restrict__ crit,
                               const int64_t* __restrict__ n_dev, int per_anchor,
                               unsigned long long* fcount) {
  const int64_t n = *n_dev;
  const int lane = threadIdx.x & 31;
  // the saddles are in field order, so the lanes of a warp mostly share a
  // field: one atomic per field present in the warp, not one per pair
  for (int64_t base = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) - lane; base < n;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = base + lane;
    const int f = (i < n && T.s[i].res != kNone) ? field_of_vertex(ft, crit[i] / per_anchor) : -1;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, f);
    if (f >= 0 && lane == __ffs(peers) - 1) atomicAdd(fcount + f, (unsigned long long)__popc(peers));
  }
}

__global__ void b_field_offsets(const unsigned long long* __restrict__ fcount, int nfields,
                                int64_t* offsets, int64_t* total, int64_t cap, int32_t* dstatus) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  int64_t acc = 0;
  for (int f = 0; f < nfields; ++f) {
    offsets[f] = acc;
    acc += (int64_t)fcount[f];
  }
  offsets[nfields] = acc;
  *total = acc;
  if (acc > cap) set_status(dstatus, DMS_ERR_CAPACITY);
}

// pairs in saddle order (= field order), ids made local to the field
__global__ void __launch_bounds__(PNT) b_write_pairs(int dim, const FieldTab ft,
                                                     const float* __restrict__ f,
                                                     const uint32_t* __restrict__ order,
                                                     const int64_t* __restrict__ critA,
                                                     const int64_t* __restrict__ critB, const Tri T,
                                                     const int64_t* __restrict__ n_dev,
                                                     unsigned long long* look,
                                                     dms_pair* out, int64_t cap, int32_t* dstatus) {
  __shared__ PairSmem sm;
  const int64_t nsad = *n_dev;
  const int64_t tile = take_tile(sm, look), base = tile * PTILE + threadIdx.x;
  if (tile * PTILE >= nsad) return;  // (no tile with saddles waits for this one)
  bool paired[PITEMS];
  int64_t at[PITEMS];
#pragma unroll
  for (int k = 0; k < PITEMS; ++k)
    paired[k] = base + k * PNT < nsad && T.s[base + k * PNT].res != kNone;
  place_pairs(sm, look, tile, paired, at, dstatus);
#pragma unroll
  for (int k = 0; k < PITEMS; ++k) {
    const int64_t i = base + k * PNT;
    if (paired[k] && at[k] < cap) {
      dms_pair p;
      if (dim == 0) {
        const int64_t m = critA[T.s[i].res];
        const int64_t id = critB[i];
        const int64_t a = id / 7;
        const int kk = (int)(id - a * 7);
        const dms_field_desc fd = ft.fd[field_of_vertex(ft, a)];
        const Grid g = grid_of(fd);
        int64_t v[2] = {a, a + corner_delta(g, edge_corner(kk))};
        const int64_t top = top_of(Dev{}, order, v, 2);
        p.birth_id = m - fd.offset;
        p.death_id = id - 7 * fd.offset;
        p.birth = __ldg(f + m);
        p.death = __ldg(f + top);
        p.birth_vtx = (uint32_t)(m - fd.offset);
        p.death_vtx = (uint32_t)(top - fd.offset);
      } else {
        const int64_t tet = critB[T.s[i].res - 1];
        const int64_t tri = critA[i];
        const int64_t a = tri / 12;
        const int kk = (int)(tri - a * 12);
        const dms_field_desc fd = ft.fd[field_of_vertex(ft, a)];
        const Grid g = grid_of(fd);
        int64_t tv[3] = {a, a + corner_delta(g, tri_p(kk)), a + corner_delta(g, tri_q(kk))};
        const int64_t b = tet / 6;
        const int kq = (int)(tet - b * 6);
        int64_t qv[4] = {b, b + corner_delta(g, tet_c1(kq)), b + corner_delta(g, tet_c2(kq)),
                         b + corner_delta(g, 7)};
        const int64_t st = top_of(Dev{}, order, tv, 3), qt = top_of(Dev{}, order, qv, 4);
        p.birth_id = tri - 12 * fd.offset;
        p.death_id = tet - 6 * fd.offset;
        p.birth = __ldg(f + st);
        p.death = __ldg(f + qt);
        p.birth_vtx = (uint32_t)(st - fd.offset);
        p.death_vtx = (uint32_t)(qt - fd.offset);
      }
      out[at[k]] = p;
    }
  }
}

}  // namespace

// rounds of one launch per phase ahead of pair_rounds, which takes whatever is
// live then: on noise and on mixtures the live saddles fell to a third or less
// per round, so that six leave a thousandth
constexpr unsigned int kBatchLarge = 6;
int diagram_batch_rounds() { return (int)kMaxExactRounds; }

// Workspace of the batched pairing: the DiagWs of the capacities plus the
// per-field counters and pair-tile sums.
size_t diagram_batch_workspace_bytes(int64_t nfields, const int64_t* caps, int64_t total) {
  WsCarver c(nullptr);
  c.take<unsigned char>(carve_diag(nullptr, caps, 6 * total).bytes);
  const int64_t nsad = std::max<int64_t>(std::max<int64_t>(caps[1], caps[2]), 1);
  c.take<unsigned long long>(2 * (nfields + 1));
  c.take<unsigned long long>(look_words(nsad));
  c.take<int64_t>(nfields + 1);
  return c.used;
}

int launch_diagram_batch(const float* f, const uint32_t* order, const uint8_t* desc,
                         const uint64_t* rec, const dms_field_desc* fields_host,
                         const dms_field_desc* fields_dev, int nfields, int64_t total_vertices, int64_t* const crit[4], const int64_t* cnt_dev,
                         const int64_t* caps, dms_pair* d0, dms_pair* d2, int64_t cap_pairs,
                         int64_t* pair_offsets, dms_pair* ess, int64_t* pair_totals, void* ws,
                         int32_t* dstatus, cudaStream_t s) {
  WsCarver c(ws);
  unsigned char* dbase = c.take<unsigned char>(carve_diag(nullptr, caps, 6 * total_vertices).bytes);
  DiagWs w = carve_diag(dbase, caps, 6 * total_vertices);
  const int64_t nsad = std::max<int64_t>(std::max<int64_t>(caps[1], caps[2]), 1);
  unsigned long long* fcount = c.take<unsigned long long>(2 * (nfields + 1));
  unsigned long long* look = c.take<unsigned long long>(look_words(nsad));
  int64_t* brick0 = c.take<int64_t>(nfields + 1);
  const FieldTab ft{fields_dev, nfields};
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned G = (unsigned)sms * 8, TB = 256;  // grid-stride launches
  DMS_CUDA_OK(cudaMemsetAsync(fcount, 0, 2 * (nfields + 1) * sizeof(unsigned long long), s));

  // the spanning forest and the exact rounds on its saddles, as in the
  // single-field path, the node count (ncnt + extra) read on the device
  const bool large = nsad > kOneLaunch;
  auto rounds = [&](Tri T, const int64_t* ncnt, int64_t extra) -> int {
    // kBatchLarge rounds of one launch per phase (they do nothing on an empty
    // list), the rest in one launch
    uint32_t *cur = w.live0, *nxt = w.live1;
    unsigned int *cur_n = w.ctr + kCtrLive, *nxt_n = w.ctr + kCtrNext;
    bool mem_ok = true;
    unsigned int round = 1;
    for (; large && round <= kBatchLarge; ++round) {
      mem_ok = mem_ok && cudaMemsetAsync(nxt_n, 0, sizeof(unsigned int), s) == cudaSuccess;
      if (round > 1) {  // link_d0 / link_d2 did round 1's search
        round_find<<<G, TB, 0, s>>>(cur, cur_n, T, w.nd, round); count_launch();
      }
      boruvka_hook<<<G, TB, 0, s>>>(cur, cur_n, T, w.nd, round, nxt, nxt_n, w.forest,
                                    w.ctr + kCtrForest); count_launch();
      std::swap(cur, nxt);
      std::swap(cur_n, nxt_n);
    }
    Rounds r;
    r.T = T;
    r.nd = w.nd;
    r.cur = cur;
    r.nxt = nxt;
    r.n = cur_n;
    r.round = round;
    r.forest = w.forest;
    r.forest_only = large;
    r.first_found = round == 1;
    r.left = w.live1;
    r.ctr = w.ctr;
    r.n_dev = ncnt;
    r.nnode = extra;
    DMS_TRY(launch_rounds(r, nsad, dstatus, s));
    if (large) {
      reset_nodes<<<G, TB, 0, s>>>(w.nd, ncnt, extra); count_launch();
      mem_ok = mem_ok && cudaMemsetAsync(w.ctr + kCtrRound, 0, (kCtrWords - kCtrRound) * sizeof(unsigned int),
                                         s) == cudaSuccess;
      cur = w.forest;
      cur_n = w.ctr + kCtrForest;
      nxt = w.live0;
      nxt_n = w.ctr + kCtrLive;
      for (round = 1; round <= kBatchLarge; ++round) {
        mem_ok = mem_ok && cudaMemsetAsync(nxt_n, 0, sizeof(unsigned int), s) == cudaSuccess;
        round_find<<<G, TB, 0, s>>>(cur, cur_n, T, w.nd, round); count_launch();
        round_merge<<<G, TB, 0, s>>>(cur, cur_n, T, w.nd, round, nxt, nxt_n); count_launch();
        std::swap(cur, nxt);
        std::swap(cur_n, nxt_n);
      }
      r.cur = cur;
      r.nxt = nxt;
      r.n = cur_n;
      r.round = round;
      r.forest = nullptr;
      r.forest_only = r.first_found = false;
      DMS_TRY(launch_rounds(r, nsad, dstatus, s));
    }
    if (!mem_ok) return DMS_ERR_CUDA;
    const unsigned int* left_n = w.ctr + kCtrLeft;
    b_finish<<<1, 1024, 0, s>>>(w.live1, left_n, T, w.nd, dstatus); count_launch();
    // more than the one-CTA finish holds: sort them by weight on the device
    // and finish them in that order (one thread; nothing runs when the
    // count is small)
    unsigned int* big_n = w.ctr + kCtrBig;
    b_big_count<<<1, 32, 0, s>>>(left_n, big_n); count_launch();
    gather_live<<<G, TB, 0, s>>>(w.live1, big_n, T, w.rb.ka, w.rb.va); count_launch();
    const bool in_a = radix64::sort(w.rb, nsad, 44, s, big_n);
    sequential_finish<<<1, 32, 0, s>>>(in_a ? w.rb.va : w.rb.vb, big_n, T, w.nd); count_launch();
    return DMS_OK;
  };
  auto write = [&](int dim, Tri T, const int64_t* critA, const int64_t* critB, const int64_t* n_dev,
                   dms_pair* out, int64_t* offs, int64_t* total, unsigned long long* fc) -> int {
    DMS_CUDA_OK(cudaMemsetAsync(look, 0, look_words(nsad) * sizeof(*look), s));
    b_write_pairs<<<(unsigned)(look_words(nsad) - 1), PNT, 0, s>>>(dim, ft, f, order, critA, critB, T,
                                                                   n_dev, look, out, cap_pairs,
                                                                   dstatus); count_launch();
    b_count_fields<<<G, TB, 0, s>>>(ft, T, dim == 0 ? critB : critA, n_dev, dim == 0 ? 7 : 12, fc); count_launch();
    b_field_offsets<<<1, 32, 0, s>>>(fc, nfields, offs, total, cap_pairs, dstatus); count_launch();
    return DMS_OK;
  };

  // ---- D0
  DMS_CUDA_OK(cudaMemsetAsync(w.ctr, 0, kCtrWords * sizeof(unsigned int), s));
  b_init_nodes_d0<<<G, TB, 0, s>>>(order, crit[0], cnt_dev, w.nd); count_launch();
  b_essential<<<G, TB, 0, s>>>(ft, f, order, crit[0], cnt_dev, ess); count_launch();
  using Desc = DescPaths<ManyFields>;
  using Dual = DualPaths<ManyFields>;
  int64_t bricks0 = 0, bricks2 = 0;
  for (int i = 0; i < nfields; ++i) {
    bricks0 += brick_count<Desc>(fields_host[i].nx, fields_host[i].ny, fields_host[i].nz);
    bricks2 += brick_count<Dual>(fields_host[i].nx, fields_host[i].ny, fields_host[i].nz);
  }
  const ManyFields mf{fields_dev, nfields, brick0};
  brick_table<<<1, 32, 0, s>>>(ft, Desc::LX, Desc::LY, Desc::LZ, brick0); count_launch();
  mark_ends<<<G, TB, 0, s>>>(crit[0], cnt_dev + 0, 0, 0, w.path); count_launch();
  resolve_paths<<<(unsigned)bricks0, kBrickThreads, 0, s>>>(Desc{mf, desc, crit[0], cnt_dev + 0, 0}, w.path); count_launch();
  w.nd.immortal = kNone;
  link_d0<kBricks, Desc><<<G, TB, 0, s>>>(Desc{mf, desc, crit[0], cnt_dev + 0, 0}, order, crit[1], cnt_dev + 1,
                                          0, w.path, w.T0, w.live0, w.ctr + kCtrLive, nullptr, nullptr, nullptr,
                                          dstatus, true, w.nd); count_launch();
  DMS_TRY(rounds(w.T0, cnt_dev + 0, 0));
  DMS_TRY(write(0, w.T0, crit[0], crit[1], cnt_dev + 1, d0, pair_offsets, pair_totals + 0, fcount));

  // ---- D2
  DMS_CUDA_OK(cudaMemsetAsync(w.ctr, 0, kCtrWords * sizeof(unsigned int), s));
  b_init_nodes_d2<<<G, TB, 0, s>>>(ft, order, crit[3], cnt_dev, w.nd); count_launch();
  mark_ends<<<G, TB, 0, s>>>(crit[3], cnt_dev + 3, 0, 1, w.path); count_launch();
  brick_table<<<1, 32, 0, s>>>(ft, Dual::LX, Dual::LY, Dual::LZ, brick0); count_launch();
  resolve_paths<<<(unsigned)bricks2, kBrickThreads, 0, s>>>(Dual{mf, rec, crit[3], cnt_dev + 3, 0}, w.path); count_launch();
  w.nd.immortal = 0;  // OUTSIDE, shared by all fields
  link_d2<kBricks, Dual><<<G, TB, 0, s>>>(Dual{mf, rec, crit[3], cnt_dev + 3, 0}, order, crit[2], cnt_dev + 2,
                                          0, w.path, w.T2, w.live0, w.ctr + kCtrLive, nullptr, nullptr, nullptr,
                                          dstatus, true, w.nd); count_launch();
  DMS_TRY(rounds(w.T2, cnt_dev + 3, 1));
  DMS_TRY(write(2, w.T2, crit[2], crit[3], cnt_dev + 2, d2, pair_offsets + (nfields + 1), pair_totals + 1,
                fcount + (nfields + 1)));
  return launch_status();
}

}  // namespace dms

// ===========================================================================
// 2D grids: D0 (minima against saddle edges) and D1 (saddle edges against
// maxima, on the dual graph of triangles plus OUTSIDE) -- the same walks,
// links and rounds as in 3D, one dimension down.
//
// 2D conventions (include/dms.h): vertex v = x + nx*y; edge 3a+k, corner
// {1,2,3}[k] (+x, +y, +x+y); triangle 2a+k = {a, a+p, a+(1,1)}, p = {+x,
// +y}[k].  A vertex's six neighbour slots: s < 3 -> +corner, s >= 3 ->
// -corner of edge type s % 3.  rec2[a] (uint16): bits 3k..3k+2 edge k (0 =
// absent or paired with its top vertex, 1..2 = paired with the (code-1)-th
// triangle holding it by increasing id on the unbounded lattice, 7 =
// critical); bits 9+3k..11+3k triangle k (0 = absent, 1..3 = paired with the
// facet that omits vertex (code-1) of its chain a < a+p < a+(1,1), 7 =
// critical).
// ===========================================================================
namespace dms {
namespace {

struct Grid2d {
  int64_t nx, ny, n;
};

__device__ __forceinline__ int64_t cdelta2(const Grid2d& g, int c) {
  return (c & 1) + ((c >> 1) & 1) * g.nx;
}
__device__ __forceinline__ int64_t slot_delta2(const Grid2d& g, int s) {
  const int64_t d = cdelta2(g, corner2(s));
  return s < 3 ? d : -d;
}
__device__ __forceinline__ void xy2(const Grid2d& g, int64_t v, int64_t& x, int64_t& y) {
  const uint32_t u = (uint32_t)v, nx = (uint32_t)g.nx;
  y = u / nx;
  x = u - (uint32_t)y * nx;
}
// the square anchored at (x, y) exists
__device__ __forceinline__ bool square2(const Grid2d& g, int64_t x, int64_t y) {
  return x >= 0 && y >= 0 && x + 1 < g.nx && y + 1 < g.ny;
}

// rank of neighbour order ou among the lower neighbours of vertex t
__device__ __forceinline__ uint32_t local_rank2d(const Grid2d& g, const uint32_t* __restrict__ order,
                                                 int64_t t, uint32_t ou) {
  int64_t x, y;
  xy2(g, t, x, y);
  uint32_t r = 0;
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const int c = corner2(s), sg = s < 3 ? 1 : -1;
    const int64_t nx = x + sg * (c & 1), ny = y + sg * ((c >> 1) & 1);
    if (nx < 0 || ny < 0 || nx >= g.nx || ny >= g.ny) continue;
    r += __ldg(order + t + slot_delta2(g, s)) < ou ? 1u : 0u;
  }
  return r;
}

// node 0 = OUTSIDE (age 0, the oldest); node j + 1 = maximum crit2[j], a
// higher one older
__global__ void init_nodes_d1_2d(Grid2d g, const uint32_t* __restrict__ order,
                                 const int64_t* __restrict__ crit2, int64_t nmax, Nodes nd) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i > nmax) return;
  nd.parent[i] = (uint32_t)i;
  nd.best[i] = 0ull;
  if (i == 0) {
    nd.age[0] = 0;
    return;
  }
  const int64_t id = crit2[i - 1];
  const int64_t a = id / 2;
  const int k = (int)(id - a * 2);
  const int64_t v[3] = {a, a + cdelta2(g, k + 1), a + cdelta2(g, 3)};
  uint32_t o[3];
  int it = 0;
  for (int j = 0; j < 3; ++j) {
    o[j] = __ldg(order + v[j]);
    if (o[j] > o[it]) it = j;
  }
  uint32_t r[2];
  int n = 0;
  for (int j = 0; j < 3; ++j)
    if (j != it) r[n++] = local_rank2d(g, order, v[it], o[j]);
  const uint32_t h = max(r[0], r[1]), l = min(r[0], r[1]);
  const uint64_t key = ((uint64_t)o[it] << 8) | (h << 4) | l;
  nd.age[i] = (kMask44 - key) + 1;
}

__host__ __device__ __forceinline__ Grid grid_of2d(const Grid2d& g) { return Grid{g.nx, g.ny, 1, g.n, g.n}; }

// D0: each critical edge's weight, its two descending paths
__global__ void __launch_bounds__(256) link2d_d0(Grid2d g, const uint32_t* __restrict__ order,
                                                 const int64_t* __restrict__ crit1, int64_t ne,
                                                 const uint32_t* __restrict__ path, Tri T,
                                                 uint32_t* live, unsigned int* live_n,
                                                 int32_t* dstatus, Nodes nd) {
  __shared__ CtaAppend sh;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool keep = false;
  if (i < ne) {
    const int64_t id = crit1[i], a = id / 3;
    const int c = (int)(id - a * 3) + 1;
    const int64_t b = a + cdelta2(g, c);
    const Grid g3 = grid_of2d(g);
    int64_t x, y;
    xy2(g, a, x, y);
    Walk wa = walk_from<DescPaths2d>(path, g3, a, (int)x, (int)y, 0, 0);
    Walk wb = walk_from<DescPaths2d>(path, g3, b, (int)x + (c & 1), (int)y + ((c >> 1) & 1), 0, 0);
    const uint32_t oa = __ldg(order + a), ob = __ldg(order + b);
    const uint64_t w = ((uint64_t)(oa > ob ? oa : ob) << 4) |
                       local_rank2d(g, order, oa > ob ? a : b, oa > ob ? ob : oa);
    walk_both<DescPaths2d>(path, g3, 0, wa, wb);
    keep = store_saddle(T, i, w, walk_end(wa.w, dstatus), walk_end(wb.w, dstatus), false, nd);
  }
  cta_append2(sh, keep, live, live_n, false, live, live_n, (uint32_t)i);
}

// D1: saddles are visited by decreasing edge key (D0's weight, complemented),
// two dual paths each.  On a 2D grid (a disk, no 1-cycles survive) every
// critical edge is either a D0 death or a D1 birth: the edges that D0 paired
// take no part.
__global__ void __launch_bounds__(256) link2d_d1(Grid2d g, const int64_t* __restrict__ crit1, int64_t ne,
                                                 const uint32_t* __restrict__ path, Tri T,
                                                 uint32_t* live, unsigned int* live_n,
                                                 int32_t* dstatus, Nodes nd) {
  __shared__ CtaAppend sh;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool keep = false;
  if (i < ne) {
    if (T.s[i].res != kNone) {
      T.s[i].res = kNone;
    } else {
      const int64_t id = crit1[i], a = id / 3;
      const int t = (int)(id - a * 3);
      const Grid g3 = grid_of2d(g);
      int64_t ax, ay;
      xy2(g, a, ax, ay);
      Walk wk[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        // triangle j of the edge: the diagonal's are both in the square at a;
        // a horizontal edge's: type 0 above, type 1 below; a vertical edge's:
        // type 1 to the right, type 0 to the left
        const int64_t bx = ax - (j == 1 && t == 1), by = ay - (j == 1 && t == 0);
        const int k = t == 2 ? j : (j == 0 ? t : 1 - t);
        wk[j] = square2(g, bx, by) ? walk_from<DualPaths2d>(path, g3, bx + g.nx * by, (int)bx, (int)by, 0, k)
                                   : Walk{kEnd, 0, 0, 0};
      }
      walk_both<DualPaths2d>(path, g3, 0, wk[0], wk[1]);
      keep = store_saddle(T, i, kMask44 - T.s[i].w, walk_end(wk[0].w, dstatus), walk_end(wk[1].w, dstatus),
                          false, nd);
    }
  }
  cta_append2(sh, keep, live, live_n, false, live, live_n, (uint32_t)i);
}

__device__ __forceinline__ int64_t top2(const uint32_t* order, const int64_t* v, int m) {
  int64_t best = v[0];
  uint32_t ob = __ldg(order + v[0]);
  for (int j = 1; j < m; ++j) {
    const uint32_t o = __ldg(order + v[j]);
    if (o > ob) {
      ob = o;
      best = v[j];
    }
  }
  return best;
}

// dim 0: (minimum, edge); dim 1: (edge, triangle) -- in saddle-id order
__global__ void __launch_bounds__(PNT) write_pairs2d(int dim, Grid2d g, const float* __restrict__ f,
                                                     const uint32_t* __restrict__ order,
                                                     const int64_t* __restrict__ nodes,
                                                     const int64_t* __restrict__ crit1, const Tri T,
                                                     int64_t nsad, unsigned long long* look,
                                                     dms_pair* out, int64_t cap, int64_t* n_out,
                                                     int32_t* dstatus) {
  __shared__ PairSmem sm;
  const int64_t tile = take_tile(sm, look), base = tile * PTILE + threadIdx.x;
  bool paired[PITEMS];
  int64_t at[PITEMS];
#pragma unroll
  for (int k = 0; k < PITEMS; ++k)
    paired[k] = base + k * PNT < nsad && T.s[base + k * PNT].res != kNone;
  place_pairs(sm, look, tile, paired, at, dstatus);
  if (tile == gridDim.x - 1 && threadIdx.x == 0) {
    const int64_t total = sm.before + sm.total;
    *n_out = total;
    if (total > cap) set_status(dstatus, DMS_ERR_CAPACITY);
  }
#pragma unroll
  for (int k = 0; k < PITEMS; ++k) {
    const int64_t i = base + k * PNT;
    if (paired[k] && at[k] < cap) {
      const int64_t e = crit1[i];
      const int64_t a = e / 3;
      const int64_t ev[2] = {a, a + cdelta2(g, (int)(e - a * 3) + 1)};
      const int64_t et = top2(order, ev, 2);
      dms_pair p;
      if (dim == 0) {
        const int64_t m = nodes[T.s[i].res];
        p.birth_id = m;
        p.death_id = e;
        p.birth = __ldg(f + m);
        p.death = __ldg(f + et);
        p.birth_vtx = (uint32_t)m;
        p.death_vtx = (uint32_t)et;
      } else {
        const int64_t tri = nodes[T.s[i].res - 1];  // node 0 (OUTSIDE) never dies
        const int64_t b = tri / 2;
        const int64_t tv[3] = {b, b + cdelta2(g, (int)(tri - b * 2) + 1), b + cdelta2(g, 3)};
        const int64_t tt = top2(order, tv, 3);
        p.birth_id = e;
        p.death_id = tri;
        p.birth = __ldg(f + et);
        p.death = __ldg(f + tt);
        p.birth_vtx = (uint32_t)et;
        p.death_vtx = (uint32_t)tt;
      }
      out[at[k]] = p;
    }
  }
}

}  // namespace

size_t diagram2d_workspace_bytes(int64_t n, const int64_t* nc) {
  const int64_t nc4[4] = {nc[0], nc[1], nc[1], nc[2]};
  return carve_diag(nullptr, nc4, 2 * n).bytes;
}

int launch_diagram2d(const float* f, const uint32_t* order, const uint8_t* desc, const uint16_t* rec,
                     int64_t nx, int64_t ny, const int64_t* crit0, const int64_t* crit1,
                     const int64_t* crit2, const int64_t* nc, dms_pair* d0, int64_t cap0,
                     dms_pair* d1, int64_t cap1, dms_pair* ess, int64_t* n_out, void* ws,
                     int32_t* dstatus, cudaStream_t s) {
  const Grid2d g{nx, ny, nx * ny};
  const int64_t nc4[4] = {nc[0], nc[1], nc[1], nc[2]};
  DiagWs w = carve_diag(ws, nc4, 2 * g.n);
  const int TB = 256;
  auto nb = [&](int64_t n) { return (unsigned)std::max<int64_t>(1, (n + TB - 1) / TB); };
  const int64_t ne = nc[1];
  auto write = [&](int dim, const int64_t* nodes, dms_pair* out, int64_t cap,
                   int64_t* nout) -> int {
    if (ne <= 0)
      return cudaMemsetAsync(nout, 0, sizeof(int64_t), s) == cudaSuccess ? DMS_OK : DMS_ERR_CUDA;
    unsigned long long* look = w.rb.ka;
    DMS_CUDA_OK(cudaMemsetAsync(look, 0, look_words(ne) * sizeof(*look), s));
    write_pairs2d<<<(unsigned)(look_words(ne) - 1), PNT, 0, s>>>(dim, g, f, order, nodes, crit1, w.T0, ne,
                                                                 look, out, cap, nout, dstatus); count_launch();
    return launch_status();
  };

  // ---- D0
  DMS_CUDA_OK(cudaMemsetAsync(w.ctr, 0, kCtrWords * sizeof(unsigned int), s));
  init_nodes_d0<<<nb(nc[0]), TB, 0, s>>>(order, crit0, nc[0], w.nd); count_launch();
  write_essential<<<nb(nc[0]), TB, 0, s>>>(f, order, crit0, nc[0], ess); count_launch();
  if (ne > 0) {
    mark_ends<<<nb(nc[0]), TB, 0, s>>>(crit0, nullptr, nc[0], 0, w.path); count_launch();
    resolve_paths<<<(unsigned)brick_count<DescPaths2d>(nx, ny, 1), kBrickThreads, 0, s>>>(
        DescPaths2d{OneField{grid_of2d(g)}, desc, crit0, nc[0]}, w.path); count_launch();
    link2d_d0<<<nb(ne), TB, 0, s>>>(g, order, crit1, ne, w.path, w.T0, w.live0, w.ctr + kCtrLive, dstatus,
                                    w.nd); count_launch();
  }
  w.nd.immortal = kNone;
  int st = run_pairing(w, w.T0, ne, nc[0], s, dstatus, false);
  if (st) return st;
  st = write(0, crit0, d0, cap0, n_out + 0);
  if (st) return st;

  // ---- D1
  DMS_CUDA_OK(cudaMemsetAsync(w.ctr, 0, kCtrWords * sizeof(unsigned int), s));
  init_nodes_d1_2d<<<nb(nc[2] + 1), TB, 0, s>>>(g, order, crit2, nc[2], w.nd); count_launch();
  if (ne > 0) {
    if (nc[2] > 0) {
      mark_ends<<<nb(nc[2]), TB, 0, s>>>(crit2, nullptr, nc[2], 1, w.path); count_launch();
    }
    resolve_paths<<<(unsigned)brick_count<DualPaths2d>(nx, ny, 1), kBrickThreads, 0, s>>>(
        DualPaths2d{OneField{grid_of2d(g)}, rec, crit2, nc[2]}, w.path); count_launch();
    link2d_d1<<<nb(ne), TB, 0, s>>>(g, crit1, ne, w.path, w.T0, w.live0, w.ctr + kCtrLive, dstatus,
                                    w.nd); count_launch();
  }
  w.nd.immortal = 0;  // OUTSIDE
  st = run_pairing(w, w.T0, ne, nc[2] + 1, s, dstatus, false);
  if (st) return st;
  st = write(1, crit2, d1, cap1, n_out + 1);
  if (st) return st;
  return launch_status();
}

}  // namespace dms
