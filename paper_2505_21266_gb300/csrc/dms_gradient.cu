// Robins et al.'s lower-star discrete gradient (Sec. 2.3) on the Freudenthal
// triangulation of a 3D grid -- the first and most time-consuming step of DMS.
//
// dms_lowerstar.cuh gives ProcessLowerStars as a rule per edge of the grid
// (its pair and the pairs of the tets whose two highest vertices are the
// edge's ends, from the 4 or 6 orders around the edge) and a correction of
// the vertices whose lower link is not a disk built arc by arc.  The rule
// costs the same everywhere, so it runs for all anchors with full warps; the
// vertices to correct are gathered in a list per slab, so that the correction,
// whose length varies, runs with full warps as well.
//
// Work layout: a CTA owns a TX x TY x ZC block of ANCHORS and streams it along
// z.  Per slab z, in two phases of tasks of 32 that the warps draw from a
// counter (corrections differ in length), over what of the tile lies in the
// grid (over whole tiles, grids thin in x or y paid for the rest: 4096 x 2 x
// 4096 smooth 9.7 ms, now 3.1; 4096 x 4096 x 2 13.6, now 6.7):
//   1. every vertex of the slab reads the kinds of the 14 edges whose higher
//      end it may be: desc, or an entry in one of four lists by how long its
//      correction takes; the records two slabs down, final by now, are written
//      out; the order window two slabs up is completed;
//   2. the listed vertices are corrected, on the records in shared memory;
//      the rule for the 7 edges of every anchor of the next slab (a halo of
//      one on both sides in x and y): edge and tet codes go to the records
//      (tets by OR: around an edge lie up to four anchors), kinds to a word
//      per anchor.
// Simplices are decided in the lower star of their highest vertex, which lies
// in anchor + {0,1}^3; the records of the last three slabs are kept.  A
// slab's corrections and the next slab's rule change different bits of the
// records, so they need no barrier between them.
//
// What bounds it: instruction issue, the integer (ALU) pipe above all, and on
// noise the correction's code in the instruction cache.  The rule takes 370
// lane-instructions per vertex with its halo; its sums of positions are
// predicated multiply-adds so that they leave the ALU pipe to the comparisons.
// Every part has one call site and the correction's loops stay rolled: with
// the correction inlined four times and its loops unrolled by the compiler a
// 512^3 noise field took 37 ms instead of 17.  The correction's lanes advance
// in step (any_lane); left to diverge in nested loops it took 75 ms.
// Measured (GB300): 1024^3 mixture with noise 124 -> 90 ms, 512^3 quantised
// noise 17.8 -> 16.9 ms, 64^3 and 24^3 mixtures 0.28 -> 0.11 and 0.19 -> 0.06
// ms, against ProcessLowerStars run queue by queue with one thread per vertex.
// It is slower than that on noise in grids of fewer than 24 vertices in x, or
// 9 to 16 in y, whose slabs have too few vertices for a CTA's warps: 2048 x
// 2048 x 8 11.2 against 9.1 ms, 1024 x 1024 x 16 3.8 against 3.1.
#include <algorithm>
#include <cstdint>
#include <cstring>

#include <cuda.h>  // CUtensorMap (the encoder is fetched from the driver at run time)

#include "dms_common.cuh"
#include "dms_lowerstar.cuh"
#include "dms_star.cuh"

namespace dms {
namespace {

constexpr int TX = 32;

// (device memory, not constant: the CTAs copy it with an index per lane)
__device__ const lowerstar::Tables cTables = lowerstar::make_tables();

using lowerstar::kCyc;
using lowerstar::static_for;

constexpr uint64_t kEdgeLsb = 0x49249ull;      // bits 0,3,..,18
constexpr uint64_t kTriMask = 0xFFFull << 21;  // bits 21..32
constexpr uint64_t kTetLsb = 0x9249ull << 33;  // bits 33,36,..,48

// threads of a CTA and CTAs of an SM
constexpr int threads_of(int ty) { return ty == 8 ? 256 : (ty == 16 ? 256 : (ty == 24 ? 384 : 512)); }
constexpr int ctas_of(int ty) { return ty == 24 ? 3 : (ty == 32 ? 2 : 4); }

// Grids up to kSmallGrid vertices are tiled TX x kSmallTY, in chunks of as few
// slabs as fill the GPU once: there a CTA's slabs, one after the other (10-15
// us each where corrections are many), are the time.  24^3 and 64^3 mixtures:
// 51 and 107 us against 392 and 832 us in tiles of 24 rows and chunks of 32
// slabs; above the line the taller tile's smaller halo wins (203 x 131 x 77
// noise, 2.0 M vertices: 434 us against 551 us).  Grids of up to kSmallTY rows
// take these tiles at any size, which they fill (2048 x 8 x 2048 noise 6.4 ms,
// in tiles of 24 rows 8.5; from 9 rows on the tall tile is faster: 300 x 10 x
// 1500 noise 1.19 against 1.56 ms).
constexpr int kSmallTY = 8;
constexpr int64_t kSmallGrid = (int64_t)1 << 20;

// parts of an anchor's edges worked by different threads: all seven types,
// or the three axis types and the four diagonal ones (18 orders compared each)
template <int PARTS>
constexpr int part_of_type(int t) {
  return PARTS == 1 ? 0 : (t < 3 ? 0 : 1);
}

// rows of equal length, numbered through: row of number i < 1156 of at most 34
// columns ((i * inv) >> 16 is exact for i * cols < 2^16)
struct Rows {
  int cols, rows, n, inv;
  Rows() = default;
  __device__ __forceinline__ Rows(int c, int r) : cols(c), rows(r), n(c * r), inv(65536 / c + 1) {}
  __device__ __forceinline__ int row(int i) const { return (i * inv) >> 16; }
};

// shared memory of a CTA working on tiles of TX x TY anchors.  The order
// field is staged slab by slab in windows of WY rows x WX columns: with TMA
// (TMA = true) a ring of five windows whose rows start at x0 - 4 (a
// 16-byte-aligned start: x0 is a multiple of 32) and are TX + 8 wide, else
// a ring of four windows starting at x0 - 2, TX + 4 wide.  Column XOFF + lx,
// row 2 + ly of a window hold grid (x0 + lx, y0 + ly).  Record words and
// kinds are kept for anchors from -2 (records) or -1 (kinds) to TX, TY.
template <int TY, bool TMA = false, int PARTS = 1>
struct Smem {
  static constexpr int NT = threads_of(TY), P = PARTS;
  static constexpr int part_of(int t) { return part_of_type<PARTS>(t); }
  static constexpr int WY = TY + 4;
  static constexpr int WX = TMA ? TX + 8 : TX + 4;
  static constexpr int XOFF = TMA ? 4 : 2;
  static constexpr int NSLAB = TMA ? 5 : 4;
  static constexpr int SLAB = (WY * WX + 31) / 32 * 32;  // words; a multiple of 128 bytes
  static constexpr int RX = TX + 3, RN = RX * (TY + 3);  // record words of a slab
  static constexpr int FX = TX + 2, FN = FX * (TY + 2);  // kind words of a slab
  lowerstar::Tables tb;
  alignas(128) uint32_t win[NSLAB][SLAB];
  unsigned long long bar[NSLAB];  // TMA: one mbarrier per window
  uint32_t lo[PARTS][3][RN];  // record bits 0..31 (edge codes by part) of slab z in [z % 3]
  uint32_t hi[3][RN];         // record bits 32..63
  uint32_t kinds[PARTS][3][FN];
  // the vertices to correct, by how long it takes: class 0 no kArcs or kWhole
  // edge, 1 one kArcs edge, 2 more, 3 with kWhole edges; list[class >> 1] from
  // the front (even) or the back (odd)
  static constexpr int VN = (TX + 1) * (TY + 1);
  uint16_t list[2][VN];
  // where the correction finds things, relative to the vertex: by window slot
  // of the slab, slot s's order and those of its cycle (position n and on:
  // slot s itself); by record slab, slot s's edge, the star tets and triangles
  // (word offset x 32 + bit)
  int16_t oAt[NSLAB][14], cAt[NSLAB][14][8];
  int eAt[3][14], qAt[3][24], jAt[3][36];
  alignas(16) unsigned int nlist[2][4];  // their lengths, for slab j in [j & 1]
  unsigned int task[2];      // the next task of the two phases
  unsigned int counts[4];
  uint32_t one;    // the number 1 (see add_if_less)
  Rows verts, anchors;  // what of the tile lies in the grid
  long long tile;  // batched kernel: the tile this CTA works on
};

template <int TY, int PARTS>
__device__ __forceinline__ void load_slab(Smem<TY, false, PARTS>& sm,
                                          const uint32_t* __restrict__ order, const Grid& g, int x0,
                                          int y0, int64_t zs, int slot) {
  using S = Smem<TY, false, PARTS>;
  const bool none = zs < 0 || zs >= g.nz;
  const uint32_t* slab = order + (none ? 0 : g.sxy * zs);
#pragma unroll 1
  for (int i = threadIdx.x; i < S::WX * S::WY; i += S::NT) {
    const int gx = x0 - S::XOFF + i % S::WX, gy = y0 - 2 + i / S::WX;
    uint32_t v = 0xFFFFFFFFu;
    if (!none && (uint32_t)gx < (uint32_t)g.nx && (uint32_t)gy < (uint32_t)g.ny)
      v = __ldg(slab + ((uint32_t)gx + (uint32_t)g.nx * (uint32_t)gy));
    sm.win[slot][i] = v;
  }
}

// ---- TMA staging (one field; its order array viewed as an nx x ny x nz
// tensor of u32) ----------------------------------------------------------
// A window is one box of WX x WY x 1 at (x0 - 4, y0 - 2, zs): loads may start
// outside the grid (only x has to be 16-byte aligned), and TMA fills what
// lies outside with zeros, which the border windows then overwrite with
// 0xFFFFFFFF (never lower).  Each window has an mbarrier; thread 0 arms it
// with the box's byte count and issues the copy, and every thread waits on
// its phase, at most kTmaWaitLimit polls (a copy that never lands marks the
// call failed and the CTA stops, see gradient_kernel).
constexpr uint32_t kTmaWaitLimit = 1u << 22;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

template <class S>
__device__ __forceinline__ void tma_init(S& sm) {
  if (threadIdx.x == 0) {
    for (int b = 0; b < S::NSLAB; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&sm.bar[b])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

// thread 0 only; the window's previous contents were last read before a
// __syncthreads that the caller passed
template <class S>
__device__ __forceinline__ void tma_issue(S& sm, const CUtensorMap* tm, int b, int x0, int y0,
                                          int64_t zs) {
  constexpr uint32_t kBytes = S::WX * S::WY * 4;
  const uint32_t bar = smem_u32(&sm.bar[b]), dst = smem_u32(sm.win[b]);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(kBytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x0 - 4), "r"(y0 - 2), "r"((int)zs), "r"(bar)
      : "memory");
}

// waits for the phase `parity` of window b; false after kTmaWaitLimit polls
template <class S>
__device__ __forceinline__ bool tma_wait(S& sm, int b, uint32_t parity) {
  const uint32_t bar = smem_u32(&sm.bar[b]);
#pragma unroll 1
  for (uint32_t it = 0; it < kTmaWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// out-of-grid entries of a window of slab zs -> never lower
template <class S>
__device__ __forceinline__ void tma_fix_border(S& sm, const Grid& g, int b, int x0, int y0, int64_t zs) {
  const bool none = zs < 0 || zs >= g.nz;
  const int nx = (int)g.nx, ny = (int)g.ny;
#pragma unroll 1
  for (int i = threadIdx.x; i < S::WX * S::WY; i += S::NT) {
    const int gx = x0 - 4 + i % S::WX, gy = y0 - 2 + i / S::WX;
    if (none || (uint32_t)gx >= (uint32_t)nx || (uint32_t)gy >= (uint32_t)ny) sm.win[b][i] = 0xFFFFFFFFu;
  }
}

// the shared tables of a CTA (the caller's __syncthreads makes them visible)
template <class S>
__device__ __forceinline__ void load_tables(S& sm) {
  static_assert(sizeof(lowerstar::Tables) % 4 == 0, "word copy");
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&cTables);
  uint32_t* dst = reinterpret_cast<uint32_t*>(&sm.tb);
  for (int i = threadIdx.x; i < (int)(sizeof(lowerstar::Tables) / 4); i += S::NT) dst[i] = __ldg(src + i);
  auto window_of = [&](int s, int b) {  // slot s from a vertex of the slab in window b
    const int up = s < 7 ? 1 : -1, c = (0x7653421 >> (4 * (s < 7 ? s : s - 7))) & 15;
    const int dz = up * ((c >> 2) & 1);
    const int at = dz < 0 ? (b ? b - 1 : S::NSLAB - 1) : (dz > 0 ? (b + 1 < S::NSLAB ? b + 1 : 0) : b);
    return at * S::SLAB + up * ((c & 1) + ((c >> 1) & 1) * S::WX);
  };
  auto record_of = [&](int c, int r) {  // the anchor at corner c below a vertex of record slab r
    return ((c >> 2) ? (r ? r - 1 : 2) : r) * S::RN - (c & 1) - ((c >> 1) & 1) * S::RX;
  };
  for (int i = threadIdx.x; i < S::NSLAB * 14 * 8; i += S::NT) {
    const int b = i / 112, s = (i / 8) % 14, k = i & 7;
    const int n = cTables.cyc[s][6];
    sm.cAt[b][s][k] = (int16_t)window_of(k < n ? cTables.cyc[s][k] : s, b);
    if (k == 0) sm.oAt[b][s] = (int16_t)window_of(s, b);
  }
  for (int i = threadIdx.x; i < 3 * 36; i += S::NT) {
    const int r = i / 36, k = i % 36;
    const int j = cTables.triAt[k];
    sm.jAt[r][k] = record_of(j >> 4, r) * 32 + ((21 + (j & 15)) & 31);
    if (k < 24) {
      const int q = cTables.tetAt[k];
      sm.qAt[r][k] = record_of(q >> 3, r) * 32 + lowerstar::kTetBit + 3 * (q & 7);
    }
    if (k < 14) {
      const int e = cTables.edgeAt[k];
      sm.eAt[r][k] = (S::part_of(e & 7) * 3 * S::RN + record_of(e >> 3, r)) * 32 + 3 * (e & 7);
    }
  }
  if (threadIdx.x < 4) sm.counts[threadIdx.x] = 0;
  if (threadIdx.x == 0) *(volatile uint32_t*)&sm.one = 1u;
}

// record bits of tets around the edge of type t, by the corner c of their
// anchor (the edge's anchor - c); 0 for corners that hold none
constexpr uint32_t tet_bits(int t, int c) {
  uint32_t m = 0;
  for (int i = 0; i < kCyc.n[t]; ++i) {
    const int q = kCyc.tet[t][i];
    if (kStar.qCorner[q] == c) m |= 7u << (lowerstar::kTetBit + 3 * kStar.qType[q]);
  }
  return m;
}
// record bits (low word, high word) of simplices that reach corner bit b
constexpr uint32_t reach_lo(int b) {
  uint32_t m = 0;
  for (int t = 0; t < 7; ++t)
    if ((kStar.corner[t] >> b) & 1) m |= 7u << (3 * t);
  for (int k = 0; k < 11; ++k)
    if ((star_detail::kTriPQ[k][1] >> b) & 1) m |= 1u << (21 + k);
  return m;
}
static_assert(star_detail::kTriPQ[11][1] == 7, "triangle type 11 and the tets span the cube");

// the slot that each edge code of slot s stands for, four bits per code (code
// 0, unpaired: 15)
constexpr uint32_t code_slots(int s) {
  uint32_t m = 15u;
  for (int i = 0; i < kCyc.n[s]; ++i)
    m |= (uint32_t)kCyc.v[s][i] << (4 * (lowerstar::cof_of(s, kCyc.v[s][i]) + 1));
  return m;
}

// whether edges of a part lie around tets anchored at the corner c below
template <int PART, int PARTS>
constexpr bool part_reaches(int c) {
  for (int t = 0; t < 7; ++t)
    if (part_of_type<PARTS>(t) == PART && tet_bits(t, c)) return true;
  return false;
}

// the facet number that each code of tet q stands for, two bits per code
constexpr uint32_t code_facets(int q) {
  uint32_t m = 0;
  for (int w = 0; w < 3; ++w) m |= (uint32_t)(w + 1) << (2 * kStar.facetCode[q][w]);
  return m;
}

// The correction's view of one vertex: record words in shared memory (their
// other bits may change under it, so all changes are atomic), orders from the
// windows.
template <class S>
struct TileStar {
  S& sm;
  int wv, rv;          // the vertex in a window, in a record slab
  int win, rz, rzm;    // the slab's window slot; the record slabs of its anchors
  __device__ __forceinline__ uint32_t o(int s) const { return (&sm.win[0][0])[wv + sm.oAt[win][s]]; }
  __device__ __forceinline__ uint32_t o(int s, int i) const {
    return (&sm.win[0][0])[wv + sm.cAt[win][s][i]];
  }
  __device__ __forceinline__ uint32_t lo_word(int part, int c) const {
    return *(volatile uint32_t*)&sm.lo[part][(c >> 2) ? rzm : rz]
                                      [rv - (c & 1) - S::RX * ((c >> 1) & 1)];
  }
  __device__ __forceinline__ uint64_t parents() const {
    uint32_t p[2] = {0, 0};
    static_for<0, 14>([&](auto I) {
      constexpr int s = decltype(I)::value, t = s % 7;
      constexpr int c = s < 7 ? 0 : kStar.corner[t], part = S::part_of(t);
      constexpr uint32_t slots = code_slots(s);
      const uint32_t w = lo_word(part, c);
      const uint32_t sh = t == 0 ? (w << 2) & 28u : (w >> (3 * t - 2)) & 28u;
      p[s >> 3] |= ((slots >> sh) & 15u) << (4 * (s & 7));
    });
    return (uint64_t)p[1] << 32 | p[0];
  }
  __device__ __forceinline__ uint64_t facets() const {
    uint32_t f[2] = {0, 0};
    static_for<0, 8>([&](auto C) {
      constexpr int c = decltype(C)::value;
      const uint32_t w = *(volatile uint32_t*)&sm.hi[(c >> 2) ? rzm : rz]
                                                    [rv - (c & 1) - S::RX * ((c >> 1) & 1)];
      static_for<0, 24>([&](auto Q) {
        constexpr int q = decltype(Q)::value;
        if constexpr (kStar.qCorner[q] == c) {
          constexpr uint32_t numbers = code_facets(q);
          constexpr int b = lowerstar::kTetBit + 3 * kStar.qType[q] - 1;
          f[q >> 4] |= ((numbers >> ((w >> b) & 14u)) & 3u) << (2 * (q & 15));
        }
      });
    });
    return (uint64_t)f[1] << 32 | f[0];
  }
  __device__ __forceinline__ void set_edge(int s, uint32_t old, uint32_t c) {
    const int e = sm.eAt[rz][s];
    atomicXor(&sm.lo[0][0][0] + rv + (e >> 5), (old ^ c) << (e & 31));
  }
  __device__ __forceinline__ void set_tet(int q, uint32_t old, uint32_t c) {
    const int e = sm.qAt[rz][q];
    atomicXor(&sm.hi[0][0] + rv + (e >> 5), (old ^ c) << (e & 31));
  }
  __device__ __forceinline__ void crit_tri(int j) {
    const int e = sm.jAt[rz][j];  // bit 21 + type: type 11 is bit 0 of the high word
    if ((e & 31) == 0) atomicOr(&sm.hi[0][0] + rv + (e >> 5), 1u);
    else atomicOr(&sm.lo[0][0][0] + rv + (e >> 5), 1u << (e & 31));
  }
};

// the kinds of 14 slots, two bits each -> the slots of one kind as a mask
__device__ __forceinline__ uint32_t slots_of(uint32_t spaced) {  // bit 2s -> bit s
  uint32_t m = spaced;
  m = (m | (m >> 1)) & 0x33333333u;
  m = (m | (m >> 2)) & 0x0F0F0F0Fu;
  m = (m | (m >> 4)) & 0x00FF00FFu;
  return (m | (m >> 8)) & 0xFFFFu;
}

// the rule for the edges of the types of one part, at anchor (lx, ly)
template <int PART, class S, int PARTS>
__device__ __forceinline__ void apply_rule(S& sm, const uint32_t* wm, const uint32_t* w0,
                                           const uint32_t* wp, int lx, int ly, int rz, int rzm,
                                           uint32_t one) {
  const int at = (ly + 2) * S::WX + lx + S::XOFF;
  const uint32_t oa = w0[at];
  uint32_t o[13];
  static_for<0, 13>([&](auto I) {
    constexpr int s = decltype(I)::value;
    constexpr int dx = kStar.off[s][0], dy = kStar.off[s][1], dz = kStar.off[s][2];
    o[s] = (dz < 0 ? wm : (dz > 0 ? wp : w0))[at + dy * S::WX + dx];
  });
  uint32_t acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  uint32_t edges = 0, kinds = 0;
  static_for<0, 7>([&](auto I) {
    constexpr int t = decltype(I)::value;
    if constexpr (part_of_type<PARTS>(t) == PART) {
      const uint32_t e = *reinterpret_cast<const uint32_t*>(
          reinterpret_cast<const unsigned char*>(sm.tb.entry + lowerstar::entry_base(t)) +
          lowerstar::edge_offset<t>(oa, o, one));
      // code and kind off the top, each added at its place, the kind's by the
      // end that is higher
      const uint32_t code = e >> lowerstar::kEdgeBit;
      const uint32_t kind = (e >> lowerstar::kKindBit) - code * 4u;
      edges += code * (1u << (3 * t));
      kinds += kind * (1u << (2 * t + (o[t] > oa ? 14 : 0)));
      static_for<0, 8>([&](auto C) {
        constexpr int c = decltype(C)::value;
        if constexpr (tet_bits(t, c) != 0) acc[c] |= e & tet_bits(t, c);
      });
    }
  });
  const int ra = (ly + 2) * S::RX + lx + 2;
  sm.lo[PART][rz][ra] = edges;
  sm.kinds[PART][rz][(ly + 1) * S::FX + lx + 1] = kinds;
  static_for<0, 8>([&](auto C) {
    constexpr int c = decltype(C)::value;
    constexpr int back = (c & 1) + S::RX * ((c >> 1) & 1);
    if constexpr (part_reaches<PART, PARTS>(c))
      atomicOr(&sm.hi[(c >> 2) ? rzm : rz][ra - back], acc[c]);
  });
}

// the kinds of the 14 edges of vertex (lx, ly) where it is the higher end,
// two bits per slot
template <class S>
__device__ __forceinline__ uint32_t vertex_kinds(const S& sm, int lx, int ly, int rz, int rzm) {
  const int fa = (ly + 1) * S::FX + lx + 1;
  uint32_t w = sm.kinds[0][rz][fa];
  if constexpr (S::P == 2) w |= sm.kinds[S::P - 1][rz][fa];
  w &= 0x3FFFu;
  static_for<0, 7>([&](auto I) {
    constexpr int t = decltype(I)::value, c = kStar.corner[t];
    constexpr int back = (c & 1) + S::FX * ((c >> 1) & 1);
    w |= sm.kinds[S::part_of(t)][(c >> 2) ? rzm : rz][fa - back] & (3u << (14 + 2 * t));
  });
  return w;
}

// The anchors [x0, x0+TX) x [y0, y0+TY) x [z0, zend) of one field: writes
// their records and desc.  Adds the critical simplices of the written records
// to ncrit (per thread) and the minima to sm.counts[0].  Requires the shared
// tables loaded, sm.hi zero, sm.nlist zero.
// With TMA (tm: the field's tensor map), windows come from the TMA ring, slab
// z0 - 1 + j in window j % 5; returns false if a copy did not land (the tile
// is then left unfinished).
template <int TY, bool TMA = false, int PARTS = 1>
__device__ bool gradient_tile(Smem<TY, TMA, PARTS>& sm, const uint32_t* __restrict__ order,
                              const Grid& g, int x0, int y0, int64_t z0, int64_t zend,
                              uint8_t* __restrict__ desc, uint64_t* __restrict__ rec,
                              unsigned int (&ncrit)[3], const CUtensorMap* tm = nullptr) {
  using S = Smem<TY, TMA, PARTS>;
  constexpr int NT = S::NT, NS = S::NSLAB;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t zlast = (zend < g.nz - 1) ? zend : g.nz - 1;  // vertex slabs [z0, zlast]
  const int J = (int)(zlast - z0) + 2;                        // windows 0..J: slabs z0-1..zlast+1
  const bool edge_tile = x0 - 4 < 0 || x0 - 4 + S::WX > g.nx || y0 - 2 < 0 || y0 - 2 + S::WY > g.ny;
  int issued = 0, waited = 0;
  auto issue = [&]() {  // the next window, by TMA
    if constexpr (TMA) {
      if (tid == 0) tma_issue(sm, tm, issued % NS, x0, y0, z0 - 1 + issued);
      ++issued;
    }
  };
  // the next window complete (all threads together see it, and the result,
  // only after the caller's __syncthreads_and): one warp waits for the copy,
  // or, where the window has entries outside the grid to overwrite, every one
  auto land = [&]() -> bool {
    bool ok = true;
    if constexpr (TMA) {
      const int64_t zs = z0 - 1 + waited;
      const bool fix = edge_tile || zs < 0 || zs >= g.nz;
      const int b = waited % NS;
      if (fix || tid < 32) ok = tma_wait(sm, b, (uint32_t)((waited / NS) & 1));
      if (fix && ok) tma_fix_border(sm, g, b, x0, y0, zs);
    } else {
      load_slab<TY, PARTS>(sm, order, g, x0, y0, z0 - 1 + waited, waited % NS);
    }
    ++waited;
    return ok;
  };
  // the next task of a phase, for a warp
  auto next_task = [&](int phase) -> int {
    unsigned int t = 0;
    if (lane == 0) t = atomicAdd(&sm.task[phase], 1u);
    return (int)__shfl_sync(0xFFFFFFFFu, t, 0);
  };

  // tasks are drawn over what of the tile lies in the grid: its vertices, and
  // its anchors from -1 on
  if (tid == 0) {
    const int vx = (int)min(g.nx - x0, (int64_t)TX + 1), vy = (int)min(g.ny - y0, (int64_t)TY + 1);
    sm.verts = Rows(vx, vy);
    sm.anchors = Rows(vx + 1, vy + 1);
  }

  // the rule for 64 anchors (their edges of one part) of the slab with window
  // b0 (its neighbours' bm, bp) and record slab rz (the one below: rzm)
  auto rule_task = [&](int task, int bm, int b0, int bp, int rz, int rzm, uint32_t one) {
    const uint32_t *wm = sm.win[bm], *w0 = sm.win[b0], *wp = sm.win[bp];
    const Rows anchors = sm.anchors;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      const int a = (PARTS == 2 ? task >> 1 : task) * 64 + k * 32 + lane;
      if (a >= anchors.n) return;
      const int row = anchors.row(a), lx = a - row * anchors.cols - 1, ly = row - 1;
      if (PARTS == 2 && (task & 1))
        apply_rule<PARTS - 1, S, PARTS>(sm, wm, w0, wp, lx, ly, rz, rzm, one);
      else
        apply_rule<0, S, PARTS>(sm, wm, w0, wp, lx, ly, rz, rzm, one);
    }
  };

  // desc of 32 vertices of slab z, or their entries in the lists of `fz`
  auto vert_task = [&](int task, int64_t z, int rz, int rzm, int fz) {
    const int i = task * 32 + lane;
    const Rows verts = sm.verts;
    const int ly = verts.row(i), lx = i - ly * verts.cols;
    int cls = -1;
    if (i < verts.n) {
      const uint32_t w = vertex_kinds(sm, lx, ly, rz, rzm);
      const uint32_t b0 = w & 0x5555555u, b1 = (w >> 1) & 0x5555555u, empty = b0 & ~b1;
      if (empty != 0 && (b1 != 0 || (empty & (empty - 1)) != 0)) {
        cls = (b0 & b1) ? 3 : (b1 == 0 ? 0 : ((b1 & (b1 - 1)) ? 2 : 1));
      } else if (lx < TX && ly < TY && z < zend) {
        const int d = empty ? (__ffs(empty) - 1) >> 1 : 15;
        (desc + z * g.sxy)[(uint32_t)(x0 + lx) + (uint32_t)g.nx * (uint32_t)(y0 + ly)] = (uint8_t)d;
        if (d == 15) atomicAdd(&sm.counts[0], 1u);
      }
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, cls >= 0);
    if (!m) return;
    const unsigned m0 = __ballot_sync(0xFFFFFFFFu, cls & 1), m1 = __ballot_sync(0xFFFFFFFFu, cls & 2);
    // lane k < 4 takes the places of class k; every lane the mask of its class
    auto of_class = [&](int c) { return m & ((c & 1) ? m0 : ~m0) & ((c & 2) ? m1 : ~m1); };
    unsigned int at = 0;
    if (lane < 4) at = atomicAdd(&sm.nlist[fz][lane], (unsigned)__popc(of_class(lane)));
    at = __shfl_sync(0xFFFFFFFFu, at, cls & 3);
    if (cls >= 0) {
      at += __popc(of_class(cls) & ((1u << lane) - 1u));
      sm.list[cls >> 1][(cls & 1) ? S::VN - 1 - at : at] = (uint16_t)i;
    }
  };

  // corrects 32 vertices of one class of slab z (window slot b0)
  auto correct_task = [&](int cls, int first, int count, int64_t z, int b0, int rz, int rzm) {
    const int e = first + lane;
    const bool on = e < count;
    const int i = on ? sm.list[cls >> 1][(cls & 1) ? S::VN - 1 - e : e] : 0;
    const Rows verts = sm.verts;
    const int ly = verts.row(i), lx = i - ly * verts.cols;
    const int at = (ly + 2) * S::WX + lx + S::XOFF;
    TileStar<S> star{sm, at, (ly + 2) * S::RX + lx + 2, b0, rz, rzm};
    uint32_t lm = 0;
    if (cls == 3) {
      const uint32_t ox = sm.win[b0][at];
#pragma unroll
      for (int s = 0; s < 14; ++s) lm |= (star.o(s) < ox ? 1u : 0u) << s;
    }
    const uint32_t w = vertex_kinds(sm, lx, ly, rz, rzm);
    const uint32_t k0 = w & 0x5555555u, k1 = (w >> 1) & 0x5555555u;
    const int d = lowerstar::correct_star(star, sm.tb, on, lm, slots_of(k0 & ~k1), slots_of(k1 & ~k0),
                                          slots_of(k0 & k1));
    if (on && lx < TX && ly < TY && z < zend)
      (desc + z * g.sxy)[(uint32_t)(x0 + lx) + (uint32_t)g.nx * (uint32_t)(y0 + ly)] = (uint8_t)d;
  };

  // writes out a row of anchors of slab zw in record slab r (all of whose
  // vertices' slabs are done) and clears the row's words for the slab that
  // takes them over; the last three are the halo's, only cleared
  auto flush_task = [&](int row, int64_t zw, int r) {
    const int frows = min(sm.verts.rows, TY);
    const int ry = row < frows ? row + 2 : (row == frows + 2 ? TY + 2 : row - frows);
    uint32_t* hi = &sm.hi[r][ry * S::RX];
    const int64_t gx = x0 + lane, gy = y0 + row;
    if (row < frows && zw >= z0 && zw < zend && gx < g.nx) {
      uint32_t l = sm.lo[0][r][ry * S::RX + 2 + lane], h = hi[2 + lane];
      if constexpr (PARTS == 2) l |= sm.lo[PARTS - 1][r][ry * S::RX + 2 + lane];
      // simplices that leave the grid are absent
      if (gx == g.nx - 1) l &= ~reach_lo(0), h = 0;
      if (gy == g.ny - 1) l &= ~reach_lo(1), h = 0;
      if (zw == g.nz - 1) l &= ~reach_lo(2), h = 0;
      (rec + (gy + g.ny * zw) * g.nx)[gx] = (uint64_t)h << 32 | l;
      // code 7: the three bits; the counts of a lane stay far below 2^32
      const uint32_t ce = l & (l >> 1) & (l >> 2) & (uint32_t)kEdgeLsb;
      const uint32_t ct = (l & (uint32_t)kTriMask) | (h & 1u);
      const uint32_t cq = h & (h >> 1) & (h >> 2) & (uint32_t)(kTetLsb >> 32);
      if (ce | ct | cq) {
        ncrit[0] += __popc(ce);
        ncrit[1] += __popc(ct);
        ncrit[2] += __popc(cq);
      }
    }
    hi[lane] = 0;
    if (lane < S::RX - 32) hi[32 + lane] = 0;
  };

  for (int i = tid; i < 3 * S::RN; i += NT) (&sm.hi[0][0])[i] = 0;
  // the window under the first slab's is not loaded: what it decides there
  // belongs to that slab's vertices, which are not this tile's
  for (int i = tid; i < S::SLAB; i += NT) sm.win[NS - 1][i] = 0xFFFFFFFFu;
  if (tid < 8) sm.nlist[tid >> 2][tid & 3] = 0;
  if (tid < 2) sm.task[tid] = 0;
#pragma unroll 1
  for (int j = 0; j < 3; ++j) issue();  // J >= 2: all three are needed

  // j = -1: only the first slab's rule; past jlast: only records.  (Every part
  // has one place in the loop: the code has to stay in the instruction cache.)
  const int jlast = (int)(zlast - z0) + 1;
  int b0 = NS - 1, rz = 2;  // window slot j % NS and record slab j % 3 of slab z0 - 1 + j
#pragma unroll 1
  for (int j = -1; j <= jlast + 2; ++j) {
    const int fz = j & 1, rzm = rz ? rz - 1 : 2, rzp = rz < 2 ? rz + 1 : 0;
    const int bp = b0 + 1 < NS ? b0 + 1 : 0, bpp = bp + 1 < NS ? bp + 1 : 0;
    const int64_t z = z0 - 1 + j;
    const bool in = j >= 1 && j <= jlast;  // a slab of this tile's vertices
    // ---- kinds -> desc and lists; records two slabs down; the window two up
    if (j >= 0 && j + 3 <= J) issue();  // window j - 2 was last read by the correction of slab j - 1
    bool ok = true;
#pragma unroll 1
    for (int k = j < 0 ? 0 : (j + 2 <= J ? 1 : 2); k < 2; ++k) ok = land() && ok;
    if (j >= 1) {
      const int vertTasks = (sm.verts.n + 31) / 32, first = in ? 0 : vertTasks;
      const int all = vertTasks + min(sm.verts.rows, TY) + 3;
      for (int t = next_task(1) + first; t < all; t = next_task(1) + first) {
        if (t < vertTasks) vert_task(t, z, rz, rzm, fz);
        else flush_task(t - vertTasks, z - 2, rzp);
      }
    }
    if (tid < 4) sm.nlist[fz ^ 1][tid] = 0;  // the next slab's; the last slab's are done
    if (tid == 4) sm.task[0] = 0;
    if (!__syncthreads_and(ok)) {
      if constexpr (TMA)  // wait (bounded) for the copies in flight
        for (; waited < issued; ++waited) (void)tma_wait(sm, waited % NS, (uint32_t)((waited / NS) & 1));
      return false;
    }
    // ---- corrections of this slab, the longest first, then the next slab's rule
    if (tid == 0) sm.task[1] = 0;
    uint4 nl = *reinterpret_cast<const uint4*>(sm.nlist[fz]);
    if (!in) nl = make_uint4(0, 0, 0, 0);
    // a warp takes as many lanes' worth as keeps all warps busy: a correction
    // takes as long as its longest lane
    const int listed = (int)(nl.x + nl.y + nl.z + nl.w);
    const int per = listed >= NT ? 32 : max(4, (listed + NT / 32 - 1) / (NT / 32));
    const int t3 = ((int)nl.w + per - 1) / per, t2 = t3 + ((int)nl.z + per - 1) / per;
    const int t1 = t2 + ((int)nl.y + per - 1) / per, tasks = t1 + ((int)nl.x + per - 1) / per;
    const int all = tasks + (j < jlast ? (sm.anchors.n + 63) / 64 * PARTS : 0);
    const uint32_t one = *(volatile uint32_t*)&sm.one;
    for (int t = next_task(0); t < all; t = next_task(0)) {
      if (t >= tasks) {
        rule_task(t - tasks, b0, bp, bpp, rzp, rz, one);
      } else {
        const int cls = t < t3 ? 3 : (t < t2 ? 2 : (t < t1 ? 1 : 0));
        const int first = t - (cls == 3 ? 0 : (cls == 2 ? t3 : (cls == 1 ? t2 : t1)));
        const int count = (int)(cls == 3 ? nl.w : (cls == 2 ? nl.z : (cls == 1 ? nl.y : nl.x)));
        correct_task(cls, first * per, min(count, (first + 1) * per), z, b0, rz, rzm);
      }
    }
    __syncthreads();
    b0 = bp;
    rz = rzp;
  }
  return true;
}

// adds the CTA's critical counts to counts[4] (all threads must call)
template <class S>
__device__ __forceinline__ void add_counts(S& sm, unsigned int (&ncrit)[3],
                                           unsigned long long* counts) {
  const int tid = threadIdx.x, lane = tid & 31;
  for (int d = 0; d < 3; ++d) {
    unsigned int v = ncrit[d];
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (lane == 0 && v) atomicAdd(&sm.counts[d + 1], v);
    ncrit[d] = 0;
  }
  __syncthreads();
  if (tid < 4) {
    if (sm.counts[tid]) atomicAdd(&counts[tid], (unsigned long long)sm.counts[tid]);
    sm.counts[tid] = 0;
  }
  __syncthreads();
}

// one field, one CTA per tile of anchors; with TMA the order slabs come
// through the tensor map tmap.  A TMA copy that does not land sets bit 63
// of counts[0] (the call has failed) and ends the CTA.
template <int TY, bool TMA>
__global__ void __launch_bounds__(threads_of(TY), ctas_of(TY))
    gradient_kernel(const uint32_t* __restrict__ order, Grid g, int zc, uint8_t* __restrict__ desc,
                    uint64_t* __restrict__ rec, unsigned long long* __restrict__ counts,
                    const __grid_constant__ CUtensorMap tmap) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Smem<TY, TMA>& sm = *reinterpret_cast<Smem<TY, TMA>*>(smem_raw);
  const int tid = threadIdx.x;
  load_tables(sm);
  if constexpr (TMA) tma_init(sm);
  const int64_t z0 = (int64_t)blockIdx.z * zc;
  const int64_t zend = (z0 + zc < g.nz) ? z0 + zc : g.nz;
  unsigned int ncrit[3] = {0, 0, 0};
  if (!gradient_tile<TY, TMA>(sm, order, g, blockIdx.x * TX, blockIdx.y * TY, z0, zend, desc, rec,
                              ncrit, &tmap)) {
    if (tid == 0) atomicOr(counts, 1ull << 63);
    return;
  }
  add_counts(sm, ncrit, counts);
}

// Many fields, persistent: every CTA takes tiles from one queue that runs over
// all fields (field f owns tiles [tile0[f], tile0[f+1])), so uneven fields
// share the GPU without one launch per field.
struct BatchTiles {
  const dms_field_desc* fields;
  const long long* tile0;  // nfields + 1 prefix counts of tiles
  int nfields;
  int zc;                  // anchor slabs per tile
  unsigned long long* queue;
};

template <int TY, int PARTS>
__global__ void __launch_bounds__(threads_of(TY), ctas_of(TY))
    gradient_batch_kernel(const uint32_t* __restrict__ order, BatchTiles bt,
                          uint8_t* __restrict__ desc, uint64_t* __restrict__ rec,
                          unsigned long long* __restrict__ counts) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using S = Smem<TY, false, PARTS>;
  S& sm = *reinterpret_cast<S*>(smem_raw);
  const int tid = threadIdx.x;
  load_tables(sm);
  const long long total = bt.tile0[bt.nfields];
  unsigned int ncrit[3] = {0, 0, 0};
  for (;;) {
    __syncthreads();
    if (tid == 0) sm.tile = (long long)atomicAdd(bt.queue, 1ull);
    __syncthreads();
    const long long t = sm.tile;
    if (t >= total) break;
    int lo = 0, hi = bt.nfields;  // the field holding tile t
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (bt.tile0[mid] <= t) lo = mid;
      else hi = mid;
    }
    const dms_field_desc fd = bt.fields[lo];
    Grid g;
    g.nx = fd.nx;
    g.ny = fd.ny;
    g.nz = fd.nz;
    g.sxy = (int64_t)fd.nx * fd.ny;
    g.n = g.sxy * fd.nz;
    const long long local = t - bt.tile0[lo];
    const int tx = (fd.nx + TX - 1) / TX, ty = (fd.ny + TY - 1) / TY;
    const long long bx = local % tx, by = (local / tx) % ty, bz = local / ((long long)tx * ty);
    const int64_t z0 = bz * bt.zc;
    const int64_t zend = (z0 + bt.zc < g.nz) ? z0 + bt.zc : g.nz;
    gradient_tile<TY, false, PARTS>(sm, order + fd.offset, g, (int)bx * TX, (int)by * TY, z0, zend,
                                  desc + fd.offset, rec + fd.offset, ncrit);
    add_counts(sm, ncrit, counts + 4 * lo);
  }
}

// tile counts per field -> prefix (one small CTA)
__global__ void batch_tiles_kernel(const dms_field_desc* __restrict__ fields, int nfields, int ty,
                                   int zc, long long* tile0, unsigned long long* queue) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  long long acc = 0;
  for (int f = 0; f < nfields; ++f) {
    tile0[f] = acc;
    const dms_field_desc fd = fields[f];
    acc += (long long)((fd.nx + TX - 1) / TX) * ((fd.ny + ty - 1) / ty) * ((fd.nz + zc - 1) / zc);
  }
  tile0[nfields] = acc;
  *queue = 0ull;
}

// cuTensorMapEncodeTiled from the driver (the library links only the runtime)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// the order field as an nx x ny x nz u32 tensor with WX x WY x 1 boxes; false
// where TMA cannot stage it (row pitch not a multiple of 16 bytes, an
// unaligned pointer, no encoder) -- the kernel then loads with __ldg
template <int TY>
bool order_tensor_map(CUtensorMap* m, const uint32_t* order, const Grid& g) {
  if (g.nx % 4 != 0 || (reinterpret_cast<uintptr_t>(order) & 15) != 0) return false;
  const EncodeTiledFn fn = encode_tiled();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz};
  const cuuint64_t strides[2] = {(cuuint64_t)g.nx * 4, (cuuint64_t)g.sxy * 4};
  const cuuint32_t box[3] = {(cuuint32_t)Smem<TY, true>::WX, (cuuint32_t)Smem<TY, true>::WY, 1};
  const cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<uint32_t*>(order), dims, strides, box,
            es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int TY, bool TMA>
int launch_single(const uint32_t* order, const Grid& g, uint8_t* desc, uint64_t* rec,
                  int64_t* crit_counts, const CUtensorMap& tmap, cudaStream_t s) {
  static bool configured = false;
  const size_t smem = sizeof(Smem<TY, TMA>);
  constexpr int NT = threads_of(TY);
  if (!configured) {
    if (cudaFuncSetAttribute(gradient_kernel<TY, TMA>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
      return DMS_ERR_CUDA;
    configured = true;
  }
  int dev = 0, sms = 148, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gradient_kernel<TY, TMA>, NT, smem) !=
          cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  const int64_t tx = (g.nx + TX - 1) / TX, ty = (g.ny + TY - 1) / TY;
  const int64_t cap = (int64_t)sms * per_sm, tiles = tx * ty;
  int64_t nzc;
  if (g.n <= kSmallGrid) {
    // a small grid: the CTAs' slabs one after the other are the time, so as
    // few slabs each as fill the GPU once
    nzc = std::max<int64_t>(1, std::min<int64_t>(cap / tiles, g.nz));
  } else {
    // about 16 waves of resident CTAs, so that the last, partly filled wave
    // costs little, in chunks of at least 32 slabs (each chunk also applies
    // the rule to the slabs below and above it); a grid that such chunks leave under two
    // waves takes chunks down to 8 slabs, and one wave where the second would
    // be nearly empty (300 x 300 x 16 noise, 494 CTAs for 456 places: 0.56 ms
    // against 0.40 in one wave)
    nzc = std::max<int64_t>(1, std::min<int64_t>((16 * cap + tiles - 1) / tiles, g.nz / 32));
    if (tiles * nzc < 2 * cap)
      nzc = std::max<int64_t>(1, std::min<int64_t>((2 * cap + tiles - 1) / tiles, (g.nz + 7) / 8));
    if (tiles <= cap && tiles * nzc > cap && tiles * nzc * 4 < cap * 5) nzc = cap / tiles;
  }
  const int zc = (int)((g.nz + nzc - 1) / nzc);
  nzc = (g.nz + zc - 1) / zc;
  if (cudaMemsetAsync(crit_counts, 0, 4 * sizeof(int64_t), s) != cudaSuccess) return DMS_ERR_CUDA;
  dim3 grid((unsigned)tx, (unsigned)ty, (unsigned)nzc);
  gradient_kernel<TY, TMA><<<grid, NT, smem, s>>>(
      order, g, zc, desc, rec, reinterpret_cast<unsigned long long*>(crit_counts), tmap); count_launch();
  return launch_status();
}

template <int TY, int PARTS>
int launch_batch(const uint32_t* order, const dms_field_desc* fields_dev, int nfields, int zc,
                 uint8_t* desc, uint64_t* rec, int64_t* counts, long long* tile0,
                 unsigned long long* queue, cudaStream_t s) {
  static bool configured = false;
  const size_t smem = sizeof(Smem<TY, false, PARTS>);
  constexpr int NT = threads_of(TY);
  if (!configured) {
    if (cudaFuncSetAttribute(gradient_batch_kernel<TY, PARTS>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
      return DMS_ERR_CUDA;
    configured = true;
  }
  int dev = 0, sms = 148, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gradient_batch_kernel<TY, PARTS>, NT,
                                                    smem) !=
          cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  DMS_CUDA_OK(cudaMemsetAsync(counts, 0, 4 * sizeof(int64_t) * nfields, s));
  batch_tiles_kernel<<<1, 32, 0, s>>>(fields_dev, nfields, TY, zc, tile0, queue); count_launch();
  BatchTiles bt{fields_dev, tile0, nfields, zc, queue};
  gradient_batch_kernel<TY, PARTS><<<(unsigned)(sms * per_sm), NT, smem, s>>>(
      order, bt, desc, rec, reinterpret_cast<unsigned long long*>(counts)); count_launch();
  return launch_status();
}

}  // namespace

// the batch variants the autotuner chooses from: tile height (variant % 3:
// 24, 16, 32 anchor rows) x threads per anchor (1 + variant / 3)
constexpr int kTileVariants = 6;
int gradient_batch_variants() { return kTileVariants; }
int gradient_tile_height(int variant) {
  const int t = variant % 3;
  return t == 1 ? 16 : (t == 2 ? 32 : 24);
}

template <int TY>
int launch_gradient_tiles(const uint32_t* order, const Grid& g, uint8_t* desc, uint64_t* rec,
                          int64_t* crit_counts, cudaStream_t s) {
  CUtensorMap tmap;
  if (order_tensor_map<TY>(&tmap, order, g))
    return launch_single<TY, true>(order, g, desc, rec, crit_counts, tmap, s);
  std::memset(&tmap, 0, sizeof(tmap));
  return launch_single<TY, false>(order, g, desc, rec, crit_counts, tmap, s);
}

int launch_gradient(const uint32_t* order, const Grid& g, uint8_t* desc, uint64_t* rec,
                    int64_t* crit_counts, cudaStream_t s) {
  return g.n <= kSmallGrid || g.ny <= kSmallTY
             ? launch_gradient_tiles<kSmallTY>(order, g, desc, rec, crit_counts, s)
                           : launch_gradient_tiles<24>(order, g, desc, rec, crit_counts, s);
}

int launch_gradient_batch(const uint32_t* order, const dms_field_desc* fields_dev, int nfields,
                          int variant, int zc, uint8_t* desc, uint64_t* rec, int64_t* counts,
                          long long* tile0, unsigned long long* queue, cudaStream_t s) {
  switch (variant) {
    case 1: return launch_batch<16, 1>(order, fields_dev, nfields, zc, desc, rec, counts, tile0, queue, s);
    case 2: return launch_batch<32, 1>(order, fields_dev, nfields, zc, desc, rec, counts, tile0, queue, s);
    case 3: return launch_batch<24, 2>(order, fields_dev, nfields, zc, desc, rec, counts, tile0, queue, s);
    case 4: return launch_batch<16, 2>(order, fields_dev, nfields, zc, desc, rec, counts, tile0, queue, s);
    case 5: return launch_batch<32, 2>(order, fields_dev, nfields, zc, desc, rec, counts, tile0, queue, s);
    default: return launch_batch<24, 1>(order, fields_dev, nfields, zc, desc, rec, counts, tile0, queue, s);
  }
}

}  // namespace dms
