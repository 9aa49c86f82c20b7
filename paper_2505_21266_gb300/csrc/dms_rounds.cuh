// The counters of the pairing rounds, and when CTA 0 works them alone.
// Host-compilable as well: the CPU tests run the hand-over from the grid to
// CTA 0 on these.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define DMS_ROUNDS_HD __host__ __device__ __forceinline__
#else
#define DMS_ROUNDS_HD inline
#endif

namespace dms {

constexpr unsigned int kSolo = 4096;     // live saddles that CTA 0 works alone
constexpr int64_t kSoloNodes = 1 << 16;  // nodes that it sets back alone

// words of DiagWs::ctr
enum : int {
  kCtrLive = 0,      // saddles live after the walks
  kCtrNext = 1,      // live saddles of the rounds of one launch per phase: with kCtrLive in turn
  kCtrForest = 2,    // saddles of the spanning forest
  kCtrChanged = 3,   // (self-correcting pairing)
  kCtrBig = 4,       // saddles left to the device-wide sorted finish (batch)
  kCtrRound = 8,     // three live counts in turn, of the grid's rounds
  kCtrLeft = 11,     // saddles left live by the exact rounds
  kCtrBarrier = 12,
  kCtrAbort = 13,
  kCtrSolo = 14,     // three live counts in turn, of the rounds of CTA 0 alone
  kCtrWords = 20
};

// where round r counts the saddles that stay live.  CTA 0 alone meets nobody
// at a barrier, so it counts in words of its own: the others read the count of
// the grid's last round, by which they leave, whenever they get to it.
DMS_ROUNDS_HD int count_word(unsigned int round, bool solo) {
  return (solo ? kCtrSolo : kCtrRound) + (int)(round % 3);
}

// whether CTA 0 goes on alone with n live saddles of nn nodes
DMS_ROUNDS_HD bool goes_solo(unsigned int n, int64_t nn, bool forest) {
  return n <= kSolo && (!forest || nn <= kSoloNodes);  // (many nodes are set back by the whole grid)
}

}  // namespace dms
