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

constexpr unsigned int kSolo = 4096;  // live saddles that CTA 0 works alone

// words of DiagWs::ctr
enum : int {
  kCtrLive = 0,      // saddles live after the walks
  kCtrNext = 1,      // live saddles of the rounds of one launch per phase: with kCtrLive in turn
  kCtrForest = 2,    // saddles of the spanning forest
  kCtrChanged = 3,   // (self-correcting pairing)
  kCtrBig = 4,       // saddles left to the device-wide sorted finish (batch)
  kCtrFar = 5,       // saddles whose paths are long (see kCells)
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

// whether CTA 0 goes on alone with n live saddles of nn nodes.  From the forest's
// rounds it goes on to the exact rounds on the forest's saddles, up to nn - 1:
// those have to be few as well, however few are live before.  With the line at
// 65,536 nodes instead, the D0/D2 stage of noise took 1.00 ms at 64^3 and 2.50
// at 96^3 (17 K and 58 K nodes); it takes 0.66 and 0.90.
DMS_ROUNDS_HD bool goes_solo(unsigned int n, int64_t nn, bool forest) {
  return n <= kSolo && (!forest || nn <= (int64_t)kSolo + 1);
}

}  // namespace dms
