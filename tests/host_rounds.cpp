// Host build of the counters of the pairing rounds (dms_rounds.cuh), for the
// simulation of their hand-over in test_rounds_handover.py.
#include "dms_rounds.cuh"

extern "C" {
int host_count_word(unsigned round, int solo) { return dms::count_word(round, solo != 0); }
int host_goes_solo(unsigned n, long long nn, int forest) { return dms::goes_solo(n, nn, forest != 0); }
unsigned host_solo() { return dms::kSolo; }
int host_words() { return dms::kCtrWords; }
int host_forest_word() { return dms::kCtrForest; }
int host_first_round_word() { return dms::kCtrRound; }
}
