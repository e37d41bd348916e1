// barrier.h -- the grid barrier's word: what a value of it says about a barrier.
//
// One 32-bit word per launch, zero before it.  Open (top bit clear): arrivals so far; barrier
// number e of nb blocks is complete at e nb arrivals (its target).  Closed (top bit set): the rest
// is the target of the barrier that some block gave up on, plus the arrivals since then (fewer
// than nb: that barrier's stragglers).  A block closes the word only by a compare-and-swap from an
// open value below its target, so the order of the operations on this one word decides each barrier
// for all blocks alike: a barrier that was complete before the word was closed passes in every
// block, however late it looks; the one the word was closed at fails in every block that reaches
// it, and nobody gets beyond it.  (Blocks that judged a barrier by what else they saw -- a status
// word, their own clock -- disagreed about it, and one could leave while another went on to read
// its shared memory.)  2^31 arrivals, 1.5 million iterations of a solve on 152 blocks, read as
// closed.  Every instruction between a barrier's last arrival and its release counts, so both
// halves of the verdict are one comparison: at 690 barriers of 112 blocks a pass (3.34 ms) this
// form costs nothing measurable against a counter without a verdict, one that told waiting, passed
// and failed apart in the poll 1.8%, and the same in a 64-bit word 2.7%.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ETD_BAR_FN __host__ __device__ __forceinline__
#else
#define ETD_BAR_FN inline
#endif

namespace etd {

constexpr uint32_t kBarClosed = 0x80000000u;

// Target of the barrier at which a block arrives, from the word before its arrival (for a straggler
// at a closed word, the one after: not passed either).
ETD_BAR_FN uint32_t bar_target(uint32_t before, uint32_t nb) { return ((before & ~kBarClosed) / nb + 1u) * nb; }

// Whether a value of the word decides the barrier, and then how.
ETD_BAR_FN bool bar_decided(uint32_t word, uint32_t target) { return word >= target; }
ETD_BAR_FN bool bar_passed(uint32_t word, uint32_t target, uint32_t nb) {
  return word < kBarClosed || (word & ~kBarClosed) >= target + nb;
}

// An open word closed at `target`.
ETD_BAR_FN uint32_t bar_closed(uint32_t target) { return kBarClosed | target; }

}  // namespace etd
