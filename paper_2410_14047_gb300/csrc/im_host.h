// Host-side bookkeeping that needs no CUDA (compiled and tested on the CPU as
// well): which counter set a phase runs on.
#pragma once
#include <algorithm>

#ifdef __CUDACC__
#define IM_HD __host__ __device__ __forceinline__
#else
#define IM_HD inline
#endif

namespace imi {

// Entries at the start of a counter set (of `all`) that the phase which ran
// there last may have left nonzero: those of a phase of `levels` levels, or the
// whole set once a phase has given up (its blocks may have come further than
// the one that recorded the levels, and the phases after it record none).
IM_HD int set_entries_used(bool gave_up, int levels, int all) {
    return gave_up || levels + 2 > all ? all : levels + 2;
}

// The two sets of per-level counters, work counters and barrier words that the
// phases of a sketch use in turn.  A set has to be zero when its phase begins
// (level 0 is written by the kernels before the phase's launch): the phase
// launch in between zeroes what the one before it used, otherwise the host
// zeroes all of it (after a phase that ran in launches of their own, or whose
// launch failed: then nothing ran).
class PhaseSets {
public:
    int cur() const { return cur_; }
    int other() const { return cur_ ^ 1; }
    // The next phase begins, on the other set; true: the host zeroes it first.
    bool begin() {
        cur_ ^= 1;
        const bool zero = state_[cur_] != kZeroed;
        state_[cur_] = kDirty;
        return zero;
    }
    // Its launch is to zero what the phase before it used in the other set.
    bool zero_other() const { return state_[other()] == kUsed; }
    // That launch went out.
    void launched() {
        if (zero_other()) state_[other()] = kZeroed;
        state_[cur_] = kUsed;
    }

private:
    enum State { kDirty, kZeroed, kUsed };
    int cur_ = 0;
    State state_[2] = {kDirty, kDirty};
};

}  // namespace imi
