// Host-side bookkeeping that needs no CUDA (compiled and tested on the CPU as
// well): which counter set a phase runs on, how the calls that run at the same
// time divide a device's blocks, and how long a phase on some of them may wait.
#pragma once
#include <condition_variable>
#include <cstdint>
#include <map>
#include <mutex>

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

// The blocks of one device that fit it at once in every phase launch, divided
// among the calls that run phases.  A phase runs all its levels in one
// cooperative launch whose blocks wait for one another, so the grids in flight
// must never add up to more than the device holds: a call takes blocks before
// its first phase, gives back or takes more only while none of its phases is in
// flight, and returns them at its end.  The even share is total / running: a
// call that joins waits until the others have come down to it, a selection at
// its next seed.
class BlockAccount {
public:
    explicit BlockAccount(int total) : total_(total), free_(total) {}
    int total() const { return total_; }

    // A call starts; leave ends it and returns what it holds.
    void enter() {
        std::lock_guard<std::mutex> lk(mu_);
        ++running_;
    }
    void leave(int held) {
        std::lock_guard<std::mutex> lk(mu_);
        --running_;
        free_ += held;
        cv_.notify_all();
    }
    // Its first phase comes: waits for its share, returns it.
    int take() {
        std::unique_lock<std::mutex> lk(mu_);
        cv_.wait(lk, [&] { return free_ >= even(); });
        const int take = even();
        free_ -= take;
        return take;
    }
    // No phase of it is in flight: its new share in place of `held`.
    int adjust(int held) {
        std::lock_guard<std::mutex> lk(mu_);
        const int want = even(), most = held + free_;
        const int take = want < most ? want : most;
        free_ += held - take;
        if (take < held) cv_.notify_all();
        return take;
    }

private:
    int even() const { return total_ > running_ ? total_ / running_ : 1; }
    std::mutex mu_;
    std::condition_variable cv_;
    const int total_;
    int free_;
    int running_ = 0;
};

// The bound on a barrier wait of a phase on `blocks` of the device's `total`, from
// the bound `ns` for all of them: a level's work is the same on fewer blocks, so
// it and the wait for its slowest block take up to total / blocks times as long
// (one of 40 queries holds 7 of 304 blocks).  0 (give up at the first poll)
// stays 0.
inline uint64_t wait_limit(uint64_t ns, int total, int blocks) {
    const uint64_t times = blocks < total ? ((uint64_t)total + (uint64_t)blocks - 1) / (uint64_t)blocks : 1;
    return ns > UINT64_MAX / times ? UINT64_MAX : ns * times;
}

// The device's account: one for the whole process, from which every server's
// queries and every context's calls take (`total`: the device's blocks, the
// same at each call).  It lives until the process ends.
inline BlockAccount* account_of(int device, int total) {
    static std::mutex mu;
    static auto* accounts = new std::map<int, BlockAccount*>;
    std::lock_guard<std::mutex> lk(mu);
    BlockAccount*& a = (*accounts)[device];
    if (!a) a = new BlockAccount(total);
    return a;
}

}  // namespace imi
