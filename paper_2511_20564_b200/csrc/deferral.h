// Which callers' streams have waited for which helper streams' deferred work (host bookkeeping, plain C++).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <vector>

namespace e2egrec {

// The helper streams of one device, numbered 0, 1, ... in the order of their creation; a caller's stream goes by the number
// of its own helper.  Every caller's stream waits for every deferral once: that another one has waited for it orders
// nothing here (the owner of the work reuses the sampler scratch and reads the blocks that the work is still using).
class DeferralLedger {
public:
    // helper `h` leaves work behind, inside the stream capture `capture` (0: none)
    void defer(size_t h, uint64_t capture)
    {
        Work &w = at(h);
        ++w.generation;
        w.capture = capture;
        w.open = true;
    }

    // Calls wait(h) for every helper whose last deferred work the stream of helper `waiter` has not waited for.  Work that
    // no stream has waited for is always waited for.  Work that some stream has waited for is skipped where the capture
    // (what capture() returns, asked for at most once) is another one: inside a capture no wait for work outside it can be
    // recorded, and a capture that has ended has joined all that was forked in it.
    template <class Capture, class Wait> void join(size_t waiter, Capture capture, Wait wait)
    {
        at(waiter);
        std::vector<uint64_t> &seen = work_[waiter].seen;
        seen.resize(work_.size(), 0);
        bool asked = false;
        uint64_t mine = 0;
        for (size_t h = 0; h < work_.size(); ++h) {
            Work &w = work_[h];
            if (seen[h] == w.generation) continue;
            if (!w.open) {
                if (!asked) mine = capture();
                asked = true;
                if (mine != w.capture) continue;
            }
            wait(h);
            w.open = false;
            seen[h] = w.generation;
        }
    }

private:
    struct Work {
        uint64_t generation = 0;          // deferrals so far
        uint64_t capture = 0;             // of the last one
        bool open = false;                // no stream has waited for it
        std::vector<uint64_t> seen;       // per helper: the generation that this helper's caller has waited for
    };
    Work &at(size_t h)
    {
        if (h >= work_.size()) work_.resize(h + 1);
        return work_[h];
    }
    std::vector<Work> work_;
};

}  // namespace e2egrec
