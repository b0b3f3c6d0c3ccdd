// What the launches that may still be running touch, and what the next one therefore has to wait for.  Host only.
//
// For launches that overlap their neighbours on a context that trusts its producers: every one completes after the one ahead
// of it (all its threads wait for that before they exit), and lets the one behind it start either at its first instruction or
// ("late") only once its own wait for the one ahead is over.  So a launch that waits before it stores has everything ahead of
// it complete by then, but the launch behind one that lets go early knows nothing about them: what it may run beside is
// everything since the last late launch, and that is what the list holds.
#pragma once

#include <cstddef>

namespace kvzap {

class InFlight {
public:
    struct Use { const void *p; size_t n; bool write; };
    enum Wait { kNone, kAll, kStores };                       // before nothing, before the first load, before the first store
    struct Order {
        Wait wait;
        bool late;      // the launch behind starts behind this one's wait (or waits itself, on a context that does not trust)
    };

    // Whether a launch in the list uses [p, p + n) in a conflicting way (a write on either side).
    bool busy(const void *p, size_t n, bool write) const
    {
        if (p == nullptr || n == 0) return false;
        const char *a = static_cast<const char *>(p);
        for (int i = 0; i < n_; ++i) {
            const char *b = static_cast<const char *>(uses_[i].p);
            if ((write || uses_[i].write) && a < b + uses_[i].n && b < a + n) return true;
        }
        return false;
    }

    // The order of the next launch, which uses `uses`; it is in the list behind this call.  wait_all: it has to wait for
    // everything ahead in any case (work that is not in the list lies between).  stores_may_wait: its stores can wait by
    // themselves, everything up to them goes ahead.
    Order next(const Use *uses, int n, bool wait_all, bool stores_may_wait)
    {
        Order order{kNone, false};
        if (wait_all || chain_ >= kMaxChain || n_ + n > kMaxUses) order.wait = kAll;
        for (int i = 0; i < n && order.wait != kAll; ++i)
            if (busy(uses[i].p, uses[i].n, uses[i].write)) order.wait = uses[i].write && stores_may_wait ? kStores : kAll;
        order.late = order.wait == kAll;
        if (order.late) n_ = chain_ = 0;
        else ++chain_;
        for (int i = 0; i < n; ++i)
            if (uses[i].p != nullptr && uses[i].n > 0) uses_[n_++] = uses[i];
        return order;
    }

    static constexpr int kMaxChain = 14;    // launches behind a late one that may all run beside it, each with scratch of its own

private:
    static constexpr int kMaxUses = 128;    // of some ten a launch
    Use uses_[kMaxUses];
    int n_ = 0, chain_ = 0;
};

}  // namespace kvzap
