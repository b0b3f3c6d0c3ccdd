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
    bool busy(const void *p, size_t n, bool write) const { return back({p, n, write}) > 0; }

    // The order of the next launch, which uses `uses`; it is in the list behind this call.  wait_all: it has to wait for
    // everything ahead in any case (work that is not in the list lies between).  stores_wait: where only what it writes is in
    // use, last by one of so many launches ahead, its stores wait by themselves and everything up to them goes ahead.  It
    // is not late then, and the list grows; with outputs that come round after more launches than that, all of it would soon
    // be of launches that have long finished, and every launch would wait.  One launch of a round then waits altogether, and
    // the list starts again behind it.
    Order next(const Use *uses, int n, bool wait_all, int stores_wait)
    {
        Order order{kNone, false};
        if (wait_all || chain_ >= kMaxChain || n_ + n > kMaxUses) order.wait = kAll;
        int nearest = kMaxChain + 1;
        for (int i = 0; i < n && order.wait != kAll; ++i) {
            const int b = back(uses[i]);
            if (b == 0) continue;
            order.wait = uses[i].write ? kStores : kAll;
            if (b < nearest) nearest = b;
        }
        if (order.wait == kStores && nearest > stores_wait) order.wait = kAll;
        order.late = order.wait == kAll;
        if (order.late) n_ = chain_ = 0;
        else ++chain_;
        for (int i = 0; i < n; ++i) {
            if (uses[i].p == nullptr || uses[i].n == 0) continue;
            uses_[n_] = uses[i];
            at_[n_++] = chain_;
        }
        return order;
    }

    static constexpr int kMaxChain = 14;    // launches behind a late one that may all run beside it, each with scratch of its own

private:
    // how many launches back the last one is that conflicts with the use, 0 if none does
    int back(const Use &u) const
    {
        if (u.p == nullptr || u.n == 0) return 0;
        const char *a = static_cast<const char *>(u.p);
        for (int i = n_ - 1; i >= 0; --i) {
            const char *b = static_cast<const char *>(uses_[i].p);
            if ((u.write || uses_[i].write) && a < b + uses_[i].n && b < a + u.n) return chain_ + 1 - at_[i];
        }
        return 0;
    }

    static constexpr int kMaxUses = 128;    // of some ten a launch
    Use uses_[kMaxUses];
    int at_[kMaxUses];                      // of which launch behind the last late one
    int n_ = 0, chain_ = 0;
};

}  // namespace kvzap
