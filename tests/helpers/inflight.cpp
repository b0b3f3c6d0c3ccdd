// Test helper, not part of the library: the order rule of launches that may overlap, behind a C interface.
#include "inflight.h"

using kvzap::InFlight;

extern "C" {
InFlight *inflight_new() { return new InFlight; }
void inflight_delete(InFlight *f) { delete f; }
int inflight_max_chain() { return InFlight::kMaxChain; }
// uses: n triples (address, bytes, write); returns wait | late << 4
int inflight_next(InFlight *f, const long long *uses, int n, int wait_all, int stores_wait)
{
    InFlight::Use u[16];
    for (int i = 0; i < n; ++i) u[i] = {reinterpret_cast<const void *>(uses[3 * i]), static_cast<size_t>(uses[3 * i + 1]), uses[3 * i + 2] != 0};
    const InFlight::Order o = f->next(u, n, wait_all != 0, stores_wait);
    return o.wait | (o.late ? 16 : 0);
}
int inflight_busy(const InFlight *f, long long p, long long n, int write)
{
    return f->busy(reinterpret_cast<const void *>(p), static_cast<size_t>(n), write != 0) ? 1 : 0;
}
}
