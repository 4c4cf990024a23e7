// serving.cuh -- the serving loop's rules that need no device.
#pragma once

#include <algorithm>
#include <cstdint>

namespace dpd {

// How many handles a box that starts now is expected to run beside, itself
// included: those admitted and the queued boxes that will take one (not those
// routed to the ensemble kernel), at most max_active.
template <typename Jobs>
int handles_expected(int64_t active, const Jobs &pending, int max_active)
{
    int64_t queued = 0;
    for (const auto &j : pending) queued += j.ens ? 0 : 1;
    return (int)std::min<int64_t>(active + queued, max_active);
}

}  // namespace dpd
