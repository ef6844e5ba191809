// at_resident.cu -- instantiations of the one-subdomain-per-CTA stepper (float
// and double state, order 2 and 4, with and without forcing, 1 to 8 points per
// thread).
#include "at_resident.cuh"

namespace {
template <typename T, int ORDER, bool FORCED>
void *by_points(int ppt)
{
    switch (ppt) {
    case 1: return (void *)atk::at_resident<T, ORDER, 1, FORCED>;
    case 2: return (void *)atk::at_resident<T, ORDER, 2, FORCED>;
    case 4: return (void *)atk::at_resident<T, ORDER, 4, FORCED>;
    default: return (void *)atk::at_resident<T, ORDER, 8, FORCED>;
    }
}

template <typename T>
void *by_order(int order, int ppt, bool forced)
{
    if (order == 2) return forced ? by_points<T, 2, true>(ppt) : by_points<T, 2, false>(ppt);
    return forced ? by_points<T, 4, true>(ppt) : by_points<T, 4, false>(ppt);
}
}  // namespace

// For word size w, ppt points per thread (see atk::resident_points).
__attribute__((visibility("hidden"))) void *atk_resident_kernel(int w, int order, int ppt, bool forced)
{
    return w == 8 ? by_order<double>(order, ppt, forced) : by_order<float>(order, ppt, forced);
}
