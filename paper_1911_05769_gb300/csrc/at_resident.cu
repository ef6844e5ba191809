// at_resident.cu -- instantiations of the one-subdomain-per-CTA stepper (float
// and double state, order 2 and 4, with and without forcing, 1 to 8 points per
// thread).
#include "at_resident.cuh"

namespace {
template <typename T, int ORDER, bool FORCED, bool CL>
void *by_points(int ppt)
{
    switch (ppt) {
    case 1: return (void *)atk::at_resident<T, ORDER, 1, FORCED, CL>;
    case 2: return (void *)atk::at_resident<T, ORDER, 2, FORCED, CL>;
    case 4: return (void *)atk::at_resident<T, ORDER, 4, FORCED, CL>;
    default: return (void *)atk::at_resident<T, ORDER, 8, FORCED, CL>;
    }
}

template <typename T, bool CL>
void *by_order(int order, int ppt, bool forced)
{
    if (order == 2) return forced ? by_points<T, 2, true, CL>(ppt) : by_points<T, 2, false, CL>(ppt);
    return forced ? by_points<T, 4, true, CL>(ppt) : by_points<T, 4, false, CL>(ppt);
}
}  // namespace

// For word size w, ppt points per thread (see atk::resident_points); cluster: the
// variant whose CTAs are one cluster.
__attribute__((visibility("hidden"))) void *atk_resident_kernel(int w, int order, int ppt, bool forced, bool cluster)
{
    if (cluster) return w == 8 ? by_order<double, true>(order, ppt, forced) : by_order<float, true>(order, ppt, forced);
    return w == 8 ? by_order<double, false>(order, ppt, forced) : by_order<float, false>(order, ppt, forced);
}
