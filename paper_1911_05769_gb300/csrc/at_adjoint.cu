// at_adjoint.cu -- instantiations of the adjoint interval kernels (float and
// double state, stencil order 2 and 4).
#include "at_adjoint.cuh"

// Adjoint kernel (one checkpoint interval per launch) for word size w (4 or
// 8) and stencil order 2|4.
__attribute__((visibility("hidden"))) void *atk_adjoint_kernel(int w, int order)
{
    if (w == 8) return order == 2 ? (void *)atk::at_adjoint_interval<double, 2> : (void *)atk::at_adjoint_interval<double, 4>;
    return order == 2 ? (void *)atk::at_adjoint_interval<float, 2> : (void *)atk::at_adjoint_interval<float, 4>;
}

namespace {
template <typename T, int ORDER, bool FULL>
void *warp_gw(int gw)
{
    return gw == 1 ? (void *)atk::at_adjoint_warp<T, ORDER, 1, FULL>
                   : gw == 2 ? (void *)atk::at_adjoint_warp<T, ORDER, 2, FULL>
                   : gw == 4 ? (void *)atk::at_adjoint_warp<T, ORDER, 4, FULL>
                             : (void *)atk::at_adjoint_warp<T, ORDER, 8, FULL>;
}

template <typename T>
void *warp_kernel(int order, int gw, bool full)
{
    if (order == 2) return full ? warp_gw<T, 2, true>(gw) : warp_gw<T, 2, false>(gw);
    return full ? warp_gw<T, 4, true>(gw) : warp_gw<T, 4, false>(gw);
}
}  // namespace

// The one-subdomain-per-warp kernel for gw groups of 4 points per lane, whole
// runs (full) or not.
__attribute__((visibility("hidden"))) void *atk_adjoint_warp_kernel(int w, int order, int gw, bool full)
{
    return w == 8 ? warp_kernel<double>(order, gw, full) : warp_kernel<float>(order, gw, full);
}
