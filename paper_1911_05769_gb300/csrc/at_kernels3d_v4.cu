// at_kernels3d_v4.cu -- instantiations of the FP32 3D stepper with 4-point
// groups (at_kernels3d_v4.cuh): the scalar equation (equal or unequal spacing)
// and the system of 3, 4 or 5 fields, in CTAs of 32 to 256 threads.
#include "at_kernels3d_v4.cuh"

namespace {
template <int NT, int TC, int TEAMS>
void *v4_scalar(bool iso)
{
    return iso ? (void *)atk::at_stepper3d_v4<1, false, NT, TC, true, TEAMS>
               : (void *)atk::at_stepper3d_v4<1, false, NT, TC, false, TEAMS>;
}

template <int NT, int CTAS = atk::v4_min_ctas(3, NT)>
void *v4_system(int nf)
{
    return nf == 3 ? (void *)atk::at_stepper3d_v4<3, true, NT, 1, false, 1, CTAS>
                   : nf == 4 ? (void *)atk::at_stepper3d_v4<4, true, NT, 1, false, 1, CTAS>
                             : (void *)atk::at_stepper3d_v4<5, true, NT, 1, false, 1, CTAS>;
}
}  // namespace

// nf fields (1: the scalar equation), CTAs of `teams` teams of nt threads (32, 64,
// 128, 256; the scalar equation: 1 to 256 / nt teams, with tc = 2 groups per thread
// one team of 128; the system: one team, or with teams = 2 the 256-thread kernel
// compiled for two CTAs an SM).
__attribute__((visibility("hidden"))) void *atk_stepper3d_v4_kernel(int nf, int nt, int tc, int teams, int iso)
{
    if (nf > 1) return nt == 32 ? v4_system<32>(nf) : nt == 64 ? v4_system<64>(nf) : nt == 128 ? v4_system<128>(nf)
                                : teams == 1 ? v4_system<256>(nf) : v4_system<256, 2>(nf);
    if (tc == 2) return v4_scalar<128, 2, 1>(iso);
    switch (nt * 16 + teams) {
    case 32 * 16 + 8: return v4_scalar<32, 1, 8>(iso);
    case 32 * 16 + 4: return v4_scalar<32, 1, 4>(iso);
    case 32 * 16 + 2: return v4_scalar<32, 1, 2>(iso);
    case 32 * 16 + 1: return v4_scalar<32, 1, 1>(iso);
    case 64 * 16 + 4: return v4_scalar<64, 1, 4>(iso);
    case 64 * 16 + 2: return v4_scalar<64, 1, 2>(iso);
    case 64 * 16 + 1: return v4_scalar<64, 1, 1>(iso);
    case 128 * 16 + 2: return v4_scalar<128, 1, 2>(iso);
    default: return v4_scalar<128, 1, 1>(iso);
    }
}
