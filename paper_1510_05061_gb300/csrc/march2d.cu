// march2d.cu -- FP64 and FP32 instantiations of the marched 2D step and of the
// two Runge-Kutta stages.
#include <algorithm>

#include "launchers.h"
#include "march2d.cuh"
#include "per_device.h"

namespace hydro {

namespace {

template <typename T, int NT, int ST>
cudaError_t launch_nt(const StepArgs &a0, cudaStream_t s)
{
    auto k = march2d_kernel<T, NT, ST>;
    constexpr size_t smem = March2DSmem<T, NT>::bytes;
    static PerDeviceInt resident;   // resident CTAs, per device
    int g = 0;
    const cudaError_t e = persistent_grid(resident, k, smem, NT, &g);
    if (e != cudaSuccess) return e;
    StepArgs a = a0;
    a.tiles_x = (a.n[0] + March2DSmem<T, NT>::UX - 1) / March2DSmem<T, NT>::UX;
    const long long rows = (long long)a.tiles_x * a.n[1];
    g = (int)std::min<long long>(std::min(g, MARCH2D_MAX_CTAS), rows);
    return launch_step<true>(k, g, NT, smem, s, a);
}

template <int ST>
cudaError_t launch_st(const StepArgs &a, int nt, cudaStream_t s, bool fp32)
{
    if (!fp32) return nt == 128 ? launch_nt<double, 128, ST>(a, s) : cudaErrorInvalidValue;
    if (nt == 128) return launch_nt<float, 128, ST>(a, s);
    return nt == 256 ? launch_nt<float, 256, ST>(a, s) : cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_march2d(const StepArgs &a, int nt, cudaStream_t s, bool fp32, int stage)
{
    switch (stage) {
    case STAGE_HANCOCK: return launch_st<STAGE_HANCOCK>(a, nt, s, fp32);
    case STAGE_RK1: return launch_st<STAGE_RK1>(a, nt, s, fp32);
    case STAGE_RK2: return launch_st<STAGE_RK2>(a, nt, s, fp32);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hydro
