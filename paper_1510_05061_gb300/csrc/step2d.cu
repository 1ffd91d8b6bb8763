// step2d.cu -- FP64 and FP32 instantiations of the fused 2D step and of
// the two Runge-Kutta stages, tile by tile, and the choice of the launch shape.
#include "launchers.h"
#include "per_device.h"
#include "plan.h"
#include "step2d.cuh"

namespace hydro {

namespace {

template <typename T, int TX, int TY, int ST, int RC>
cudaError_t launch2d(const StepArgs &a0, cudaStream_t s)
{
    auto k = step2d_kernel<T, TX, TY, ST, RC>;
    constexpr size_t smem = Step2DSmem<T, TX, TY, RC>::bytes;
    static PerDeviceOnce configured;   // the attribute is per function and device
    const cudaError_t e = ensure_smem_limit(configured, k, smem);
    if (e != cudaSuccess) return e;
    StepArgs a = a0;
    a.tiles_x = (a.n[0] + TX - 1) / TX;
    return launch_step<true>(k, a.tiles_x * ((a.n[1] + TY - 1) / TY), TX * TY, smem, s, a);
}

template <int ST, int RC>
cudaError_t launch2d_p(const StepArgs &a, cudaStream_t s, bool fp32)
{
    const Plan2D p = plan2d(a.n[0], a.n[1], fp32, RC == RECON_PPM);
    if constexpr (RC == RECON_PLM)
        if (p.march) return launch_march2d(a, p.march, s, fp32, ST);
    if (fp32) {
        if constexpr (RC == RECON_PPM) return launch2d<float, 16, 16, ST, RC>(a, s);
        else return launch2d<float, 32, 16, ST, RC>(a, s);
    }
    return p.ty == 8 ? launch2d<double, 16, 8, ST, RC>(a, s) : launch2d<double, 16, 16, ST, RC>(a, s);
}

}  // namespace

cudaError_t launch_step2d(const StepArgs &a, cudaStream_t s, bool fp32, int stage, int recon)
{
    if (recon == RECON_PPM) {
        if (stage == STAGE_RK1) return launch2d_p<STAGE_RK1, RECON_PPM>(a, s, fp32);
        if (stage == STAGE_RK2) return launch2d_p<STAGE_RK2, RECON_PPM>(a, s, fp32);
        return cudaErrorInvalidValue;
    }
    switch (stage) {
    case STAGE_HANCOCK: return launch2d_p<STAGE_HANCOCK, RECON_PLM>(a, s, fp32);
    case STAGE_RK1: return launch2d_p<STAGE_RK1, RECON_PLM>(a, s, fp32);
    case STAGE_RK2: return launch2d_p<STAGE_RK2, RECON_PLM>(a, s, fp32);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hydro
