// ctu3d.cu -- FP64 and FP32 instantiations of the fused 3D corner transport
// upwind step.  Tiles: FP32 16 x 16 (512 threads, 152 KB of shared memory),
// FP64 16 x 8 (256 threads, 171 KB); one CTA per SM.
#include <algorithm>

#include "ctu3d.cuh"
#include "launchers.h"
#include "per_device.h"

namespace hydro {

namespace {

constexpr int CTU_TX = 16;
int ctu_ty(bool fp32) { return fp32 ? 16 : 8; }

// z partition of T tiles of nz planes on G resident CTAs, one per SM: 0, the
// balanced grid (equal shares of the plane-tiles, no partial last wave), or the
// planes of z-chunks, one piece per CTA, where they cost less: a piece predicts
// two planes beside its own, and a balanced CTA marches parts of two columns.  us
// per step, chunks of 8 planes and more in several waves -> balanced / one
// piece, FP32: 16^3 44 -> 18 / 17, 80^3 89 -> 78 / 73, 101x75x130 189 -> 148 /
// 152, 128^3 318 -> 253 / 292, 240^3 1702 -> 1627; FP64 balanced / one piece:
// 40^3 225 / 182, 80^3 969 / 921, 64^3 548 / 568, 128^3 3605 / 4202.
int ctu_partition(long long T, int nz, int G)
{
    if (T > G) return 0;
    const int zc = (int)((nz + G / T - 1) / (G / T));
    return zc + 2.0 <= std::max(1.0, (double)T * nz / G) + 4.0 ? zc : 0;
}

template <typename T, bool HSE, int TX, int TY, bool GZ>
cudaError_t launch_ctu(const StepArgs &a0, cudaStream_t s)
{
    auto k = ctu3d_kernel<T, HSE, TX, TY, GZ>;
    constexpr int NT = CTU3D_THREADS<T, TX, TY>;
    constexpr size_t smem = Ctu3DSmem<T, TX, TY>::bytes;
    static PerDeviceInt resident;   // resident CTAs of the balanced grid, per device
    int g = 0;
    const cudaError_t e = persistent_grid(resident, k, smem, NT, &g);
    if (e != cudaSuccess) return e;
    StepArgs a = a0;
    a.tiles_x = (a.n[0] + TX - 1) / TX;
    const long long tiles = (long long)a.tiles_x * ((a.n[1] + TY - 1) / TY);
    a.zchunk = ctu_partition(tiles, a.n[2], g);
    const dim3 grid = a.zchunk > 0 ? dim3((unsigned)tiles, (a.n[2] + a.zchunk - 1) / a.zchunk)
                                   : dim3((unsigned)std::min<long long>(g, tiles * a.n[2]));
    return launch_step<sizeof(T) == 4>(k, grid, NT, smem, s, a);
}

}  // namespace

long long ctu3d_blocks(const int n[3], bool fp32)
{
    // upper bound over chunk lengths (at least one plane per chunk)
    return (long long)((n[0] + CTU_TX - 1) / CTU_TX) * ((n[1] + ctu_ty(fp32) - 1) / ctu_ty(fp32)) * n[2];
}

cudaError_t launch_ctu3d(const StepArgs &a, cudaStream_t s, bool fp32, bool hse)
{
    // FP64: gravity along z only (always so with the background) leaves out the
    // x and y gravity terms, whose additions of zero are not folded
    if (fp32) return hse ? launch_ctu<float, true, 16, 16, false>(a, s) : launch_ctu<float, false, 16, 16, false>(a, s);
    if (hse) return launch_ctu<double, true, 16, 8, true>(a, s);
    if (a.grav[0] == 0.0 && a.grav[1] == 0.0) return launch_ctu<double, false, 16, 8, true>(a, s);
    return launch_ctu<double, false, 16, 8, false>(a, s);
}

}  // namespace hydro
