// march2d.cuh -- the fused 2D step for a column strip marched along y.
//
// A CTA of NT threads owns a strip of NT - 4 columns, one thread per column
// with two halo columns on either side, and marches up the rows of its piece.
// Per row p it
//   1. takes the row's primitives (own column in registers, the neighbours'
//      through shared memory) and forms the MC slopes and the half step, or
//      the stage's face states, of every column;
//   2. evaluates the HLLC flux of the column's low x face and of the y face
//      p - 1/2 (the lower state kept in registers from the row before);
//   3. completes row p - 1 and loads the row after next.
// Each row is staged, converted and predicted once per strip and each face
// solved once, against 1.41 to 1.88 conversions, 1.19 to 1.38 predictions and
// 1.05 to 1.09 face passes per cell of the tiles (step2d.cuh); a strip repeats
// 4 of NT columns and two predicted rows per piece, so it pays on large grids
// (plan2d in plan.h).  What bounds it is what bounds the tiles: the FP64 pipe,
// or instruction issue in FP32.  Measured on GB300, us per MUSCL-Hancock step:
// FP32 2048^2 128.7 (32 x 16 tile) -> 101, 1448^2 67.4 -> 53.3;
// FP64 1448^2 1114 (16 x 16 tile) -> 965.  Linear states only: the parabolic
// stages' five rows in registers cost what the march saves (FP32 1448^2 179 us
// a step for both, FP64 724^2 1048 against 1072).
#pragma once

#include "hydro_device.cuh"

namespace hydro {

template <typename T, int NT>
struct March2DSmem {
    static constexpr int NV = 4;
    static constexpr int H = 2;             // halo columns on either side
    static constexpr int UX = NT - 2 * H;   // columns the strip updates
    static constexpr size_t row = (size_t)NV * NT;
    static constexpr size_t elems = 4 * row;   // primitives of two rows, x high states, x fluxes
    static constexpr size_t bytes = elems * sizeof(T);
};

// One piece: strip `strip`, rows [r0, r1), time step dtd.  ST as in
// step3d_body; the same arithmetic per cell and face as step2d_body, in the
// same order, so the same bits.
template <typename T, int NT, int ST = STAGE_HANCOCK>
__device__ __forceinline__ void march2d_body(const StepArgs &a, int strip, int r0, int r1, double dtd,
                                             unsigned char *smem_raw, T &smax, bool &bad)
{
    constexpr int ND = 2, NV = 4;
    using S = March2DSmem<T, NT>;
    constexpr int H = S::H;
    T *prim = reinterpret_cast<T *>(smem_raw);   // [2][NV][NT]
    T *xhi = prim + 2 * S::row, *fxs = xhi + S::row;

    const int nx = a.n[0], ny = a.n[1];
    const int t = threadIdx.x;
    const int gx = strip * S::UX - H + t;
    const int tl = max(t - 1, 0), tr = min(t + 1, NT - 1);
    const bool own = t >= H && t < NT - H && gx < nx;
    const T *__restrict__ U = static_cast<const T *>(a.U);
    const T *__restrict__ U0 = static_cast<const T *>(a.U0);
    T *__restrict__ Un = static_cast<T *>(a.Unew);
    const long long vs = a.vstride;
    const T dt = T(dtd), hdt = T(0.5) * T(dtd);
    const T gam = arg_t<T>(a.gamma, a.gamma_f);
    const T igm1 = arg_t<T>(1.0 / (a.gamma - 1.0), a.igm1_f), sgam = speed_factor<T>(a);
    const T inv_dx[3] = {arg_t<T>(a.inv_dx[0], a.inv_dx_f[0]), arg_t<T>(a.inv_dx[1], a.inv_dx_f[1]), T(0)};
    const T grav[3] = {arg_t<T>(a.grav[0], a.grav_f[0]), arg_t<T>(a.grav[1], a.grav_f[1]), T(0)};
    const CellBG<T> nobg = cell_bg<T, false>(static_cast<const PlaneBGT<T> *>(nullptr), 0);

    bool fx;
    const int sx = map_index(gx, nx, a.bc_lo[0], a.bc_hi[0], fx);

    // the column's conserved values of row r (boundary index mapping), and
    // their primitives (mirrored momenta negated)
    auto load = [&](int r, T (&v)[NV]) {
        bool fy;
        const int sy = map_index(r, ny, a.bc_lo[1], a.bc_hi[1], fy);
        const T *src = U + (sy * nx + sx);   // a plane holds fewer than 2^31 cells
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = src[q * vs];
        if (fx) v[1] = -v[1];
        if (fy) v[2] = -v[2];
    };
    auto convert = [&](const T (&v)[NV], T (&w)[NV]) {
        const T rinv = rcp_t(v[0]);
        const T m[2] = {v[1], v[2]};
        const T u[2] = {mul_rn(m[0], rinv), mul_rn(m[1], rinv)};
        w[0] = v[0];
        w[1] = u[0];
        w[2] = u[1];
        w[3] = pressure_of<T, 2>(m, u, v[3], gam - T(1));
    };
    auto P = [&](int row, int q, int i) -> T & { return prim[((row & 1) * NV + q) * NT + i]; };

    // rows p and p + 1 of the column, the conserved row p + 2 in flight, the y
    // difference below row p, and what row p - 1 left
    T w[NV], wn[NV], raw[NV], dz[NV];
    T ytop_prev[NV], fy_prev[NV], fxd_prev[NV], fxm_prev = T(0);
#pragma unroll
    for (int q = 0; q < NV; ++q) { ytop_prev[q] = T(0); fy_prev[q] = T(0); fxd_prev[q] = T(0); }
    smax = T(0);
    bad = false;

    // FP64: a signal speed some cell of the step has reached (step3d_body)
    constexpr bool PRUNE = sizeof(T) == 8;
    __shared__ int s_reached;
    if (PRUNE && t == 0) s_reached = *const_cast<volatile int *>(&a.ctrl->reached);

    load(r0 - 2, raw);
    convert(raw, wn);
    load(r0 - 1, raw);
    convert(raw, w);
    load(r0, raw);
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        dz[q] = w[q] - wn[q];
        P(r0 - 1, q, t) = w[q];
    }
    convert(raw, wn);
    load(r0 + 1, raw);
    __syncthreads();

    for (int p = r0 - 1; p <= r1; ++p) {
        const bool xr = p >= r0 && p < r1;   // the row's x faces are needed
        const bool fin = p > r0 && own;      // row p - 1 is completed at the end
        T ufin[NV], u0fin[NV];
        const int cfin = (p - 1) * nx + gx;
        if (fin) {
#pragma unroll
            for (int q = 0; q < NV; ++q) ufin[q] = U[cfin + q * vs];
            if constexpr (ST == STAGE_RK2) {
#pragma unroll
                for (int q = 0; q < NV; ++q) u0fin[q] = U0[cfin + q * vs];
            }
        }

        // ---- face states of the row's cells
        T xlo[NV], ylo[NV], ytop[NV];
        {
            T dw[ND][NV], wh[NV], rp[ND][4];
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                dw[0][q] = mc_slope(w[q] - P(p, q, tl), P(p, q, tr) - w[q]);
                const T dr = wn[q] - w[q];
                dw[1][q] = mc_slope(dz[q], dr);
                dz[q] = dr;
            }
            if constexpr (ST == STAGE_HANCOCK) {
                hancock<T, ND, false>(w, dw, wh, rp, hdt, inv_dx, gam, grav, nobg);
            } else {
                mol_faces<T, ND, false>(w, dw, nobg, rp);
#pragma unroll
                for (int q = 0; q < NV; ++q) wh[q] = w[q];
            }
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                ylo[q] = face_value<T, ND>(q, 1, false, wh, dw, rp);
                ytop[q] = face_value<T, ND>(q, 1, true, wh, dw, rp);
                xlo[q] = face_value<T, ND>(q, 0, false, wh, dw, rp);
                if (xr) xhi[q * NT + t] = face_value<T, ND>(q, 0, true, wh, dw, rp);
            }
        }
        // the next row for the neighbours (its buffer was last read before the
        // previous iteration's barriers)
#pragma unroll
        for (int q = 0; q < NV; ++q) P(p + 1, q, t) = wn[q];
        __syncthreads();

        // ---- fluxes: the column's low x face, and the y face below the row.
        // Reflecting walls replace the far-side state by the mirror of the
        // near side's.
        T fy[NV], fxv[NV];
        {
            const bool w_lo = p == 0 && a.bc_lo[1] == BC_REFLECT, w_hi = p == ny && a.bc_hi[1] == BC_REFLECT;
            T wl[NV], wr[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                wl[q] = w_lo ? (q == 2 ? -ylo[q] : ylo[q]) : ytop_prev[q];
                wr[q] = w_hi ? (q == 2 ? -ytop_prev[q] : ytop_prev[q]) : ylo[q];
            }
            if (xr) {
                const bool xw_lo = gx == 0 && a.bc_lo[0] == BC_REFLECT, xw_hi = gx == nx && a.bc_hi[0] == BC_REFLECT;
                T wlx[NV], wrx[NV];
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    const T xl = xhi[q * NT + tl];
                    wlx[q] = xw_lo ? (q == 1 ? -xlo[q] : xlo[q]) : xl;
                    wrx[q] = xw_hi ? (q == 1 ? -xl : xl) : xlo[q];
                }
                hllc<T, ND, 0, false>(wlx, wrx, T(0), T(0), sgam, igm1, fxv);
#pragma unroll
                for (int q = 0; q < NV; ++q) fxs[q * NT + t] = fxv[q];
            }
            if (p >= r0) hllc<T, ND, 1, false>(wl, wr, T(0), T(0), sgam, igm1, fy);
            else {
#pragma unroll
                for (int q = 0; q < NV; ++q) fy[q] = T(0);
            }
        }
        __syncthreads();

        // ---- complete row p - 1: update, admissibility, CFL signal speed
        if (fin) {
            T u[NV], du[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                u[q] = ufin[q];
                du[q] = -(fxd_prev[q] * inv_dx[0] + (fy[q] - fy_prev[q]) * inv_dx[1]);
            }
            const T msrc = grav[0] * T(0.5) * fxm_prev + grav[1] * T(0.5) * (fy_prev[0] + fy[0]);
            const T r_old = u[0];
            const T r_new = r_old + dt * du[0];
            u[0] = r_new;
            const T rsum = ST == STAGE_HANCOCK ? T(0.5) * (r_old + r_new) : r_old;
            u[1] += dt * (du[1] + grav[0] * rsum);
            u[2] += dt * (du[2] + grav[1] * rsum);
            u[3] += dt * (du[3] + msrc);
            if constexpr (ST == STAGE_RK2) {
#pragma unroll
                for (int q = 0; q < NV; ++q) u[q] = T(0.5) * (u0fin[q] + u[q]);
            }
#pragma unroll
            for (int q = 0; q < NV; ++q) Un[cfin + q * vs] = u[q];
            // (FP64: only of the cells that could raise the maximum the CTA knows)
            bool skip = false;
            if constexpr (PRUNE)
                skip = speed_below<2>(u, 0.0, 0.0, a.gamma_f, a.inv_dx_f,
                                      ST == STAGE_RK1 ? INFINITY : __int_as_float(*const_cast<volatile int *>(&s_reached)));
            if (!skip) {
                const T rinv = rcp_t(u[0]);
                const T pres = (gam - T(1)) * (u[3] - half_nonneg(u[1] * u[1] + u[2] * u[2]) * rinv);
                const T gp = gam * pres;
                const T cs = gp * rsqrt_t(gp * u[0]);
                const T s = signal_speed<T, 2>(u + 1, rinv, cs, inv_dx);
                if (!(u[0] > T(0)) || !(pres > T(0)) || !isfinite(s)) bad = true;
                else if (!PRUNE) smax = max_t(smax, s);
                else if (s > smax) {
                    smax = s;
                    if constexpr (PRUNE && ST != STAGE_RK1) atomicMax(&s_reached, __float_as_int(__double2float_rd(s)));
                }
            }
        }
        // the maximum reached is shared with the other CTAs after the piece's first rows
        if constexpr (PRUNE && ST != STAGE_RK1)
            if (t == 0 && p > r0 && p <= r0 + 2)
                atomicMax(&s_reached, atomicMax(&a.ctrl->reached, *const_cast<volatile int *>(&s_reached)));
        if (xr) {
#pragma unroll
            for (int q = 0; q < NV; ++q) fxd_prev[q] = fxs[q * NT + tr] - fxv[q];
            fxm_prev = fxv[0] + fxs[tr];
        }
#pragma unroll
        for (int q = 0; q < NV; ++q) { ytop_prev[q] = ytop[q]; fy_prev[q] = fy[q]; }
        if (p < r1) {
            // row p + 2 enters the registers, the one after it is requested
#pragma unroll
            for (int q = 0; q < NV; ++q) w[q] = wn[q];
            convert(raw, wn);
            if (p + 3 <= r1 + 1) load(p + 3, raw);
        }
    }
}

// Resident warps asked of the FP32 kernel: 24 per SM (80 registers; 108
// registers and 16 warps: 132.6 us at 2048^2, 32 warps with spills: 113); 12 of
// the FP64 kernel (168 registers).
template <typename T, int NT, int ST = STAGE_HANCOCK>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 ? 768 : 384) / NT) march2d_kernel(const StepArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[32];
    __shared__ int s_last;
    chain_begin();
    const double t_now = a.ctrl->t;
    const double dt_cfl = a.ctrl->dt_next;
    // frozen: nothing moves (the host finds the current buffer from the step count)
    if (t_now >= a.t_end || a.ctrl->err != 0 || a.ctrl->step >= a.step_end) return;
    const double dtd = (dt_cfl >= a.t_end - t_now) ? a.t_end - t_now : dt_cfl;
    T smax = T(0);
    bool bad = false;
    // the CTA's share of the strips' rows (PieceIter over whole strips)
    PieceIter pieces(0, a.tiles_x, a.n[1], 0, 0, gridDim.x, blockIdx.x);
    int strip, r0, r1;
    bool first = true;
    while (pieces.next(strip, r0, r1)) {
        if (!first) __syncthreads();   // the next piece reuses shared memory
        first = false;
        T sm;
        bool bd;
        march2d_body<T, NT, ST>(a, strip, r0, r1, dtd, smem_raw, sm, bd);
        smax = max_t(smax, sm);
        bad = bad || bd;
    }
    const bool bad_cta = __syncthreads_or(bad) != 0;
    if constexpr (ST == STAGE_RK1) {
        if (bad_cta && threadIdx.x == 0) atomicOr(&a.ctrl->err_new, 1);
        return;
    }
    const double m = block_max_t<NT, T>(smax, red);
    finish_step<NT>(m, bad_cta, a, gridDim.x, blockIdx.x, dtd, true, &s_last);
}

}  // namespace hydro
