// hydro_device.cuh -- per-cell and per-face device arithmetic of the update.
//
// Pieces of one unsplit finite-volume step of the compressible Euler
// equations (gamma-law gas, constant gravity): boundary index mapping, the
// MC-limited PLM slope, the MUSCL-Hancock half step in primitive variables,
// the HLLC face flux, and the CTA-level max reduction.  T is double or float.
//
// Hydrostatic-background mode (HSE): the stored state is U' = U - U0(z).
// Primitives hold (rho', u, p'); totals are rho = rho0 + rho', p = p0 + p'.
// Face fluxes carry p' in the normal momentum; the background's discrete
// imbalance B_k enters the momentum update as a source.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "fp64_int.cuh"
#include "hydro_internal.h"
#include "pieces.h"

namespace hydro {

// Interior source index of coordinate g along an axis of n cells (n >= 2),
// for g in [-2, n+1]; flip is set for a mirror image (reflecting boundary).
// On a halo side (slab decomposition, z only) g in [-2, -1] or [n, n+1] is
// returned as is: those planes are stored in the buffer.
// Coordinates further out (cells of a ragged tile beyond the domain, whose
// results are never stored) are clamped into range.
template <bool HALO = false>
__device__ __forceinline__ int map_index(int g, int n, int bclo, int bchi, bool &flip)
{
    flip = false;
    // a halo side (z only): the two planes beyond the slab are stored next to it
    if constexpr (HALO)
        if ((g < 0 && bclo == BC_HALO) || (g >= n && bchi == BC_HALO)) return g;
    if (g < 0) {
        if (bclo == BC_PERIODIC) g += n;
        else if (bclo == BC_REFLECT) { g = -1 - g; flip = true; }
        else g = 0;
    } else if (g >= n) {
        if (bchi == BC_PERIODIC) g -= n;
        else if (bchi == BC_REFLECT) { g = 2 * n - 1 - g; flip = true; }
        else g = n - 1;
    }
    return min(max(g, 0), n - 1);
}

// ---- Row vectors for the staging loads.  A haloed tile row whose x range
// lies inside the grid is fetched as aligned vectors of W cells (16 bytes:
// float4 / double2; or 8 bytes: float2) instead of one 4- or 8-byte load per
// cell: vector k of the row covers the cells x0 - W + W k .. x0 - 1 + W k,
// TX / W + 2 vectors in all, so the row's halo of depth 2 is covered (with
// W = 4 also the two cells beyond it on each side, which lie in the same
// 32-byte sectors as the halo cells).  Two adjacent cells -- a pair -- are
// then written to shared memory as one 8- or 16-byte store.
template <typename T, int W> struct RowVec;
template <> struct RowVec<float, 4> { using V = float4; };
template <> struct RowVec<float, 2> { using V = float2; };
template <> struct RowVec<double, 2> { using V = double2; };

template <typename T, int W>
__device__ __forceinline__ T vec_lane(const typename RowVec<T, W>::V &v, int e)
{
    return reinterpret_cast<const T *>(&v)[e];   // e a compile-time constant: a register
}

template <typename T, int W>
__device__ __forceinline__ typename RowVec<T, W>::V ld_vec(const T *p)
{
    return __ldg(reinterpret_cast<const typename RowVec<T, W>::V *>(p));
}

// Whether the rows of a tile starting at x0, TX cells wide, can be fetched
// as vectors of W cells: the state's base and variable planes aligned to a
// vector (nx a multiple of W, so every row is), and the vectors' x range
// [x0 - W, x0 + TX + W) inside [0, nx) -- no x boundary mapping in the halo.
template <typename T, int TX, int W>
__device__ __forceinline__ bool rows_vectorisable(const void *U, int nx, long long vs, int x0)
{
    static_assert(TX % W == 0, "tile width a multiple of the vector width");
    constexpr unsigned long long align = W * sizeof(T);
    return (reinterpret_cast<unsigned long long>(U) & (align - 1)) == 0 && nx % W == 0 && vs % W == 0 &&
           x0 >= W && x0 + TX + W <= nx;
}

// Reciprocal square root, quotient and reciprocal in the working precision.
// FP64: the hardware's seed refined on the integer pipe (fp64_int.cuh), no
// FP64 instruction; FP32: the SFU approximations (rsqrtf, __fdividef: at most
// 2 ulp), well inside the FP32 path's error budget.
//
// The FP64 reciprocal square root takes normal positive arguments; the rest
// (zero, negative, subnormal, infinite, NaN) goes to CUDA's rsqrt.
__device__ __forceinline__ double rsqrt_t(double x)
{
    if (static_cast<unsigned>(__double2hiint(x)) - 0x00100000u >= 0x7fe00000u) return rsqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return __longlong_as_double(rsqrt_bits(__double_as_longlong(x), __double2hiint(y)));
}
__device__ __forceinline__ float rsqrt_t(float x) { return rsqrtf(x); }

// k / sqrt(x), k normal and positive, in one rounding and no FP64 instruction.
__device__ __forceinline__ double scaled_rsqrt(double x, double k)
{
    if (static_cast<unsigned>(__double2hiint(x)) - 0x00100000u >= 0x7fe00000u) return k * rsqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return __longlong_as_double(rsqrt_scaled_bits(__double_as_longlong(x), __double2hiint(y), __double_as_longlong(k)));
}

// FP64 reciprocal, within 0.53 ulp for every b whose reciprocal is normal;
// NaN for zero, subnormal, infinite or NaN b, and 0 from 2^1022 on.
__device__ __forceinline__ double rcp_t(double b)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    const double r = __longlong_as_double(rcp_bits(__double_as_longlong(b), __double2hiint(y)));
    const unsigned be = static_cast<unsigned>(__double2hiint(b)) & 0x7ff00000u;
    if (be - 0x00100000u < 0x7fc00000u) return r;
    return __hiloint2double((be == 0u || be == 0x7ff00000u) ? 0x7ff80000 : 0, 0);
}
__device__ __forceinline__ float rcp_t(float b) { return __fdividef(1.0f, b); }
__device__ __forceinline__ double div_t(double a, double b) { return a * rcp_t(b); }
__device__ __forceinline__ float div_t(float a, float b) { return __fdividef(a, b); }

// Conserved -> primitive pieces of the staging conversion with every
// rounding spelled out (explicit multiplies and fused multiply-adds): the
// compiler then has no contraction choices, so each staging path (row
// vectors or mapped cells, in whichever kernel) gives the same bits.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// p = (gamma - 1)(E - |m|^2 / (2 rho)) from the momentum components m, the
// velocities u = m / rho, the total energy e and gm1 = gamma - 1: |m|^2 / rho
// as u . m summed in axis order, then (gamma - 1) fma(-1/2, u . m, E).
template <typename T, int ND>
__device__ __forceinline__ T pressure_of(const T (&m)[ND], const T (&u)[ND], T e, T gm1)
{
    T k = mul_rn(u[0], m[0]);
#pragma unroll
    for (int d = 1; d < ND; ++d) k = fma_rn(u[d], m[d], k);
    return mul_rn(gm1, fma_rn(T(-0.5), k, e));
}

// The factor hllc takes for its sound speeds: gamma in FP32, sqrt(gamma) in FP64.
template <typename T>
__device__ __forceinline__ T speed_factor(const StepArgs &a)
{
    if constexpr (sizeof(T) == 4) return a.gamma_f;
    else return a.sqrt_gamma;
}

// A step constant in the kernel's precision: the FP64 value, or its FP32
// copy rounded on the host (the same value as a device-side conversion).
template <typename T>
__device__ __forceinline__ T arg_t(double d, float f)
{
    if constexpr (sizeof(T) == 4) return f;
    else return d;
}

// x > 0 (false for +-0 and for negative values).  For doubles the test is
// an integer test of the bit pattern, which keeps it off the FP64 pipe.
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }
// x / 2 of a non-negative x.  For doubles an exact halving on the integer
// pipe (one off the exponent field; the same bits as 0.5 * x for normal
// results) rather than on the FP64 pipe: 0 for x below 2^-1021, where the
// half would not be normal; infinities and NaNs are passed through.
__device__ __forceinline__ double half_nonneg(double x)
{
    const long long b = __double_as_longlong(x);
    const long long h = b >= (2ll << 52) ? b - (1ll << 52) : 0ll;
    return __longlong_as_double(b >= (0x7ffll << 52) ? b : h);
}
__device__ __forceinline__ float half_nonneg(float x) { return 0.5f * x; }
// x / 2 of any x, likewise (0 below 2^-1021).
__device__ __forceinline__ double half_signed(double x)
{
    const unsigned e = static_cast<unsigned>(__double2hiint(x)) & 0x7ff00000u;
    const long long b = __double_as_longlong(x);
    return __longlong_as_double(e == 0x7ff00000u ? b : (e >= 0x00200000u ? b - (1ll << 52) : 0ll));
}
// Sign tests for the HLLC fan branches: x >= 0 and x <= 0 as numeric
// comparisons (both zeros satisfy both), done on the bit pattern for doubles:
// x >= 0 holds for a clear sign bit and for -0 (whose pattern is the most
// negative 64-bit integer); x <= 0 holds for a set sign bit and for +0.
// A wave speed S* of -0 (reached at reflecting walls, where the two states
// are mirror images) therefore takes the left branch, as S* = +0 does.
__device__ __forceinline__ bool nonnegative(double x)
{
    const long long b = __double_as_longlong(x);
    return b >= 0 || b == (long long)0x8000000000000000ull;
}
__device__ __forceinline__ bool nonnegative(float x) { return x >= 0.0f; }
__device__ __forceinline__ bool nonpositive(double x) { return __double_as_longlong(x) <= 0; }
__device__ __forceinline__ bool nonpositive(float x) { return x <= 0.0f; }

// Minimum and maximum.  FP64: by the order of integer keys of the bit
// patterns (a sign-magnitude to two's-complement map that orders all
// non-NaN doubles, -0 below +0), on the integer pipe rather than the FP64
// pipe that bounds the FP64 step; FP32: the hardware min/max.
__device__ __forceinline__ long long order_key(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double min_t(double a, double b) { return order_key(a) <= order_key(b) ? a : b; }
__device__ __forceinline__ double max_t(double a, double b) { return order_key(a) >= order_key(b) ? a : b; }
__device__ __forceinline__ float min_t(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float max_t(float a, float b) { return fmaxf(a, b); }

// MC limiter (van Leer 1977): full-cell slope sign(dr) min(2|dl|, 2|dr|,
// |dl+dr|/2) when dl and dr have the same sign, else 0.
__device__ __forceinline__ float mc_slope(float dl, float dr)
{
    const float a = fminf(2.0f * fminf(fabsf(dl), fabsf(dr)), 0.5f * fabsf(dl + dr));
    return (dl * dr > 0.0f) ? copysignf(a, dr) : 0.0f;
}

// FP64 form, on the IEEE bit patterns with integer instructions only (for
// non-negative doubles integer order is numeric order; adding or removing 1
// in the exponent field multiplies a normal number by 2 or 1/2 exactly).
// With M >= m the magnitudes of two differences of one sign, 2 m is the
// smallest of the three candidates once M's exponent exceeds m's by three
// (then M + m > 5 m); below that the sum aligns by at most two bits, never
// cancels and rounds to nearest even from two or three extra bits, so the
// slope has the bits of the FP64 instructions (a sum below 2^-1021, without a
// normal half, gives a zero slope).  The sum was the last FP64 instruction of
// the slope, one for each variable and axis of every predicted cell.
__device__ __forceinline__ double mc_slope(double dl, double dr)
{
    using u64 = unsigned long long;
    constexpr u64 ABS = 0x7fffffffffffffffull, ONE_EXP = 1ull << 52, MANT = ONE_EXP - 1;
    const u64 bl = __double_as_longlong(dl), br = __double_as_longlong(dr);
    const u64 al = bl & ABS, ar = br & ABS;
    const bool same = static_cast<long long>(bl ^ br) >= 0 && al != 0 && ar != 0;
    const bool lt = al < ar;
    const u64 m = lt ? al : ar, M = lt ? ar : al;
    const u64 twice = m < (0x7feull << 52) ? m + ONE_EXP : m;             // 2 min(|dl|, |dr|)
    const unsigned eM = static_cast<unsigned>(M >> 52), d = eM - static_cast<unsigned>(m >> 52);
    const u64 sum = (((M & MANT) | ONE_EXP) << 2) + ((((m & MANT) | ONE_EXP) << 2) >> (d & 3));
    const unsigned c = static_cast<unsigned>(sum >> 55), sh = 2 + c;      // c: the sum's carry
    const u64 r = (sum + ((2u << c) - 1) + (static_cast<unsigned>(sum >> sh) & 1u)) >> sh;
    u64 half = (static_cast<u64>(eM + c - 2) << 52) + r;                  // |dl + dr| / 2
    half = eM + c >= 2 ? half : 0;
    const u64 a = d >= 3 || twice < half ? twice : half;
    return same ? copysign(__longlong_as_double(a), dr) : 0.0;
}

// CFL signal speed of a cell, sum_d (|u_d| + c) / dx_d, from its momenta m
// (ND components), rinv = 1/rho and sound speed c, arranged as
// (sum_d |m_d| / dx_d) / rho + c sum_d 1/dx_d (the sum of the 1/dx_d is
// loop-invariant in the callers).
template <typename T, int ND>
__device__ __forceinline__ T signal_speed(const T *m, T rinv, T c, const T (&inv_dx)[3])
{
    T a = fabs(m[0]) * inv_dx[0];
    T sidx = inv_dx[0];
#pragma unroll
    for (int d = 1; d < ND; ++d) {
        a = fma(fabs(m[d]), inv_dx[d], a);
        sidx += inv_dx[d];
    }
    return fma(rinv, a, c * sidx);
}

// A double divided by 2^k and cut to FP32 on the integer pipe (a conversion
// instruction holds the FP64 pipe like a multiply), bias = 0x38000000 + (k << 20)
// between 0x00100000 and 0x70000000: relative error below 2^-22; 0 below FP32's
// normal range, infinity beyond it and for infinities and NaN.
__device__ __forceinline__ float cut_f32(double x, int bias)
{
    const unsigned hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned v = (hi & 0x7fffffffu) - static_cast<unsigned>(bias);   // exponent rebiased, three bits above FP32's place
    unsigned f = __funnelshift_l(lo, v, 3);
    f = static_cast<int>(v) < 0x00100000 ? 0u : (v >= 0x0ff00000u ? 0x7f800000u : f);
    return __uint_as_float(f | (hi & 0x80000000u));
}

// Whether an FP64 cell's new state u (background rb, pb) is certainly
// admissible and its CFL signal speed certainly below `below` (or just
// finite, for below = infinity), from an FP32 estimate.  The grid's maximum is
// exact, so a cell below a speed some cell has reached needs no FP64
// evaluation; false only means that it has to be evaluated.
//
// The state is divided by a power of two near the cell's density (HSE: the
// background's), which changes neither velocities nor the sound speed: with r
// from 1/4 to 1e30 nothing depends on the unit of mass, and where the units of
// length and time put an intermediate near the ends of FP32's range the answer
// is false.  What is lost below:
//   conversions and roundings   1e-6 of every term, margins 1e-5 of every term;
//   flushed or subnormal k, m   2^-124, against p > 2^-63 / gamma (c2 > 2^-60, r > 1/4),
//                               whose margin is 1e-5 p, and c > 2^-30;
//   subnormal inv_dx            2^-150 times |u| < 500 c (p > slack), against
//                               sidx > 2^-110;
//   subnormal advection term    2^-149, against c sidx > 2^-100.
// Overflows give infinities or NaN, and those the answer false.
template <int ND>
__device__ __forceinline__ bool speed_below(const double (&u)[ND + 2], double rb, double pb, float gam,
                                            const float (&inv_dx)[3], float below)
{
    const int ref = __double2hiint(__double_as_longlong(rb) != 0 ? rb : u[0]) & 0x7ff00000;
    const int bias = min(max(ref - 0x07f00000, 0x00100000), 0x70000000);
    const float r0 = cut_f32(u[0], bias), rbf = cut_f32(rb, bias), pbf = cut_f32(pb, bias), e = cut_f32(u[ND + 1], bias);
    const float r = rbf + r0;
    const float rinv = __fdividef(1.0f, r);
    float m2 = 0.0f, adv = 0.0f, sidx = 0.0f;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const float m = fabsf(cut_f32(u[1 + d], bias));
        m2 = fmaf(m, m, m2);
        adv = fmaf(m, inv_dx[d], adv);
        sidx += inv_dx[d];
    }
    const float k = 0.5f * m2 * rinv;
    const float p = pbf + (gam - 1.0f) * (e - k);
    const float slack = 1e-5f * (fabsf(pbf) + gam * (fabsf(e) + k));
    const float c2 = gam * (p + slack) * rinv;
    const float csidx = c2 * rsqrtf(c2) * sidx;
    const float s = 1.00001f * fmaf(adv, rinv, csidx);
    return r > 0.25f * (fabsf(rbf) + fabsf(r0)) && r > 0.25f && r < 1e30f && p > slack && c2 > 0x1p-60f
        && csidx > 0x1p-100f && sidx > 0x1p-110f && s < below;
}

// Background seen by one cell in HSE mode (all zero in plain mode).
template <typename T>
struct CellBG {
    T rho, p;            // centre
    T drho, dp, B;       // z differences across the cell and imbalance
    T rho_lo, p_lo;      // low z face
    T rho_hi, p_hi;      // high z face
};

template <typename T, bool HSE>
__device__ __forceinline__ CellBG<T> cell_bg(const PlaneBGT<T> *bg, int k)
{
    CellBG<T> b;
    if constexpr (HSE) {
        const PlaneBGT<T> &c = bg[k + 2];
        const PlaneBGT<T> &u = bg[k + 3];
        b.rho = c.rho_c; b.p = c.p_c;
        b.drho = c.drho; b.dp = c.dp; b.B = c.B;
        b.rho_lo = c.rho_f; b.p_lo = c.p_f;
        b.rho_hi = u.rho_f; b.p_hi = u.p_f;
    } else {
        b.rho = b.p = b.drho = b.dp = b.B = T(0);
        b.rho_lo = b.p_lo = b.rho_hi = b.p_hi = T(0);
    }
    return b;
}

// The face densities and pressures c -/+ dw_d / 2 of a cell (c: the cell's
// half-step or centre state) into rp[d] = {rho_lo, rho_hi, p_lo, p_hi}, and
// whether all of them are positive once the background is added back (HSE:
// the face tables along z).  In plain mode the FP64 path skips the addition
// of the zero background (0 + x is not folded for doubles); the FP32 path
// keeps it (its measured instruction schedule).
template <typename T, int ND, bool HSE>
__device__ __forceinline__ bool face_rho_p_positive(const T (&c)[ND + 2], const T (&dw)[ND][ND + 2],
                                                    const CellBG<T> &bg, T (&rp)[ND][4])
{
    constexpr int NV = ND + 2;
    constexpr bool BGADD = HSE || sizeof(T) == 4;
    bool ok = true;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        T rb_lo = bg.rho, rb_hi = bg.rho, pb_lo = bg.p, pb_hi = bg.p;
        if (HSE && d == 2) { rb_lo = bg.rho_lo; rb_hi = bg.rho_hi; pb_lo = bg.p_lo; pb_hi = bg.p_hi; }
        rp[d][0] = c[0] - T(0.5) * dw[d][0];
        rp[d][1] = c[0] + T(0.5) * dw[d][0];
        rp[d][2] = c[NV - 1] - T(0.5) * dw[d][NV - 1];
        rp[d][3] = c[NV - 1] + T(0.5) * dw[d][NV - 1];
        const T r_lo = BGADD ? rb_lo + rp[d][0] : rp[d][0];
        const T r_hi = BGADD ? rb_hi + rp[d][1] : rp[d][1];
        const T p_lo = BGADD ? pb_lo + rp[d][2] : rp[d][2];
        const T p_hi = BGADD ? pb_hi + rp[d][3] : rp[d][3];
        ok = ok && positive(r_lo) && positive(r_hi) && positive(p_lo) && positive(p_hi);
    }
    return ok;
}

// MUSCL-Hancock half step (Toro, 3rd ed., sec. 14.4) in primitive variables
// for one cell: wh = w - (dt/2) sum_d A_d(w) dw_d / dx_d + (dt/2) S(w), where
// S(w) is gravity on the velocities.  On return dw holds the slopes used
// (all zero after the positivity fallback) and the face states are
// wh -/+ dw_d / 2; their densities and pressures, formed for the positivity
// test, are returned in rp[d] = {rho_lo, rho_hi, p_lo, p_hi} (the same
// values: the caller takes them instead of forming them again).  Returns
// true when the fallback was taken.
template <typename T, int ND, bool HSE, bool GZ = false, bool RINV = false>
__device__ __forceinline__ bool hancock(const T (&w)[ND + 2], T (&dw)[ND][ND + 2],
                                        T (&wh)[ND + 2], T (&rp)[ND][4], T hdt, const T (&inv_dx)[3],
                                        T gam, const T (&grav)[3], const CellBG<T> &bg,
                                        T rinv_given = T(0))
{
    constexpr int NV = ND + 2;
    const T rho = HSE ? bg.rho + w[0] : w[0];
    const T pr = HSE ? bg.p + w[NV - 1] : w[NV - 1];
    // RINV: 1/rho as computed when the cell was staged (the same value)
    const T rinv = RINV ? rinv_given : rcp_t(rho);
    const T gp = gam * pr;
    // A_d(w) dw_d / dx_d summed over d: rho: u_d drho_d + rho du_{d,d};
    // u_e: u_d du_{e,d} (+ dp_d / rho for e = d); p: u_d dp_d + gamma p du_{d,d}.
    // The rho and p rows take their normal-velocity terms through one
    // divergence, div u = sum_d du_{d,d} / dx_d; 1/dx_d is folded into the
    // other coefficients.
    T divu = dw[0][1] * inv_dx[0];
#pragma unroll
    for (int d = 1; d < ND; ++d) divu = fma(dw[d][1 + d], inv_dx[d], divu);
    T rate[NV];
    rate[0] = -rho * divu;
#pragma unroll
    for (int e = 0; e < ND; ++e) rate[1 + e] = T(0);
    rate[NV - 1] = -gp * divu;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const T un_dx = w[1 + d] * inv_dx[d];
        const T rinv_dx = rinv * inv_dx[d];
        rate[0] = fma(-un_dx, dw[d][0], rate[0]);
#pragma unroll
        for (int e = 0; e < ND; ++e) rate[1 + e] = fma(-un_dx, dw[d][1 + e], rate[1 + e]);
        rate[1 + d] = fma(-rinv_dx, dw[d][NV - 1], rate[1 + d]);
        rate[NV - 1] = fma(-un_dx, dw[d][NV - 1], rate[NV - 1]);
    }
    // gravity on the velocities: g rho'/rho - B/rho in HSE mode, g otherwise
    T gsrc[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) gsrc[d] = HSE ? grav[d] * (w[0] * rinv) : grav[d];
    if constexpr (HSE) {
        const T wz = w[3];
        rate[0] -= wz * bg.drho * inv_dx[2];
        rate[4] -= wz * bg.dp * inv_dx[2];
        gsrc[2] -= bg.B * rinv;
    }
    // (GZ: gravity along the last axis only -- the other axes' zero terms
    // are not added)
#pragma unroll
    for (int d = 0; d < ND; ++d)
        if (!GZ || d == ND - 1) rate[1 + d] += gsrc[d];
#pragma unroll
    for (int q = 0; q < NV; ++q) wh[q] = w[q] + hdt * rate[q];

    // positivity of every predicted face density and pressure
    const bool ok = face_rho_p_positive<T, ND, HSE>(wh, dw, bg, rp);
    if (!ok) {
#pragma unroll
        for (int d = 0; d < ND; ++d)
#pragma unroll
            for (int q = 0; q < NV; ++q) dw[d][q] = T(0);
#pragma unroll
        for (int q = 0; q < NV; ++q) wh[q] = w[q];
#pragma unroll
        for (int d = 0; d < ND; ++d)
            if (!GZ || d == ND - 1) wh[1 + d] += hdt * gsrc[d];
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            rp[d][0] = rp[d][1] = w[0];
            rp[d][2] = rp[d][3] = w[NV - 1];
        }
    }
    return !ok;
}

// Face state q of axis d (hi: the high face) of a cell after hancock or
// mol_faces (there with wh = w): the density and pressure as returned in rp,
// the velocities wh -/+ dw_d / 2.
template <typename T, int ND>
__device__ __forceinline__ T face_value(int q, int d, bool hi, const T (&wh)[ND + 2], const T (&dw)[ND][ND + 2],
                                        const T (&rp)[ND][4])
{
    if (q == 0) return rp[d][hi ? 1 : 0];
    if (q == ND + 1) return rp[d][hi ? 3 : 2];
    return hi ? wh[q] + T(0.5) * dw[d][q] : wh[q] - T(0.5) * dw[d][q];
}

// Face states of the method of lines (no predictor): w -/+ dw_d / 2, with
// the same positivity fallback as the half step (every slope of the cell
// zeroed when a face density or pressure would not be positive); rp as in
// hancock.
template <typename T, int ND, bool HSE>
__device__ __forceinline__ void mol_faces(const T (&w)[ND + 2], T (&dw)[ND][ND + 2], const CellBG<T> &bg,
                                          T (&rp)[ND][4])
{
    constexpr int NV = ND + 2;
    if (!face_rho_p_positive<T, ND, HSE>(w, dw, bg, rp)) {
#pragma unroll
        for (int d = 0; d < ND; ++d) {
#pragma unroll
            for (int q = 0; q < NV; ++q) dw[d][q] = T(0);
            rp[d][0] = rp[d][1] = w[0];
            rp[d][2] = rp[d][3] = w[NV - 1];
        }
    }
}

// Piecewise parabolic face values (Colella and Woodward 1984, uniform grid)
// of the cell with value a, face neighbours am and ap and MC-limited slopes
// sm, s, sp (cells i-1, i, i+1): interface values (a + a')/2 - (s' - s)/6,
// then the parabola limited to be monotone: flat at a local extremum, else
// a face value moved so that the parabola has no interior extremum.
template <typename T>
__device__ __forceinline__ void ppm_faces(T am, T a, T ap, T sm, T s, T sp, T &lo, T &hi)
{
    const T sixth = T(1.0 / 6.0);
    T aL = T(0.5) * (am + a) - (s - sm) * sixth;
    T aR = T(0.5) * (a + ap) - (sp - s) * sixth;
    const bool flat = (aR - a) * (a - aL) <= T(0);
    const T da = aR - aL;
    const T a6 = T(6) * (a - T(0.5) * (aL + aR));
    const T dd = da * da, d6 = da * a6;
    const bool fix_l = !flat && d6 > dd;
    const bool fix_r = !flat && !fix_l && -dd > d6;
    lo = flat ? a : (fix_l ? T(3) * a - T(2) * aR : aL);
    hi = flat ? a : (fix_r ? T(3) * a - T(2) * aL : aR);
}

// The FP64 parabola in two parts, with the limiter's tests on the bit patterns.
// ppm_interface: the interface value between cells of values am and a with
// slopes sm and s, (am + a)/2 - (s - sm)/6: 3 FP64 instructions.
__device__ __forceinline__ double ppm_interface(double am, double a, double sm, double s)
{
    return fma_rn(-1.0 / 6.0, s - sm, half_signed(am + a));
}

// ppm_limit: the face values of a cell of value a with interface values aL and
// aR.  With d1 = aR - a and d2 = a - aL the curvature and the difference of the
// parabola are a6 = 3 (d2 - d1) and aR - aL = d1 + d2, so its overshoots
// a6 (aR - aL) > (aR - aL)^2 and -(aR - aL)^2 > a6 (aR - aL) are, for d1 and d2
// of one sign, |d2| > 2 |d1| and |d1| > 2 |d2|, and the replaced values
// 3 a - 2 aR = a - 2 d1 and 3 a - 2 aL = a + 2 d2: 3 FP64 instructions where
// the products and comparisons took 16.
__device__ __forceinline__ void ppm_limit(double a, double aL, double aR, double &lo, double &hi)
{
    using u64 = unsigned long long;
    constexpr u64 ABS = 0x7fffffffffffffffull, ONE_EXP = 1ull << 52;
    const u64 b1 = __double_as_longlong(aR - a), b2 = __double_as_longlong(a - aL);
    const u64 m1 = b1 & ABS, m2 = b2 & ABS;
    const bool flat = static_cast<long long>(b1 ^ b2) < 0 || m1 == 0 || m2 == 0;
    const u64 t1 = m1 + ONE_EXP, t2 = m2 + ONE_EXP;   // 2 |d1|, 2 |d2|
    const bool fix_l = m2 > t1, fix_r = m1 > t2;
    const u64 x = fix_l ? t1 | (~b1 & ~ABS) : t2 | (b2 & ~ABS);   // -2 d1 or 2 d2
    const double v = a + __longlong_as_double(x);
    lo = flat ? a : (fix_l ? v : aL);
    hi = flat ? a : (fix_r ? v : aR);
}

// HLLC flux along axis D (Toro, 3rd ed., sec. 10.4-10.6) with Davis wave
// speeds S_L = min(u_L - c_L, u_R - c_R), S_R = max(u_L + c_L, u_R + c_R).
// wl, wr hold (rho', u, p') and (rb, pb) the background at the face; in plain
// mode rb = pb = 0.  The normal momentum flux carries p' (= p in plain mode).
// Branches: 0 <= S_L -> F_L; S_L < 0 <= S* -> F*_L; S* < 0 < S_R -> F*_R;
// S_R <= 0 -> F_R.  igm1 = 1/(gamma - 1).
//
// Arithmetic is arranged to need two square-root reciprocals and two
// divisions per face: c = g rsqrt(g rho) with g = gamma p (FP64: p times
// sqrt(gamma) / sqrt(p rho), the factor joining on the integer pipe).  The
// star state of Toro eq. (10.39) enters through F*_K = F_K + S_K (U*_K - U_K) and one
// factor h = S_K (S* - u_K) / (S_K - S*), zero outside the fan:
//   mass             F_0 = rho_K u_K + rho_K h = rho_K (u_K + h)
//   tangential       F_0 v_t
//   normal momentum  F_0 u_K + p_K + m_K h,           m_K = rho_K (S_K - u_K)
//   energy           (E_K + p_K)(u_K + h) + m_K h S*
// (S_K (rho*_K - rho_K) = rho_K h; S_K rho_K h = rho_K h u_K + m_K h.)  The
// star state is never formed, so nothing is subtracted from a nearly equal
// product, and the fan's branch needs one select (of h) beside those of the
// side.  33 instructions on the FP64 pipe per face; the same fluxes as
// separate sums F_K + correction took 44 and the roots and quotients 16 more, with the same rounding error (rms
// over random states against 128 bits: mass 4.3e-17, energy 2.6e-16 for both;
// forming the star state itself saves three more, at 1.3 and 1.8 times that error).
// Every rounding is spelled out, so that each kernel gives the same bits.
// The axis is an argument: a run-time axis (kernels whose warps mix faces of
// several axes) costs a few selects, no FP64 instruction, and gives the same
// bits.
template <int ND, bool HSE>
__device__ __forceinline__ void hllc_f64(int axis, const double (&wl)[ND + 2], const double (&wr)[ND + 2],
                                         double rb, double pb, double sgam, double igm1, double (&f)[ND + 2])
{
    constexpr int NV = ND + 2;
    const double rl = HSE ? rb + wl[0] : wl[0];
    const double rr = HSE ? rb + wr[0] : wr[0];
    const double pl = HSE ? pb + wl[NV - 1] : wl[NV - 1];
    const double pr = HSE ? pb + wr[NV - 1] : wr[NV - 1];
    const auto normal = [&](const double *v) {
        double n = v[0];
#pragma unroll
        for (int e = 1; e < ND; ++e) n = axis == e ? v[e] : n;
        return n;
    };
    const double ul = normal(wl + 1), ur = normal(wr + 1);
    const double cl = mul_rn(pl, scaled_rsqrt(mul_rn(pl, rl), sgam));
    const double cr = mul_rn(pr, scaled_rsqrt(mul_rn(pr, rr), sgam));
    // S_L - u_L = min(-c_L, (u_R - u_L) - c_R) and S_R - u_R = max(c_L - (u_R - u_L), c_R):
    // the offsets the star factors m_K = rho_K (S_K - u_K) need, and the chosen S_K
    const double du = ur - ul;
    const double al = min_t(-cl, du - cr);
    const double ar = max_t(cl - du, cr);

    // Branch-free: every face computes S* and h and the branch of the HLLC
    // fan is applied by selects.  The straight-line code lets a
    // thread's independent faces interleave.  S* and 1/(S_K - S*) are finite
    // for positive densities and pressures (S_L < u_L, S_R > u_R).
    const double dpp = wr[NV - 1] - wl[NV - 1];   // background cancels in the difference
    const double ml = mul_rn(rl, al), mr = mul_rn(rr, ar);
    const double sstar = div_t(fma_rn(-mr, ur, fma_rn(ml, ul, dpp)), ml - mr);
    // S_L = u_L + a_l >= 0: the whole fan moves right, F_L; S_R = u_R + a_r <= 0:
    // left, F_R (comparisons of the terms: the rounded sums have these signs)
    const bool sup_l = order_key(ul) >= order_key(-al);
    const bool sup_r = order_key(ur) <= order_key(-ar);
    const bool left = sup_l || (!sup_r && nonnegative(sstar));
    const bool star = !sup_l && !sup_r;
    const double rk = left ? rl : rr;
    const double pk = left ? pl : pr;
    const double ppk = left ? wl[NV - 1] : wr[NV - 1];
    const double mk = left ? ml : mr;
    double vk[ND];
#pragma unroll
    for (int e = 0; e < ND; ++e) vk[e] = left ? wl[1 + e] : wr[1 + e];
    const double uk = left ? ul : ur;
    const double sk = uk + (left ? al : ar);
    double ke = mul_rn(vk[0], vk[0]);
#pragma unroll
    for (int e = 1; e < ND; ++e) ke = fma_rn(vk[e], vk[e], ke);
    // E_K + p_K = p_K gamma / (gamma - 1) + rho_K |v_K|^2 / 2
    const double hk = fma_rn(pk, igm1 + 1.0, mul_rn(rk, half_nonneg(ke)));
    const double hs = mul_rn(sstar - uk, mul_rn(sk, rcp_t(sk - sstar)));
    const double h = star ? hs : 0.0;
    const double uh = uk + h, g = mul_rn(mk, h), pg = ppk + g;
    f[0] = mul_rn(rk, uh);
#pragma unroll
    for (int e = 0; e < ND; ++e) f[1 + e] = fma_rn(f[0], vk[e], axis == e ? pg : 0.0);
    f[NV - 1] = fma_rn(hk, uh, mul_rn(g, sstar));
}

// The FP32 flux: F_K plus the correction S_K (U*_K - U_K) in multiples of the
// same h, the components' increments added one by one.  (The FP64 grouping
// saves nothing here: 0 to 1 % of the step, with other bits.)
template <int ND, int D, bool HSE>
__device__ __forceinline__ void hllc_f32(const float (&wl)[ND + 2], const float (&wr)[ND + 2], float rb, float pb,
                                         float gam, float igm1, float (&f)[ND + 2])
{
    constexpr int NV = ND + 2;
    const float rl = HSE ? rb + wl[0] : wl[0];
    const float rr = HSE ? rb + wr[0] : wr[0];
    const float pl = HSE ? pb + wl[NV - 1] : wl[NV - 1];
    const float pr = HSE ? pb + wr[NV - 1] : wr[NV - 1];
    const float ul = wl[1 + D], ur = wr[1 + D];
    const float gpl = gam * pl, gpr = gam * pr;
    const float cl = gpl * rsqrt_t(gpl * rl);
    const float cr = gpr * rsqrt_t(gpr * rr);
    // S_L - u_L = min(-c_L, (u_R - u_L) - c_R) and S_R - u_R = max(c_L - (u_R - u_L), c_R):
    // the offsets the star factors m_K = rho_K (S_K - u_K) need, and S_L, S_R from them
    const float du = ur - ul;
    const float al = min_t(-cl, du - cr);
    const float ar = max_t(cl - du, cr);
    const float sl = ul + al, sr = ur + ar;

    // Branch-free: every face computes S* and the star correction and the
    // branch of the HLLC fan is applied by selects.  The chosen branch's
    // values are the same as with branches, and the straight-line code lets
    // a thread's independent faces interleave.  S* and 1/(S_K - S*) are
    // finite for positive densities and pressures (S_L < u_L, S_R > u_R).
    const float dpp = wr[NV - 1] - wl[NV - 1];   // background cancels in the difference
    const float ml = rl * al, mr = rr * ar;
    const float sstar = div_t(dpp + ml * ul - mr * ur, ml - mr);
    const bool sup_l = nonnegative(sl);     // whole fan moves right: F_L
    const bool sup_r = nonpositive(sr);     // whole fan moves left: F_R
    const bool left = sup_l || (!sup_r && nonnegative(sstar));
    const bool star = !sup_l && !sup_r;
    const float rk = left ? rl : rr;
    const float pk = left ? pl : pr;
    const float ppk = left ? wl[NV - 1] : wr[NV - 1];
    const float sk = left ? sl : sr;
    const float mk = left ? ml : mr;
    float vk[ND];
#pragma unroll
    for (int e = 0; e < ND; ++e) vk[e] = left ? wl[1 + e] : wr[1 + e];
    const float uk = vk[D];
    float ke = 0.0f;
#pragma unroll
    for (int e = 0; e < ND; ++e) ke += vk[e] * vk[e];
    // E_K + p_K = p_K gamma / (gamma - 1) + rho_K |v_K|^2 / 2
    const float hk = fma(pk, igm1 + 1.0f, rk * half_nonneg(ke));

    // Euler flux of the chosen side
    const float mflux = rk * uk;
    f[0] = mflux;
#pragma unroll
    for (int e = 0; e < ND; ++e) f[1 + e] = mflux * vk[e];
    f[1 + D] += ppk;
    f[NV - 1] = uk * hk;

    // F*_K = F_K + S_K (U*_K - U_K), applied only inside the fan
    const float h = (sk * rcp_t(sk - sstar)) * (sstar - uk);
    const float c0 = rk * h;                    // S_K (rho*_K - rho_K)
    const float fE = fma(h, fma(mk, sstar, hk), f[NV - 1]);
    const float cs = star ? c0 : 0.0f;
    f[0] += cs;
#pragma unroll
    for (int e = 0; e < ND; ++e) f[1 + e] = fma(cs, (e == D) ? sk : vk[e], f[1 + e]);
    f[NV - 1] = star ? fE : f[NV - 1];
}

// sgam: speed_factor<T>.
template <typename T, int ND, int D, bool HSE>
__device__ __forceinline__ void hllc(const T (&wl)[ND + 2], const T (&wr)[ND + 2], T rb, T pb, T sgam, T igm1,
                                     T (&f)[ND + 2])
{
    if constexpr (sizeof(T) == 8) hllc_f64<ND, HSE>(D, wl, wr, rb, pb, sgam, igm1, f);
    else hllc_f32<ND, D, HSE>(wl, wr, rb, pb, sgam, igm1, f);
}

// Mirror image of a face state across a wall normal to axis D.
template <typename T, int NV, int D>
__device__ __forceinline__ void mirror_state(const T (&src)[NV], T (&dst)[NV])
{
#pragma unroll
    for (int q = 0; q < NV; ++q) dst[q] = src[q];
    dst[1 + D] = -src[1 + D];
}

// Max over the CTA of a double (every thread passes its value; the result is
// valid in thread 0).  red must hold 32 doubles.
template <int NT>
__device__ __forceinline__ double block_max(double v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < NT / 32 ? red[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    return v;
}

// The same max taken in the working precision (max is exact in any
// precision), widened to FP64 once: an FP32 step keeps the reduction off the
// FP64 pipe.  red must hold 32 doubles.
template <int NT, typename T>
__device__ __forceinline__ double block_max_t(T v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    T *r = reinterpret_cast<T *>(red);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) r[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < NT / 32 ? r[lane] : T(0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    return double(v);
}

// First act of a step kernel (launch_step): waits for the kernel before it in
// the stream to end, its writes visible.  Nothing of the previous step is read
// before the wait; without a chained launch it is a no-op.  The next kernel's
// CTAs are let in as this one's exit, not by an earlier
// griddepcontrol.launch_dependents: placed while this kernel's CTAs still
// hold their slots, they pile up on the slots a grid of less than full
// residency leaves open, and the SMs then get unequal shares (FP32, us per
// step, early -> at exit: 288 CTAs of 96^3 on 456 slots 75.3 -> 58.2, 256 of 64^3
// 33.9 -> 27.7, 2D 384^2 12.2 -> 10.7; full grids gain 0 to 2 %).
__device__ __forceinline__ void chain_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Last-CTA finalisation of a step's time control.  Each of the nblocks
// contributions (CTAs, or work items of one instance) calls it once with its
// max signal speed (valid in thread 0), whether any of its cells failed the
// admissibility check, and its slot `part` in a.partial, after storing its
// part of the new state.
// The CTA that arrives last takes the grid maximum (max is exact, so arrival
// order does not matter), commits the error bits, sets the next dt in FP64
// and advances time.  advance = false only recomputes dt (initialisation).
// Only this CTA writes the fields that every CTA reads at kernel start, and
// it does so after all CTAs have read them.
template <int NT>
__device__ __forceinline__ void finish_step(double smax_cta, bool bad_cta, const StepArgs &a,
                                            int nblocks, int part, double dt_used, bool advance,
                                            int *s_last)
{
    if (threadIdx.x == 0) {
        if (bad_cta) atomicOr(&a.ctrl->err_new, 1);
        a.partial[part] = smax_cta;
        __threadfence();
        const unsigned prev = atomicAdd(&a.ctrl->counter, 1u);
        *s_last = (prev == (unsigned)(nblocks - 1));
    }
    __syncthreads();
    if (!*s_last) return;
    __threadfence();
    double m = 0.0;
    for (int i = threadIdx.x; i < nblocks; i += NT) m = fmax(m, __ldcg(a.partial + i));
    __shared__ double red2[32];
    m = block_max<NT>(m, red2);
    if (threadIdx.x == 0) {
        Ctrl *C = a.ctrl;
        if (advance) {
            const double t = C->t;
            C->t = (dt_used >= a.t_end - t) ? a.t_end : t + dt_used;
            C->dt_last = dt_used;
            C->step = C->step + 1;
        }
        int e = atomicExch(&C->err_new, 0);
        if (!(m > 0.0) || !isfinite(m)) e |= 1;
        C->err |= e;
        C->max_speed = m;
        C->dt_next = m > 0.0 ? a.cfl / m : 0.0;
        C->counter = 0u;
        C->reached = 0;
        __threadfence();
    }
}

// Next work item of a persistent batched launch from list L of the queue
// for this launch's parity (valid in every thread), or -1 when the list is
// exhausted.  The CTA that is last to find the list exhausted resets the
// counters (every other CTA has stopped claiming by then), so the next
// launch of this parity starts from item 0.  Every thread must call it.
__device__ __forceinline__ int claim_item(BatchQueue *q, int L, int parity, int *s_it, int next = -1)
{
    if (threadIdx.x == 0 && next >= 0) {
        *s_it = next;
    } else if (threadIdx.x == 0) {
        const int n = q->nitems[L];
        int it = (int)atomicAdd(&q->next[L][parity], 1u);
        if (it >= n) {
            it = -1;
            if (atomicAdd(&q->exited[L][parity], 1u) == gridDim.x - 1) {
                q->next[L][parity] = 0u;
                q->exited[L][parity] = 0u;
                __threadfence();
            }
        }
        *s_it = it;
    }
    __syncthreads();
    return *s_it;
}

}  // namespace hydro
