// What the register-tile kernels (kernels_rt2d.cu, kernels_rt2dp.cu) share:
// vector accesses, CPML slab indices, the exact FP32 pair sum and the choice
// of the tile.
#pragma once

#include "fdtd_internal.h"
#include "launch.cuh"

namespace fdtd {

namespace {

__device__ __forceinline__ bool in_range(int v, int lo, int n) { return (unsigned)(v - lo) < (unsigned)n; }
__device__ __forceinline__ float rcp(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp(double x) { return __drcp_rn(x); }

// Slab indices of the CPML arrays (E: node positions, H: half positions); -1 outside.
__device__ __forceinline__ int slab_e(int p, int n, int np) { return p < np ? p : (p >= n - np ? p - (n - 2 * np) : -1); }
__device__ __forceinline__ int slab_h(int p, int n, int np)
{
    return p < np ? p : ((p >= n - 1 - np && p < n - 1) ? np + p - (n - 1 - np) : -1);
}

// VX adjacent words as one access (VX sizeof(R) = 8 bytes).
__device__ __forceinline__ void ldv(const float *p, float (&o)[2])
{
    const float2 t = *reinterpret_cast<const float2 *>(p);
    o[0] = t.x; o[1] = t.y;
}
__device__ __forceinline__ void stv(float *p, const float (&o)[2]) { *reinterpret_cast<float2 *>(p) = make_float2(o[0], o[1]); }
__device__ __forceinline__ void ldv(const double *p, double (&o)[1]) { o[0] = *p; }
__device__ __forceinline__ void stv(double *p, const double (&o)[1]) { *p = o[0]; }
template <typename R, int VX>
__device__ __forceinline__ void zero(R (&o)[VX])
{
#pragma unroll
    for (int v = 0; v < VX; ++v) o[v] = R(0);
}

// 16 bytes of adjacent words.
__device__ __forceinline__ void ld16(const float *p, float (&o)[4])
{
    const float4 t = *reinterpret_cast<const float4 *>(p);
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void ld16(const double *p, double (&o)[2])
{
    const double2 t = *reinterpret_cast<const double2 *>(p);
    o[0] = t.x; o[1] = t.y;
}
__device__ __forceinline__ void st16(float *p, const float (&o)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(o[0], o[1], o[2], o[3]);
}
__device__ __forceinline__ void st16(double *p, const double (&o)[2])
{
    *reinterpret_cast<double2 *>(p) = make_double2(o[0], o[1]);
}

// 8-byte asynchronous copy to shared memory.
__device__ __forceinline__ void cp8(void *s, const void *g)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(s)), "l"(g)
                 : "memory");
}

// Sum of the FP32 products of one launch (or chunk of launches) as an
// unevaluated FP32 pair (hi + lo): a node's share of the adjoint's sensitivity,
// which then goes into its FP64 accumulator.  A GB300 runs FP64 (and
// conversions to it) at 1/64 of the FP32 rate, so one FP64 product and sum per
// node and step (0.7 of 2.3 us per 316^2 adjoint step) becomes twelve FP32
// operations, and one FP64 addition per node and launch.  The product's
// rounding error is recovered by an FMA and the sum's by Knuth's two-sum; both
// join lo, which is rounded, so a launch's sum is good to about 2^-47 of its
// terms' magnitude.
//
// One factor is scaled by a power of two (PairScale; at least 1, so the scaling
// loses nothing), which keeps the tails of a wave front (1e-30 and below, at
// amplitude 1) within FP32's range; value() undoes it.  The products go with
// the square of the source's amplitude, and so does the scale (pair_scale),
// so that a strong source's products stay clear of FAR like a weak one's.
struct Pair {
    float hi, lo;
    // Products beyond FAR go into the FP64 accumulator: MAX_TERMS of them would
    // still sum to less than FP32's 2^128.  (In the band above, sums of terms
    // that each fit would overflow.)
    static constexpr float FAR = 0x1p120f;
    static constexpr int MAX_TERMS = 64;
    // The product a bs's error would be lost: it is not zero and below 2^-100;
    // or it is beyond FAR (or not a number).  Such products belong into the
    // FP64 accumulator directly.
    static __device__ __forceinline__ bool far(float a, float bs)
    {
        const float p = fabsf(__fmul_rn(a, bs));
        return (p < 0x1p-100f && a != 0.0f && bs != 0.0f) || !(p <= FAR);
    }
    __device__ __forceinline__ void add(float a, float bs)
    {
        const float p = __fmul_rn(a, bs), e = __fmaf_rn(a, bs, -p);
        const float s = __fadd_rn(hi, p), t = __fsub_rn(s, hi);
        const float r = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(p, t));
        hi = s;
        lo = __fadd_rn(lo, __fadd_rn(r, e));
    }
    __device__ __forceinline__ double value(double down) const { return ((double)hi + (double)lo) * down; }
};
static_assert(RT2D_MAX <= Pair::MAX_TERMS && RT2DP_CHUNK <= Pair::MAX_TERMS, "a pair's terms cannot overflow it");

// Halo and tile rows for an nx x ny grid on `sms` SMs: regions W columns wide,
// rpw rows per warp and at most maxw warps, halos 4 .. hmax.  The least time
// per step, where a wave of blocks costs a fixed part (launch, load, store)
// plus, per step, its rows that are still needed (th + H + 1 on average);
// `fixed` is that part in row steps.
inline Rt2DPlan rt_tile_plan(int nx, int ny, int sms, int W, int rpw, int maxw, int hmax, double fixed)
{
    Rt2DPlan best{};
    double cost = 0.0;
    for (int H = 4; H <= hmax; H += 2) {  // even: FP32 lanes hold two columns
        const int tw = W - 2 * H, bx = (nx + tw - 1) / tw;
        for (int nw = (2 * H + 2) / rpw; nw <= maxw; ++nw) {
            const int th = nw * rpw - 2 * H, by = (ny + th - 1) / th;
            const long long waves = ((long long)bx * by + sms - 1) / sms;
            const double k = (double)waves * (fixed / H + th + H + 1);
            if (best.halo == 0 || k < cost) {
                cost = k;
                best = Rt2DPlan{H, tw, th, nw, bx, by, 1};
            }
        }
    }
    return best;
}

}  // namespace
}  // namespace fdtd
