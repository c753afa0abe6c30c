// What the register-tile kernels (kernels_rt2d.cu, kernels_rt2dp.cu) share:
// vector accesses, CPML slab indices, the FP32 sums of products and the choice
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
// unevaluated sum of three FP32 words: a node's share of the adjoint's
// sensitivity, which then goes into its FP64 accumulator.  A GB300 runs FP64
// (and conversions to it) at 1/64 of the FP32 rate, so one FP64 product and sum
// per node and step (0.7 of 2.3 us per 316^2 adjoint step) becomes twelve FP32
// operations, and one FP64 addition per node and launch.
//
// hi is the running sum; what it loses is recovered, the product's rounding
// error by an FMA and the sum's by Knuth's two-sum, and added up in words of
// their own.  lo, the sums' errors, seldom rounds at all (each is a few units
// of hi's last places); c, the products', rounds at 2^-48 of a product.  With
// both in one word, which rounded every step, a short run's gradient was up to
// 24 times as far from the exact sum of the same products as FP64 sums are.
// Ten E_z and six in-plane grids of 300 to 900 steps, rms error over the design
// box relative to its gradient: FP64 sums 3.4e-16 to 1.2e-15, one word 8e-16 to
// 2e-15 (8 terms) and 2.4e-15 to 9.6e-15 (32), these 2.2e-16 to 5.5e-16 (8) and,
// in PairSum, 1.2e-16 to 3e-16 (32).
//
// One factor is scaled by a power of two (PairScale; at least 1, so the scaling
// loses nothing), which keeps the tails of a wave front (1e-30 and below, at
// amplitude 1) within FP32's range; value() undoes it.  The products go with
// the square of the source's amplitude, and so does the scale (pair_scale),
// so that a strong source's products stay clear of FAR like a weak one's.
struct Pair {
    float hi, lo, c;
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
    // a += b; the rounding error.
    static __device__ __forceinline__ float two_sum(float &a, float b)
    {
        const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
        const float r = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
        a = s;
        return r;
    }
    // Adds a bs but for its rounding error, which is returned.
    __device__ __forceinline__ float add_rounded(float a, float bs)
    {
        const float p = __fmul_rn(a, bs);
        lo = __fadd_rn(lo, two_sum(hi, p));
        return __fmaf_rn(a, bs, -p);
    }
    __device__ __forceinline__ void add(float a, float bs) { c = __fadd_rn(c, add_rounded(a, bs)); }
    __device__ __forceinline__ double value(double down) const { return ((double)hi + ((double)lo + (double)c)) * down; }
    // The sum to 2^-49 of itself.
    __device__ __forceinline__ double value49(double down) const
    {
        float h = hi;
        const float r = two_sum(h, lo);
        return ((double)h + (double)__fadd_rn(r, c)) * down;
    }
};

// The sum of more terms: groups of 8 and the products' errors in fours, joined
// exactly (d, the errors' errors, rounds far below FP64's last place).  As one
// group of 32 a node that a wave front reaches within it was up to 2e-14 of its
// terms off (FP64: 2e-15), in groups 1.3e-15.  491^2 in plane 23.7 -> 24.0 ms per
// evaluation for it.
struct PairSum {
    float hi, lo, c, d;
    __device__ __forceinline__ void errors(Pair &g)
    {
        d = __fadd_rn(d, Pair::two_sum(c, g.c));
        g.c = 0.0f;
    }
    __device__ __forceinline__ void merge(Pair &g)
    {
        const float r = Pair::two_sum(hi, g.hi), r1 = Pair::two_sum(lo, r), r2 = Pair::two_sum(lo, g.lo);
        d = __fadd_rn(d, __fadd_rn(r1, r2));
        g = Pair{};
    }
    __device__ __forceinline__ double value(double down) const
    {
        float h = hi, r = Pair::two_sum(h, lo);
        const float r2 = __fadd_rn(Pair::two_sum(r, c), d);
        return ((double)h + ((double)r + (double)r2)) * down;
    }
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
                best = Rt2DPlan{H, tw, th, nw, bx, by, 1, sms};
            }
        }
    }
    return best;
}

}  // namespace
}  // namespace fdtd
