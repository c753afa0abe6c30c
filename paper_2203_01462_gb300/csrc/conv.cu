// 3 x 3 convolutions of the surrogate network with BF16 products on the
// tensor cores (mma.sync m16n8k16, FP32 accumulation), without the im2col
// matrices: the column operand's tiles are gathered from the activations
// straight into shared memory.
//
// As im2col + GEMM + col2im + bias passes a training step of the base-24
// network on 8 x 256^2 maps moved about 25 GB: each im2col matrix is nine
// times its activations and goes through HBM twice.  Without them the step
// went from 15.8 to 4.2 ms and a prediction of one map from 0.94 to 0.35 ms.  What
// bounds these kernels now is instruction issue and shared memory: rounding
// and staging the operands (the 72 -> 24 convolution at 256^2: 140 us
// forward, 168 us input gradient, 293 us weight gradient, with 30 to 60 us of
// HBM traffic each).
//
// The products are those of nn_gemm_bf16 on the im2col matrix, in the same
// order (16 products per mma, k ascending, the same K slices where the GEMM
// splits K; in the input gradient one sum per tap, the nine added in tap
// order as col2im adds them), so the results are the same bits.
//
//   forward        y[co][p]  = act(sum_{k = (c, t)} w[co][k] x[c][p + off_t] + bias[co])
//   input gradient dx[c][p] += sum_t (sum_co w[co][(c, t)] dy[co][p - off_t])
//   weight grad.   gw[co][(c, t)] = sum_p dy[co][p] x[c][p + off_t]
//
// with off_t the t-th of the nine taps, zero outside the image.  Activations
// are [C][B][H][W]; p runs over B H W.
//
// Tiles: a warp owns 16 MF rows x 32 columns of the product; WM x WN warps
// per block; K in slices of 32, double-buffered in shared memory (rows padded
// to 80 bytes: ldmatrix and the 16-byte stores hit distinct banks), the next
// slice's global loads in flight in registers while the current one is
// multiplied, one barrier per slice.
//
// Every kernel here and in nn.cu is launched before its predecessor has ended
// and waits for it before it touches memory (programmatic dependent launch):
// a step is about 115 launches, many of a few microseconds.  128^2 x 2 training
// step 0.98 -> 0.80 ms, 256^2 prediction 0.34 -> 0.25.  The short kernels and
// the weight gradient, which leaves room on the SMs, also let their
// successor's blocks in while they run; for the forward and input-gradient
// kernels that cost the 8 x 256^2 step 1 % (3.55 -> 3.60 ms), and for the GEMMs
// and the passes around them (nn.cu) up to a third of the FP32 network: 8 x
// 256^2 training step 31.6 ms with, 28.5 without, 2 x 96^2 at base 64 6.10 and
// 4.65, 512^2 at base 8 6.37 and 4.68 (29.4, 5.20 and 5.31 as plain launches).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/surrogate.h"
#include "launch.cuh"

namespace {

constexpr int BK = 32, BKP = 40;  // slice depth, padded row length (BF16 words)

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldmatrix4(unsigned (&r)[4], const __nv_bfloat16 *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}

__device__ __forceinline__ void ldmatrix4_trans(unsigned (&r)[4], const __nv_bfloat16 *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}

// (a0, a1) += (b0, b1): one instruction, each sum rounded as by +.
__device__ __forceinline__ void add2(float &a0, float &a1, float b0, float b1)
{
    asm("{\n\t"
        ".reg .b64 a, b;\n\t"
        "mov.b64 a, {%0, %1};\n\t"
        "mov.b64 b, {%2, %3};\n\t"
        "add.rn.f32x2 a, a, b;\n\t"
        "mov.b64 {%0, %1}, a;\n\t"
        "}"
        : "+f"(a0), "+f"(a1)
        : "f"(b0), "f"(b1));
}

__device__ __forceinline__ unsigned pack(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const unsigned *>(&v);
}

// One warp's share of a slice: 16 MF rows from row m0 of As, 32 columns from
// row n0 of Bs.
template <int MF>
__device__ __forceinline__ void mma_slice(float (&acc)[MF][4][4], const __nv_bfloat16 *As, const __nv_bfloat16 *Bs, int m0,
                                          int n0, int lane)
{
    const int ar = (lane >> 3 & 1) * 8 + (lane & 7), ak = (lane >> 4) * 8;
    const int br = (lane >> 4) * 8 + (lane & 7), bk = (lane >> 3 & 1) * 8;
#pragma unroll
    for (int ks = 0; ks < BK; ks += 16) {
        unsigned b[2][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) ldmatrix4(b[j], Bs + (n0 + j * 16 + br) * BKP + ks + bk);
#pragma unroll
        for (int i = 0; i < MF; ++i) {
            unsigned a[4];
            ldmatrix4(a, As + (m0 + i * 16 + ar) * BKP + ks + ak);
#pragma unroll
            for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a, b[j >> 1][(j & 1) * 2], b[j >> 1][(j & 1) * 2 + 1]);
        }
    }
}

// Nine bits: tap t of the pixel (y, x) lies in the H x W image (sign = 1:
// the tap at + off_t, -1: at - off_t).
__device__ __forceinline__ unsigned tap_mask(int y, int x, int H, int W, int sign)
{
    unsigned m = 0;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        const int yy = y + sign * (t / 3 - 1), xx = x + sign * (t % 3 - 1);
        if (yy >= 0 && yy < H && xx >= 0 && xx < W) m |= 1u << t;
    }
    return m;
}

// Forward (DG = false): rows = output channels, k = (c, t); input gradient
// (DG = true): rows = input channels, one pass over the output channels per
// tap (relu: whether dx is added to).  Columns = pixels; a thread gathers 32 / WM of a slice's values of one
// pixel.  K slices of the forward go to blockIdx.z; with more than one, the
// partial products go to part.
template <int MF, int WM, int WN, bool DG>
__global__ void __launch_bounds__(32 * WM * WN) k_conv3(const float *__restrict__ in, const float *__restrict__ w,
                                                        const float *__restrict__ bias, float *out, int ci, int co,
                                                        long long P, int H, int W, int relu, int kc, float *part)
{
    fdtd::pdl_wait();
    constexpr int BM = 16 * MF * WM, BN = 32 * WN, NT = 32 * WM * WN, KP = BK / WM, AP = BM * 16 / NT;
    static_assert(BM * 16 % NT == 0, "whole pairs per thread");
    __shared__ __align__(16) __nv_bfloat16 As[2][BM * BKP];
    __shared__ __align__(16) __nv_bfloat16 Bs[2][BN * BKP];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp / WN, wn = warp % WN;
    const int m0 = blockIdx.y * BM, M = DG ? ci : co, K9 = ci * 9;
    const long long n0 = blockIdx.x * (long long)BN;
    // this thread's pixel and part of k
    const int px = tid % BN, kp0 = tid / BN * KP;
    const long long p = n0 + px;
    unsigned mask = 0;
    if (p < P) {
        const int r = (int)(p % ((long long)H * W));
        mask = tap_mask(r / W, r % W, H, W, DG ? -1 : 1);
    }
    const float *ip = in + (p < P ? p : 0);
    const int kb = DG ? 0 : blockIdx.z * kc, ke = DG ? co : min(K9, kb + kc);
    const int S = (ke - kb + BK - 1) / BK, steps = DG ? 9 * S : S;

    float rb[KP], ra[2 * AP];
    auto load = [&](int s) {
        const int t0 = DG ? s / S : 0, k0 = kb + (DG ? s % S : s) * BK;
#pragma unroll
        for (int q = 0; q < KP; ++q) {
            const int k = k0 + kp0 + q;
            const int c = DG ? k : k / 9, t = DG ? t0 : k - 9 * (k / 9);
            const int off = (DG ? -1 : 1) * ((t / 3 - 1) * W + t % 3 - 1);
            rb[q] = 0.0f;
            if (k < ke && (mask >> t & 1u)) rb[q] = ip[c * P + off];
        }
#pragma unroll
        for (int q = 0; q < AP; ++q) {
            const int e = tid + q * NT, m = m0 + e / 16, k = k0 + e % 16 * 2;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                ra[2 * q + h] = 0.0f;
                if (m < M && k + h < ke)
                    ra[2 * q + h] = DG ? w[(long long)(k + h) * K9 + m * 9 + t0] : w[(long long)m * K9 + k + h];
            }
        }
    };
    float acc[MF][4][4], tot[MF][4][4];
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = tot[i][j][r] = 0.0f;
    load(0);
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
        __nv_bfloat16 *A = As[s & 1], *B = Bs[s & 1];
#pragma unroll
        for (int q = 0; q < KP; q += 8)
            *reinterpret_cast<uint4 *>(B + px * BKP + kp0 + q) =
                make_uint4(pack(rb[q], rb[q + 1]), pack(rb[q + 2], rb[q + 3]), pack(rb[q + 4], rb[q + 5]),
                           pack(rb[q + 6], rb[q + 7]));
#pragma unroll
        for (int q = 0; q < AP; ++q) {
            const int e = tid + q * NT;
            *reinterpret_cast<unsigned *>(A + e / 16 * BKP + e % 16 * 2) = pack(ra[2 * q], ra[2 * q + 1]);
        }
        __syncthreads();
        if (s + 1 < steps) load(s + 1);
        mma_slice<MF>(acc, A, B, wm * 16 * MF, wn * 32, lane);
        if (DG && (s + 1) % S == 0) {
            // the tap's sum joins the others, in tap order
#pragma unroll
            for (int i = 0; i < MF; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        tot[i][j][r] += acc[i][j][r];
                        acc[i][j][r] = 0.0f;
                    }
        }
    }
    // accumulator r of fragment (i, j): row g (+ 8 for r >= 2), column 2t (+ 1 for odd r)
    const int g = lane >> 2, t2 = (lane & 3) * 2;
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const int m = m0 + wm * 16 * MF + i * 16 + g + hr * 8;
            if (m >= M) continue;
            const float b = (!DG && gridDim.z == 1) ? bias[m] : 0.0f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const long long n = n0 + wn * 32 + j * 8 + t2;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (n + h >= P) continue;
                    if (DG) {
                        float *o = out + m * P + n + h;
                        *o = (relu ? *o : 0.0f) + tot[i][j][hr * 2 + h];
                    } else if (gridDim.z > 1) {
                        part[((long long)blockIdx.z * M + m) * P + n + h] = acc[i][j][hr * 2 + h];
                    } else {
                        const float v = acc[i][j][hr * 2 + h] + b;
                        out[m * P + n + h] = relu && v < 0.0f ? 0.0f : v;
                    }
                }
            }
        }
}

// V values from e on of part[0] + part[1] + ... + part[S - 1] (slices n
// apart), in that order, the loads of eight slices in flight.
template <int V>
__device__ __forceinline__ void slices(const float *__restrict__ part, long long n, long long e, int S, float (&a)[V])
{
    auto load = [&](long long z, float (&o)[V]) {
        if constexpr (V == 4) {
            const float4 t = *reinterpret_cast<const float4 *>(part + z * n + e);
            o[0] = t.x;
            o[1] = t.y;
            o[2] = t.z;
            o[3] = t.w;
        } else {
            o[0] = part[z * n + e];
        }
    };
    constexpr int D = V == 4 ? 8 : 16;
    load(0, a);
    for (int z = 1; z < S; z += D) {
        float v[D][V];
#pragma unroll
        for (int q = 0; q < D; ++q)
            if (z + q < S) load(z + q, v[q]);
#pragma unroll
        for (int q = 0; q < D; ++q)
            if (z + q < S)
#pragma unroll
                for (int i = 0; i < V; ++i) a[i] += v[q][i];
    }
}

// y = act(sum of the S slices of part, in order, + bias); V divides P.
template <int V>
__global__ void __launch_bounds__(128) k_slices_bias_act(float *y, const float *__restrict__ part,
                                                         const float *__restrict__ bias, int M, long long P, int S,
                                                         int relu)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    const long long n = (long long)M * P;
    for (long long e = (blockIdx.x * (long long)blockDim.x + threadIdx.x) * V; e < n;
         e += (long long)gridDim.x * blockDim.x * V) {
        float a[V];
        slices<V>(part, n, e, S, a);
        const float b = bias[e / P];
#pragma unroll
        for (int i = 0; i < V; ++i) {
            a[i] += b;
            if (relu && a[i] < 0.0f) a[i] = 0.0f;
        }
        if constexpr (V == 4) *reinterpret_cast<float4 *>(y + e) = make_float4(a[0], a[1], a[2], a[3]);
        else y[e] = a[0];
    }
}

// C = the sum of the S slices of part, in order.
__global__ void __launch_bounds__(64) k_slices(float *C, const float *__restrict__ part, long long n, int S)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        float a[1];
        slices<1>(part, n, e, S, a);
        C[e] = a[0];
    }
}

// Weight gradient: rows = output channels, columns = (c, t), k = pixels.  A
// half-warp gathers one row's 32 pixels as pairs; a thread's rows stay the
// same for all slices.  blockIdx.z takes the pixels [z kc, (z + 1) kc).
template <int MF, int WM, int WN>
__global__ void __launch_bounds__(32 * WM * WN) k_conv3_wgrad(const float *__restrict__ dy, const float *__restrict__ x,
                                                              float *gw, int ci, int co, long long P, int H, int W,
                                                              long long kc, float *part)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    constexpr int BM = 16 * MF * WM, BN = 32 * WN, NT = 32 * WM * WN, HW = NT / 16, NB = (BN + HW - 1) / HW,
                  NA = (BM + HW - 1) / HW;
    __shared__ __align__(16) __nv_bfloat16 As[2][BM * BKP];
    __shared__ __align__(16) __nv_bfloat16 Bs[2][BN * BKP];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp / WN, wn = warp % WN;
    const int N = ci * 9, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const long long kb = blockIdx.z * kc, ke = min(P, kb + kc);
    const int hw = tid >> 4, l2 = (tid & 15) * 2;  // half-warp, first pixel of the pair within the slice
    // this thread's columns: offset of their tap and channel, tap (9: none)
    long long off[NB];
    unsigned tap[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
        const int n = n0 + hw + q * HW, c = n / 9, t = n % 9;
        const bool ok = hw + q * HW < BN && n < N;
        off[q] = ok ? (long long)c * P + (t / 3 - 1) * W + t % 3 - 1 : 0;
        tap[q] = ok ? t : 9;
    }
    const bool aligned = W % BK == 0;  // (kb is a multiple of 32: a slice lies in one image row)
    float rb[2 * NB], ra[2 * NA];
    auto load = [&](long long k0) {
        const long long p = k0 + l2;
        unsigned mk[2] = {0, 0};
        if (aligned) {
            const int r = (int)(k0 % ((long long)H * W)), y = r / W, xx = r % W + l2;
            mk[0] = p < ke ? tap_mask(y, xx, H, W, 1) : 0;
            mk[1] = p + 1 < ke ? tap_mask(y, xx + 1, H, W, 1) : 0;
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (p + h < ke) {
                    const int r = (int)((p + h) % ((long long)H * W));
                    mk[h] = tap_mask(r / W, r % W, H, W, 1);
                }
        }
        const float *xp = x + p;
#pragma unroll
        for (int q = 0; q < NB; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                rb[2 * q + h] = 0.0f;
                if (mk[h] >> tap[q] & 1u) rb[2 * q + h] = xp[off[q] + h];
            }
#pragma unroll
        for (int q = 0; q < NA; ++q) {
            const int m = m0 + hw + q * HW;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                ra[2 * q + h] = 0.0f;
                if (hw + q * HW < BM && m < co && p + h < ke) ra[2 * q + h] = dy[m * P + p + h];
            }
        }
    };
    float acc[MF][4][4];
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.0f;
    if (kb < ke) load(kb);
    int s = 0;
#pragma unroll 1
    for (long long k0 = kb; k0 < ke; k0 += BK, s ^= 1) {
        __nv_bfloat16 *A = As[s], *B = Bs[s];
#pragma unroll
        for (int q = 0; q < NB; ++q)
            if (BN % HW == 0 || hw + q * HW < BN)
                *reinterpret_cast<unsigned *>(B + (hw + q * HW) * BKP + l2) = pack(rb[2 * q], rb[2 * q + 1]);
#pragma unroll
        for (int q = 0; q < NA; ++q)
            if (BM % HW == 0 || hw + q * HW < BM)
                *reinterpret_cast<unsigned *>(A + (hw + q * HW) * BKP + l2) = pack(ra[2 * q], ra[2 * q + 1]);
        __syncthreads();
        if (k0 + BK < ke) load(k0 + BK);
        mma_slice<MF>(acc, A, B, wm * 16 * MF, wn * 32, lane);
    }
    const int g = lane >> 2, t2 = (lane & 3) * 2;
    float *out = gridDim.z > 1 ? part + (long long)blockIdx.z * co * N : gw;
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int m = m0 + wm * 16 * MF + i * 16 + g + (r >> 1) * 8, n = n0 + wn * 32 + j * 8 + t2 + (r & 1);
                if (m < co && n < N) out[(long long)m * N + n] = acc[i][j][r];
            }
}

// ------------------------------------------------ image rows of whole 16-byte groups
//
// With W a multiple of four the tiles need no gather per tap: a block takes
// image rows x 32 pixels (a warp per row) with a one-pixel border, rounds them
// to BF16 once and keeps them in shared memory, zeros outside the image; the
// nine taps are address offsets.  Each activation is then loaded 1.3 times
// instead of nine, in 16-byte words, and a 16 x 32 operand fragment takes two
// ldmatrix.  Against the gather kernels above: 7.6 -> 4.2 ms for the training
// step (256^2), 2.8 -> 1.7 ms with rows of 200, 100, 50 and 25 pixels.

constexpr int TH = 8;   // image rows of a block
constexpr int XS = 40;  // padded row: pixel x0 + i at index 4 + i, so the whole row goes in as 16-byte loads

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// A row of 32 pixels in three copies, shifted by a pixel (copy d: pixel
// x0 - 1 + d + i at index i), so that eight consecutive pixels are an aligned
// 16-byte row of ldmatrix at every tap: [channel][image row][copy][RS].  With
// rows of 80 bytes the eight rows of a matrix (consecutive (c, t)) lie in
// eight different 16-byte groups of the banks, if channels are 20 words apart
// (mod 32).
constexpr int RS = 40;

// Four pixels into the copies: v with its neighbours l and r.
__device__ __forceinline__ void store_quad(__nv_bfloat16 *o, float4 v, float l, float r)
{
    const unsigned mid = pack(v.y, v.z);
    *reinterpret_cast<uint2 *>(o) = make_uint2(pack(l, v.x), mid);
    *reinterpret_cast<uint2 *>(o + RS) = make_uint2(pack(v.x, v.y), pack(v.z, v.w));
    *reinterpret_cast<uint2 *>(o + 2 * RS) = make_uint2(mid, pack(v.w, r));
}

// Forward: channels in chunks of 16 (144 products, nine k-steps).
template <int MF, int WM>
__global__ void __launch_bounds__(256, 2)
k_conv3_fwd_t(const float *__restrict__ x, const float *__restrict__ w, const float *__restrict__ bias, float *y, int ci,
              int co, int B, int H, int W, int relu, int kc, float *part)
{
    fdtd::pdl_wait();
    constexpr int ROWS = TH / WM, BM = 16 * MF * WM, CH = 16, KC = 144, AS = KC + 8,
                  XC = ((ROWS + 2) * 3 * RS / 2 + 11) / 32 * 64 + 40,  // channel stride: 20 words mod 32
        XN = (ROWS + 2) / 2, AU = BM * KC / 4, AN = (AU + 255) / 256, AB = MF == 3 ? 2 : 5;
    static_assert(XC >= (ROWS + 2) * 3 * RS, "rows fit");
    extern __shared__ __align__(16) __nv_bfloat16 fsm[];
    __nv_bfloat16 *const Xs = fsm, *const As = fsm + 2 * CH * XC;  // [2][CH * XC], [2][BM * AS]
    __shared__ int Ks[KC];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp / ROWS, wr = warp % ROWS;
    const int K9 = ci * 9, m0 = blockIdx.y * BM;
    const int gw = (W + 31) / 32, gh = (H + ROWS - 1) / ROWS;
    const int x0 = blockIdx.x % gw * 32, y0 = blockIdx.x / gw % gh * ROWS, b = blockIdx.x / (gw * gh);
    const long long HW = (long long)H * W, P = HW * B;
    const int kb = blockIdx.z * kc, ke = min(K9, kb + kc);
    // offsets of the matrix rows (c, t); a lane reads row k = 16 st + (lane & 15), pixels 8 (lane >> 4) .. (+ 16)
    if (tid < KC) Ks[tid] = tid / 9 * XC + (tid % 9 / 3 * 3 + tid % 3) * RS;
    // this thread's share of a chunk: channel xc, rows xr + 2 u, pixels 4 xq .. + 3 (the first and the
    // last thread of a row also the pixel beside it); of the weights four consecutive k per unit
    const int xq = tid & 7, h16 = tid >> 3 & 15, xc = (h16 & 1) << 2 | (h16 >> 1 & 3) | (h16 & 8), xr = tid >> 7;
    const float *xp = x + xc * P + b * HW + x0 + 4 * xq;
    const bool xin = x0 + 4 * xq < W, hin = xq == 0 ? x0 > 0 : xq == 7 && x0 + 32 < W;
    const int hoff = xq == 0 ? -1 : 4;
    const bool w16 = K9 % 4 == 0 && ((uintptr_t)w & 15) == 0;
    float4 rx[XN];
    float rh[XN];
    auto load_x = [&](int q0) {  // chunk q0: channels 16 q0 ..
        const float *p = xp + q0 * CH * P;
        const bool in = xin && q0 * CH + xc < ci;
#pragma unroll
        for (int u = 0; u < XN; ++u) {
            const int yy = y0 + xr + 2 * u - 1;
            rx[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            rh[u] = 0.0f;
            if (in && yy >= 0 && yy < H) {
                rx[u] = ld4(p + (long long)yy * W);
                if (hin) rh[u] = p[(long long)yy * W + hoff];
            }
        }
    };
    auto store_x = [&](int s) {
        __nv_bfloat16 *X = Xs + s * CH * XC + xc * XC + xr * 3 * RS + 4 * xq;
#pragma unroll
        for (int u = 0; u < XN; ++u) {
            float l = __shfl_up_sync(0xffffffffu, rx[u].w, 1), r = __shfl_down_sync(0xffffffffu, rx[u].x, 1);
            if (xq == 0) l = rh[u];
            if (xq == 7) r = rh[u];
            store_quad(X + u * 6 * RS, rx[u], l, r);
        }
    };
    auto weights = [&](int q0, int s) {
        __nv_bfloat16 *A = As + s * BM * AS;
#pragma unroll
        for (int v = 0; v < AN; v += AB) {
            float4 ra[AB];
#pragma unroll
            for (int u = 0; u < AB; ++u) {
                const int e = tid + (v + u) * 256, m = m0 + e / (KC / 4), k = q0 * KC + e % (KC / 4) * 4;
                ra[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (v + u >= AN || e >= AU || m >= co) continue;
                const float *p = w + (long long)m * K9 + k;
                if (w16) {  // (kb and ke are multiples of four: all of the unit or nothing)
                    if (k >= kb && k < ke) ra[u] = ld4(p);
                } else {
                    if (k >= kb && k < ke) ra[u].x = p[0];
                    if (k + 1 >= kb && k + 1 < ke) ra[u].y = p[1];
                    if (k + 2 >= kb && k + 2 < ke) ra[u].z = p[2];
                    if (k + 3 >= kb && k + 3 < ke) ra[u].w = p[3];
                }
            }
#pragma unroll
            for (int u = 0; u < AB; ++u) {
                const int e = tid + (v + u) * 256;
                if (v + u < AN && e < AU)
                    *reinterpret_cast<uint2 *>(A + e / (KC / 4) * AS + e % (KC / 4) * 4) =
                        make_uint2(pack(ra[u].x, ra[u].y), pack(ra[u].z, ra[u].w));
            }
        }
    };
    float acc[MF][4][4];
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.0f;
    const int ar = (lane >> 3 & 1) * 8 + (lane & 7), ak = (lane >> 4) * 8;
    const int qb = kb / KC, qe = (ke + KC - 1) / KC;
    load_x(qb);
    weights(qb, qb & 1);
    store_x(qb & 1);
#pragma unroll 1
    for (int q0 = qb; q0 < qe; ++q0) {
        __syncthreads();
        if (q0 + 1 < qe) {
            load_x(q0 + 1);
            weights(q0 + 1, q0 + 1 & 1);
        }
        const __nv_bfloat16 *X = Xs + (q0 & 1) * CH * XC + wr * 3 * RS + (lane >> 4) * 8;
        const __nv_bfloat16 *A = As + (q0 & 1) * BM * AS + (wm * 16 * MF + ar) * AS + ak;
        const int sb = max(0, (kb - q0 * KC) / 16), se = min(9, (ke - q0 * KC + 15) / 16);
#pragma unroll 3
        for (int st = sb; st < se; ++st) {
            const int o = Ks[st * 16 + (lane & 15)];
            unsigned bf[2][4];
            ldmatrix4_trans(bf[0], X + o);
            ldmatrix4_trans(bf[1], X + o + 16);
#pragma unroll
            for (int i = 0; i < MF; ++i) {
                unsigned a[4];
                ldmatrix4(a, A + i * 16 * AS + st * 16);
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a, bf[j >> 1][(j & 1) * 2], bf[j >> 1][(j & 1) * 2 + 1]);
            }
        }
        if (q0 + 1 < qe) store_x(q0 + 1 & 1);
    }
    const int yy = y0 + wr;
    if (yy >= H) return;
    const int g = lane >> 2, t2 = (lane & 3) * 2;
    const long long n0 = b * HW + (long long)yy * W + x0 + t2;
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int hr2 = 0; hr2 < 2; ++hr2) {
            const int m = m0 + wm * 16 * MF + i * 16 + g + hr2 * 8;
            if (m >= co) continue;
            const float bb = gridDim.z == 1 ? bias[m] : 0.0f;
            float *o = gridDim.z == 1 ? y + m * P + n0 : part + ((long long)blockIdx.z * co + m) * P + n0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (x0 + t2 + j * 8 >= W) continue;
                float v0 = acc[i][j][hr2 * 2], v1 = acc[i][j][hr2 * 2 + 1];
                if (gridDim.z == 1) {
                    v0 += bb;
                    v1 += bb;
                    if (relu && v0 < 0.0f) v0 = 0.0f;
                    if (relu && v1 < 0.0f) v1 = 0.0f;
                }
                *reinterpret_cast<float2 *>(o + j * 8) = make_float2(v0, v1);
            }
        }
}

// Input gradient: the whole depth (output channels, as pairs: one 32-bit
// load per fragment word) of a tile stays in shared memory for all nine taps,
// the weights of G taps (nine, three or one) with it.  Kp: co rounded up to 16.
constexpr int XCD = (TH + 2) * XS + 8;  // words of a channel pair (8 mod 32 apart: the fragments' four pairs in distinct banks)

template <int MF, int G>
__global__ void __launch_bounds__(256, 2)
k_conv3_dgrad_t(const float *__restrict__ dy, const float *__restrict__ w, float *dx, int ci, int co, int Kp, int B, int H,
                int W, int add)
{
    fdtd::pdl_wait();
    constexpr int BM = 16 * MF;
    extern __shared__ __align__(16) unsigned dsm[];
    unsigned *X = dsm;  // [Kp / 2][XCD]
    const int AS = Kp + 8, AT = BM * AS + 8;
    __nv_bfloat16 *As = reinterpret_cast<__nv_bfloat16 *>(dsm + (size_t)Kp / 2 * XCD);  // [G][BM][AS], a tap AT apart
    const int tid = threadIdx.x, lane = tid & 31, wr = tid >> 5;
    const int K9 = ci * 9, m0 = blockIdx.y * BM;
    const int gw = (W + 31) / 32, gh = (H + TH - 1) / TH;
    const int x0 = blockIdx.x % gw * 32, y0 = blockIdx.x / gw % gh * TH, b = blockIdx.x / (gw * gh);
    const long long HW = (long long)H * W, P = HW * B;
    // taps t0 .. t0 + G - 1 of rows m0 .. : pairs of output channels, consecutive threads on consecutive words of w
    auto weights = [&](int t0) {
        constexpr int ROW = BM * G, EN = (ROW + 255) / 256, KB = 8 / EN < 1 ? 1 : 8 / EN;  // KB pairs in flight
        const float *p[EN];
        int o[EN];
        bool ok[EN];
#pragma unroll
        for (int u = 0; u < EN; ++u) {
            const int e = tid + u * 256, m = e / G, t = e % G;
            ok[u] = e < ROW && m0 + m < ci;
            p[u] = w + (m0 + m) * 9 + t0 + t;
            o[u] = e < ROW ? t * AT + m * AS : -1;
        }
#pragma unroll 1
        for (int k0 = 0; k0 < Kp; k0 += 2 * KB) {  // (Kp is a multiple of 16)
            float v[KB][EN][2];
#pragma unroll
            for (int q = 0; q < KB; ++q)
#pragma unroll
                for (int u = 0; u < EN; ++u)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        v[q][u][h] = 0.0f;
                        if (ok[u] && k0 + 2 * q + h < co) v[q][u][h] = p[u][(2 * q + h) * (long long)K9];
                    }
#pragma unroll
            for (int u = 0; u < EN; ++u) {
                p[u] += 2 * KB * (long long)K9;
#pragma unroll
                for (int q = 0; q < KB; ++q)
                    if (o[u] >= 0) *reinterpret_cast<unsigned *>(As + o[u] + k0 + 2 * q) = pack(v[q][u][0], v[q][u][1]);
            }
        }
    };
    const float *base = dy + b * HW + x0;
    const int units = Kp / 2 * (TH + 2) * 8;
    for (int e0 = tid; e0 < units; e0 += 5 * 256) {
        float4 v[5][2];
#pragma unroll
        for (int u = 0; u < 5; ++u) {
            const int e = e0 + u * 256, cp = e / ((TH + 2) * 8), yy = y0 + e / 8 % (TH + 2) - 1;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                v[u][h] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (2 * cp + h < co && yy >= 0 && yy < H && x0 + (e & 7) * 4 < W)
                    v[u][h] = ld4(base + (2 * cp + h) * P + (long long)yy * W + (e & 7) * 4);
            }
        }
#pragma unroll
        for (int u = 0; u < 5; ++u) {
            const int e = e0 + u * 256, cp = e / ((TH + 2) * 8), r = e / 8 % (TH + 2);
            if (e < units)
                *reinterpret_cast<uint4 *>(X + cp * XCD + r * XS + 4 + (e & 7) * 4) =
                    make_uint4(pack(v[u][0].x, v[u][1].x), pack(v[u][0].y, v[u][1].y), pack(v[u][0].z, v[u][1].z),
                               pack(v[u][0].w, v[u][1].w));
        }
    }
    for (int e = tid; e < Kp / 2 * (TH + 2) * 2; e += 256) {
        const int cp = e / ((TH + 2) * 2), r = e / 2 % (TH + 2), yy = y0 + r - 1;
        const bool ok = yy >= 0 && yy < H && (e & 1 ? x0 + 32 < W : x0 > 0);
        float v[2] = {0.0f, 0.0f};
        for (int h = 0; h < 2; ++h)
            if (ok && 2 * cp + h < co) v[h] = base[(2 * cp + h) * P + (long long)yy * W + (e & 1 ? 32 : -1)];
        X[cp * XCD + r * XS + (e & 1 ? 36 : 3)] = pack(v[0], v[1]);
    }
    float tot[MF][4][4];
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) tot[i][j][r] = 0.0f;
    const int ar = (lane >> 3 & 1) * 8 + (lane & 7), ak = (lane >> 4) * 8;
#pragma unroll 1
    for (int t = 0; t < 9; ++t) {
        if (t % G == 0) {
            if (t) __syncthreads();
            weights(t);
            __syncthreads();
        }
        const __nv_bfloat16 *A = As + t % G * AT;
        // the tap reads pixel p - off_t
        const unsigned *Xb = X + (lane & 3) * XCD + (wr + 2 - t / 3) * XS + (lane >> 2) + 5 - t % 3;
        float acc[MF][4][4];
#pragma unroll
        for (int i = 0; i < MF; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.0f;
#pragma unroll 2
        for (int ks = 0; ks < Kp; ks += 16) {
            unsigned bf[4][2];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                bf[j][0] = Xb[ks / 2 * XCD + 8 * j];
                bf[j][1] = Xb[(ks / 2 + 4) * XCD + 8 * j];
            }
#pragma unroll
            for (int i = 0; i < MF; ++i) {
                unsigned a[4];
                ldmatrix4(a, A + (i * 16 + ar) * AS + ks + ak);
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a, bf[j][0], bf[j][1]);
            }
        }
#pragma unroll
        for (int i = 0; i < MF; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int r = 0; r < 4; r += 2) add2(tot[i][j][r], tot[i][j][r + 1], acc[i][j][r], acc[i][j][r + 1]);
    }
    const int yy = y0 + wr;
    if (yy >= H) return;
    const int g = lane >> 2, t2 = (lane & 3) * 2;
    const long long n0 = b * HW + (long long)yy * W + x0 + t2;
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {
            const int m = m0 + i * 16 + g + hr * 8;
            if (m >= ci) continue;
            float2 v[4];
            float2 *o = reinterpret_cast<float2 *>(dx + m * P + n0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                v[j] = make_float2(0.0f, 0.0f);
                if (add && x0 + t2 + j * 8 < W) v[j] = o[j * 4];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (x0 + t2 + j * 8 < W)
                    o[j * 4] = make_float2(v[j].x + tot[i][j][hr * 2], v[j].y + tot[i][j][hr * 2 + 1]);
        }
}

// Weight gradient: segments of 32 pixels in order (eight groups of four, each
// in one image row).  The columns' channels (at most 16 for a tile's 128
// columns) are staged with the rows above and below, in three copies shifted
// by a pixel, so that a pair of pixels is an aligned 32-bit word at every tap.
template <int MF, int WM>
__global__ void __launch_bounds__(128 * WM) k_conv3_wgrad_t(const float *__restrict__ dy, const float *__restrict__ x,
                                                            float *gw, int ci, int co, int B, int H, int W, long long kc,
                                                            float *part)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    constexpr int WN = 4, BM = 16 * MF * WM, BN = 128, NT = 128 * WM, CH = 16, XC = 9 * RS,
                  XN = (3 + WM - 1) / WM, AN = BM * 8 / NT;
    static_assert(BM * 8 % NT == 0, "whole units per thread");
    __shared__ __align__(16) __nv_bfloat16 As[2][BM * BKP];
    __shared__ __align__(16) __nv_bfloat16 Xs[2][CH * XC];  // [buffer][channel][row][copy]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp / WN, wn = warp % WN;
    const int N = ci * 9, m0 = blockIdx.y * BM, n0 = blockIdx.x * BN, c0 = n0 / 9;
    const long long P = (long long)H * W * B, kb = blockIdx.z * kc, ke = min(P, kb + kc);
    // this lane's matrix rows: columns 8 (lane >> 4) + (lane & 7) (+ 16), pixels 8 (lane >> 3 & 1) ..
    int bo[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int n = n0 + wn * 32 + j * 16 + (lane >> 4) * 8 + (lane & 7), c = n / 9 - c0, t = n % 9;
        bo[j] = c * XC + t * RS + (lane >> 3 & 1) * 8;
    }
    // this thread's share of a segment: channel xc, rows xr + WM u, pixels 4 xq .. + 3 (their
    // neighbours come from the threads beside, or at the segment's ends from memory); of dy the
    // rows am + 16 WM u
    const int xq = tid & 7, h16 = tid >> 3 & 15, xc = (h16 & 1) << 2 | (h16 >> 1 & 3) | (h16 & 8), xr = tid >> 7;
    const int am = xr * 16 + xc;
    const bool xok = c0 + xc < ci;
    const float *xp = x + (xok ? (c0 + xc) * P : 0) + 4 * xq;
    const float *ap = dy + (long long)(m0 + am) * P + 4 * xq;
    const int p0 = (int)((kb + 4 * xq) % ((long long)H * W));
    int py = p0 / W, px = p0 % W;  // image row and column of this thread's four pixels
    // the segment in flight; lf, rt: the pixels have a neighbour to the left, to the right
    struct {
        float4 rx[XN], ra[AN];
        float rh[XN];
        bool lf, rt;
    } S;
    auto load = [&](long long k0) {
        float4 *rx = S.rx, *ra = S.ra;
        float *rh = S.rh;
        const bool in = k0 + 4 * xq < ke;
        S.lf = px > 0;
        S.rt = px + 4 < W;
        const bool hl = xq == 0 && S.lf, hr = xq == 7 && S.rt;
#pragma unroll
        for (int u = 0; u < XN; ++u) {
            const int r = xr + WM * u, yy = py + r - 1;
            rx[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            rh[u] = 0.0f;
            if (xok && in && r < 3 && yy >= 0 && yy < H) {
                const float *p = xp + k0 + (r - 1) * W;
                rx[u] = ld4(p);
                if (hl || hr) rh[u] = p[hl ? -1 : 4];
            }
        }
#pragma unroll
        for (int u = 0; u < AN; ++u) {
            ra[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (in && m0 + am + u * 16 * WM < co) ra[u] = ld4(ap + u * 16 * WM * P + k0);
        }
        px += 32;
        while (px >= W) {
            px -= W;
            if (++py == H) py = 0;
        }
    };
    float acc[MF][4][4];
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.0f;
    const int ar = (lane >> 3 & 1) * 8 + (lane & 7), ak = (lane >> 4) * 8;
    load(kb);
    int s = 0;
#pragma unroll 1
    for (long long k0 = kb; k0 < ke; k0 += BK) {
        const float4 *rx = S.rx, *ra = S.ra;
        const float *rh = S.rh;
        __nv_bfloat16 *A = As[s], *X = Xs[s];
        s ^= 1;
#pragma unroll
        for (int u = 0; u < XN; ++u) {
            const int r = xr + WM * u;
            float l = __shfl_up_sync(0xffffffffu, rx[u].w, 1), h = __shfl_down_sync(0xffffffffu, rx[u].x, 1);
            if (xq == 0) l = rh[u];
            if (xq == 7) h = rh[u];
            if (!S.lf) l = 0.0f;
            if (!S.rt) h = 0.0f;
            if (r < 3) store_quad(X + xc * XC + r * 3 * RS + 4 * xq, rx[u], l, h);
        }
#pragma unroll
        for (int u = 0; u < AN; ++u)
            *reinterpret_cast<uint2 *>(A + (am + u * 16 * WM) * BKP + 4 * xq) =
                make_uint2(pack(ra[u].x, ra[u].y), pack(ra[u].z, ra[u].w));
        __syncthreads();
        if (k0 + BK < ke) load(k0 + BK);
#pragma unroll
        for (int ks = 0; ks < BK; ks += 16) {
            unsigned bf[2][4];
            ldmatrix4(bf[0], X + bo[0] + ks);
            ldmatrix4(bf[1], X + bo[1] + ks);
#pragma unroll
            for (int i = 0; i < MF; ++i) {
                unsigned a[4];
                ldmatrix4(a, A + (wm * 16 * MF + i * 16 + ar) * BKP + ks + ak);
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a, bf[j >> 1][(j & 1) * 2], bf[j >> 1][(j & 1) * 2 + 1]);
            }
        }
    }
    const int g = lane >> 2, t2 = (lane & 3) * 2;
    float *out = gridDim.z > 1 ? part + (long long)blockIdx.z * co * N : gw;
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int m = m0 + wm * 16 * MF + i * 16 + g + (r >> 1) * 8, n = n0 + wn * 32 + j * 8 + t2 + (r & 1);
                if (m < co && n < N) out[(long long)m * N + n] = acc[i][j][r];
            }
}

int status() { return cudaGetLastError() == cudaSuccess ? 0 : 3; }

inline int slice_blocks(long long n, int per)
{
    const long long b = (n + per - 1) / per;
    return (int)(b < 152 * 64 ? b : 152 * 64);
}

// Rows whose 16-byte groups are aligned, and that fill the 32-pixel tiles to
// five eighths or more: the gather kernels take about twice the time per
// pixel, and narrower rows would compute more than that in padding.
bool tiled(int W) { return W % 4 == 0 && W * 8 >= (W + 31) / 32 * 32 * 5; }

// The dimensions of the three products (9 ci, co, B H W) are ints, as
// nn_gemm_bf16's are; beyond, the choice of the K slices would divide by what
// is left of them.
bool sizes_ok(int ci, int co, int B, int H, int W)
{
    return ci > 0 && co > 0 && B > 0 && H > 0 && W > 0 && 9LL * ci <= INT_MAX &&
           (long long)B * H <= INT_MAX && (long long)B * H * W <= INT_MAX;
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15) == 0; }

// Whether a block of kernel f can have `bytes` of shared memory on the current
// device.  The kernel's limit is raised to `most`, the largest size f is ever
// launched with, whatever this call's size: the limit belongs to the kernel,
// and one that followed the calls would let a thread lower it between another
// thread's call here and its launch.
bool smem_ready(const void *f, size_t bytes, size_t most)
{
    if (bytes > most) return false;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

template <int MF, int WM>
bool fwd_tiled(const float *x, const float *w, const float *bias, float *y, int ci, int co, int B, int H, int W, int relu,
               int kc, int splits, float *part, cudaStream_t st)
{
    constexpr int ROWS = TH / WM, BM = 16 * MF * WM, XC = ((ROWS + 2) * 3 * RS / 2 + 11) / 32 * 64 + 40;
    constexpr size_t smem = (2 * 16 * XC + 2 * BM * 152) * sizeof(__nv_bfloat16);
    if (!smem_ready((const void *)k_conv3_fwd_t<MF, WM>, smem, smem)) return false;
    const dim3 grid((unsigned)((W + 31) / 32 * ((H + ROWS - 1) / ROWS) * B), (co + BM - 1) / BM, splits);
    fdtd::launch_pdl_smem(k_conv3_fwd_t<MF, WM>, grid, 256, smem, st, x, w, bias, y, ci, co, B, H, W, relu, kc, part);
    return true;
}

template <int MF, int WM, int WN, bool DG>
void launch(const float *in, const float *w, const float *bias, float *out, int ci, int co, long long P, int H, int W,
            int relu, int kc, int splits, float *part, cudaStream_t st)
{
    const int M = DG ? ci : co, BM = 16 * MF * WM, BN = 32 * WN;
    const dim3 grid((unsigned)((P + BN - 1) / BN), (M + BM - 1) / BM, splits);
    fdtd::launch_pdl_smem(k_conv3<MF, WM, WN, DG>, grid, 32 * WM * WN, 0, st, in, w, bias, out, ci, co, P, H, W, relu, kc, part);
}

// Rows: up to 32 in one 32-row tile, up to 48 in one of 48, else tiles of 96.
// Columns: wide blocks (eight warps) once they fill the chip twice, else
// blocks of 64 pixels.
template <bool DG>
void conv3(const float *in, const float *w, const float *bias, float *out, int ci, int co, long long P, int H, int W,
           int relu, int kc, int splits, float *part, cudaStream_t st)
{
    const int M = DG ? ci : co;
    const long long wide = (P + 255) / 256 * ((M + 95) / 96) * splits;
    if (wide >= 2 * 152) {
        if (M <= 32) launch<2, 1, 8, DG>(in, w, bias, out, ci, co, P, H, W, relu, kc, splits, part, st);
        else if (M <= 48) launch<3, 1, 8, DG>(in, w, bias, out, ci, co, P, H, W, relu, kc, splits, part, st);
        else launch<3, 2, 4, DG>(in, w, bias, out, ci, co, P, H, W, relu, kc, splits, part, st);
    } else {
        if (M <= 32) launch<2, 1, 2, DG>(in, w, bias, out, ci, co, P, H, W, relu, kc, splits, part, st);
        else launch<3, 1, 2, DG>(in, w, bias, out, ci, co, P, H, W, relu, kc, splits, part, st);
    }
}

// Where the im2col matrix and one GEMM are faster: wide layers on few pixels,
// whose convolutions are few blocks with a long serial sum each, and the gather
// kernels, which multiply at half the GEMM's rate.  Estimates in us, fitted to
// 180 layers (base 8 to 128, 3 x 3 to 256 x 256 pixels; us, convolution / columns):
// input gradient 768 -> 768 7 x 7 x 2 250 / 35, 192 -> 192 32 x 32 59 / 22, 96 -> 96
// 64 x 64 21 / 20, 24 -> 24 256 x 256 9.3 / 48; forward 512 -> 512 18 x 18 80 / 45,
// 96 -> 96 50 x 50 x 4 80 / 61, 288 -> 96 16 x 16 x 8 33 / 39.  The convolution is
// left only for a gain of a seventh.
bool columns(double conv, double gemm) { return gemm < 0.87 * conv; }

bool columns_fwd(int ci, int co, long long P, int W)
{
    if (tiled(W)) return false;
    const double gf = 18e-9 * ci * co * P, pass = 18e-6 * ci * P;  // the products, the matrix through memory
    return columns(std::max(15.0, 48.0 * gf), 14.0 + 20.0 * gf + pass);
}

bool columns_dgrad(int ci, int co, long long P, int W)
{
    const double gf = 18e-9 * ci * co * P;
    double conv;  // of a tap, or a few, at a time: the depth is one chain
    if (!tiled(W)) conv = std::max(0.33 * co, 28.0 * gf);
    else if (co <= 96) conv = std::max(0.22 * co, 7.0 * gf);  // (all taps' or three taps' weights, two blocks per SM)
    else conv = std::max(0.33 * co, 18.0 * gf * ((W + 31) / 32 * 32) / W);
    const double pass = 36.0 * ci * P > 48e6 ? 18e-6 * ci * P : 0.0;  // the matrix stays in L2 otherwise
    return columns(conv, 12.0 + 16.0 * gf + pass);
}

}  // namespace

extern "C" {

// The K slices of nn_gemm_bf16 (nn.cu).
int nn_splitk_bf16(int M, long long N, long long K, long long work_elems, long long *kc);

int nn_conv3_fwd(const float *x, const float *w, const float *bias, float *y, int ci, int co, int B, int H, int W,
                 int relu, float *work, long long work_elems, void *stream)
{
    if (!x || !w || !bias || !y || !sizes_ok(ci, co, B, H, W) || work_elems < 0 || (work_elems > 0 && !work)) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    const long long P = (long long)B * H * W;
    long long kc = 0;
    const int splits = nn_splitk_bf16(co, P, 9LL * ci, work_elems, &kc);
    const auto tile = co <= 32 ? fwd_tiled<2, 1> : co <= 64 ? fwd_tiled<2, 2> : fwd_tiled<3, 2>;
    if (!(tiled(W) && aligned16(x) && aligned16(y) && aligned16(work) &&
          tile(x, w, bias, y, ci, co, B, H, W, relu, (int)kc, splits, work, st)))
        conv3<false>(x, w, bias, y, ci, co, P, H, W, relu, (int)kc, splits, work, st);
    if (splits > 1) {
        if (P % 4 == 0 && aligned16(y) && aligned16(work))
            fdtd::launch_pdl_smem(k_slices_bias_act<4>, slice_blocks(co * P, 512), 128, 0, st, y, work, bias, co, P, splits, relu);
        else
            fdtd::launch_pdl_smem(k_slices_bias_act<1>, slice_blocks(co * P, 128), 128, 0, st, y, work, bias, co, P, splits, relu);
    }
    return status();
}

int nn_conv3_dgrad(const float *dy, const float *w, float *dx, int ci, int co, int B, int H, int W, int add, void *stream)
{
    if (!dy || !w || !dx || !sizes_ok(ci, co, B, H, W)) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    const int Kp = (co + 15) / 16 * 16, BM = ci <= 32 ? 32 : 48;
    // the weights of as many taps at a time as leave room for two blocks per SM; one tap's if none do
    constexpr size_t two = 113 * 1024, one = 227 * 1024;
    const auto smem = [&](int g) { return (size_t)Kp / 2 * XCD * 4 + (size_t)g * (BM * (Kp + 8) + 8) * 2; };
    const int G = smem(9) <= two ? 9 : smem(3) <= two ? 3 : 1;
    const auto f = BM == 32 ? (G == 9 ? k_conv3_dgrad_t<2, 9> : G == 3 ? k_conv3_dgrad_t<2, 3> : k_conv3_dgrad_t<2, 1>)
                            : (G == 9 ? k_conv3_dgrad_t<3, 9> : G == 3 ? k_conv3_dgrad_t<3, 3> : k_conv3_dgrad_t<3, 1>);
    if (tiled(W) && aligned16(dy) && aligned16(dx) && smem_ready((const void *)f, smem(G), G == 1 ? one : two)) {
        const dim3 grid((unsigned)((W + 31) / 32 * ((H + TH - 1) / TH) * B), (ci + BM - 1) / BM);
        fdtd::launch_pdl_smem(f, grid, 256, smem(G), st, dy, w, dx, ci, co, Kp, B, H, W, add);
    } else {
        conv3<true>(dy, w, nullptr, dx, ci, co, (long long)B * H * W, H, W, add, 0, 1, nullptr, st);
    }
    return status();
}

int nn_conv3_wgrad(const float *dy, const float *x, float *gw, int ci, int co, int B, int H, int W, float *work,
                   long long work_elems, void *stream)
{
    if (!dy || !x || !gw || !sizes_ok(ci, co, B, H, W) || work_elems < 0 || (work_elems > 0 && !work)) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    const long long P = (long long)B * H * W;
    long long kc = 0;
    const int N = 9 * ci, splits = nn_splitk_bf16(co, N, P, work_elems, &kc);
    // tiles of 32, 48 or 96 rows x 128 columns; the K slices make about two
    // blocks per SM, so few rows take more warps with less each (32 rows: eight
    // warps of 16 rows 3.45, four of 32 3.55 ms per 8 x 256^2 training step; 48
    // rows as four of 48 or twelve of 16 the same, 96 as eight of 48 3.55, of
    // 32 3.58)
    const int gx = (N + 127) / 128;
    if (W % 4 == 0 && aligned16(dy) && aligned16(x)) {
        if (co <= 32)
            fdtd::launch_pdl_smem(k_conv3_wgrad_t<1, 2>, dim3(gx, 1, splits), 256, 0, st, dy, x, gw, ci, co, B, H, W, kc, work);
        else if (co <= 48)
            fdtd::launch_pdl_smem(k_conv3_wgrad_t<3, 1>, dim3(gx, 1, splits), 128, 0, st, dy, x, gw, ci, co, B, H, W, kc, work);
        else
            fdtd::launch_pdl_smem(k_conv3_wgrad_t<3, 2>, dim3(gx, (co + 95) / 96, splits), 256, 0, st, dy, x, gw, ci, co, B, H, W, kc, work);
    } else if (co <= 32)
        fdtd::launch_pdl_smem(k_conv3_wgrad<1, 2, 4>, dim3(gx, 1, splits), 256, 0, st, dy, x, gw, ci, co, P, H, W, kc, work);
    else if (co <= 48)
        fdtd::launch_pdl_smem(k_conv3_wgrad<1, 3, 4>, dim3(gx, 1, splits), 384, 0, st, dy, x, gw, ci, co, P, H, W, kc, work);
    else
        fdtd::launch_pdl_smem(k_conv3_wgrad<3, 2, 4>, dim3(gx, (co + 95) / 96, splits), 256, 0, st, dy, x, gw, ci, co, P, H, W, kc, work);
    if (splits > 1) fdtd::launch_pdl_smem(k_slices, slice_blocks((long long)co * N, 64), 64, 0, st, gw, work, (long long)co * N, splits);
    return status();
}

int nn_conv3_col_elems(int ci, int co, int B, int H, int W, long long *elems)
{
    if (!elems || !sizes_ok(ci, co, B, H, W)) return 1;
    const long long P = (long long)B * H * W;
    *elems = columns_fwd(ci, co, P, W) || columns_dgrad(ci, co, P, W) ? 9LL * ci * P : 0;
    return 0;
}

int nn_conv3_fwd_col(const float *x, const float *w, const float *bias, float *y, int ci, int co, int B, int H, int W,
                     int relu, float *work, long long work_elems, float *col, long long col_elems, void *stream)
{
    const long long P = (long long)B * H * W;
    if (!col || !sizes_ok(ci, co, B, H, W) || !columns_fwd(ci, co, P, W) || col_elems < 9LL * ci * P || !bias)
        return nn_conv3_fwd(x, w, bias, y, ci, co, B, H, W, relu, work, work_elems, stream);
    const int K = 9 * ci, N = (int)P;
    int rc = nn_im2col3(x, ci, B, H, W, col, stream);
    if (!rc) rc = nn_gemm_bf16(0, 0, co, N, K, 1.0f, w, K, col, N, 0.0f, y, N, work, work_elems, stream);
    return rc ? rc : nn_bias_act(y, bias, co, P, relu, stream);
}

int nn_conv3_dgrad_col(const float *dy, const float *w, float *dx, int ci, int co, int B, int H, int W, int add, float *work,
                       long long work_elems, float *col, long long col_elems, void *stream)
{
    const long long P = (long long)B * H * W;
    if (!col || !dx || !sizes_ok(ci, co, B, H, W) || !columns_dgrad(ci, co, P, W) || col_elems < 9LL * ci * P)
        return nn_conv3_dgrad(dy, w, dx, ci, co, B, H, W, add, stream);
    const int K = 9 * ci, N = (int)P;
    int rc = nn_gemm_bf16(1, 0, K, N, co, 1.0f, w, K, dy, N, 0.0f, col, N, work, work_elems, stream);
    if (!rc && !add) rc = nn_zero(dx, ci * P, stream);
    return rc ? rc : nn_col2im3_add(col, ci, B, H, W, dx, stream);
}

}  // extern "C"
