// Kernels of the learned sensitivity surrogate (a small conv U-Net): a tiled
// FP32 GEMM and a BF16 tensor-core GEMM (mma.sync, FP32 accumulation), im2col
// / col2im for 3x3 convolutions, bias + ReLU, 2x2 average pooling, 2x
// nearest upsampling, MSE loss and Adam.  Not part of the paper;
// the surrogate proposes intermediate design steps between adjoint runs.
//
// Activations use the layout [C][B][H][W]: a convolution is the product
// W[Cout][Cin K K] . col[Cin K K][B H W], and concatenating along channels is
// placing tensors next to each other in memory.
#include <cuda_bf16.h>
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <mutex>
#include <stdint.h>

#include "../../include/surrogate.h"
#include "launch.cuh"

namespace {

constexpr int TPB = 256;
inline int blocks_for(long long n, int cap = 152 * 16)
{
    long long b = (n + TPB - 1) / TPB;
    return (int)(b < 1 ? 1 : (b < cap ? b : cap));
}

// C[M][N] = alpha op(A) op(B) + beta C, row-major.  op(A) is M x K (A stored
// K x M when TA), op(B) is K x N (B stored N x K when TB).  64 x 64 output
// tiles, 16-deep K slices in shared memory, 4 x 4 outputs per thread.
constexpr int GT = 64, GK = 16;

// Split K: blockIdx.z takes the K slice [z kc, (z + 1) kc); with more than
// one slice each slice writes alpha times its partial tile to part[z] (M x N,
// row-major) and k_splitk_sum adds the slices in order, so the result does
// not depend on which block finishes first.
template <bool TA, bool TB>
__global__ void __launch_bounds__(256) k_gemm(int M, int N, int K, float alpha, const float *__restrict__ A, int lda,
                                              const float *__restrict__ B, int ldb, float beta, float *C, int ldc,
                                              int kc, float *part)
{
    fdtd::pdl_wait();
    __shared__ float As[GK][GT + 4];
    __shared__ float Bs[GK][GT + 4];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
    float acc[4][4] = {};
    const int kb = blockIdx.z * kc, ke = min(K, kb + kc);
    for (int k0 = kb; k0 < ke; k0 += GK) {
        // 64 x 16 elements of each operand, 4 per thread.
        for (int e = threadIdx.x; e < GT * GK; e += 256) {
            int mm, kk;
            if (TA) { kk = e / GT; mm = e % GT; }   // A stored K x M: consecutive m
            else { mm = e / GK; kk = e % GK; }      // A stored M x K: consecutive k
            const int gm = m0 + mm, gk = k0 + kk;
            float v = 0.0f;
            if (gm < M && gk < ke) v = TA ? A[(long long)gk * lda + gm] : A[(long long)gm * lda + gk];
            As[kk][mm] = v;
            int nn2, kk2;
            if (TB) { nn2 = e / GK; kk2 = e % GK; }  // B stored N x K: consecutive k
            else { kk2 = e / GT; nn2 = e % GT; }     // B stored K x N: consecutive n
            const int gn = n0 + nn2, gk2 = k0 + kk2;
            float u = 0.0f;
            if (gn < N && gk2 < ke) u = TB ? B[(long long)gn * ldb + gk2] : B[(long long)gk2 * ldb + gn];
            Bs[kk2][nn2] = u;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int gm = m0 + ty + 16 * i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gn = n0 + tx + 16 * j;
            if (gn >= N) continue;
            if (gridDim.z > 1) {
                part[((long long)blockIdx.z * M + gm) * N + gn] = alpha * acc[i][j];
            } else {
                float *c = C + (long long)gm * ldc + gn;
                *c = alpha * acc[i][j] + (beta != 0.0f ? beta * *c : 0.0f);
            }
        }
    }
}

// C = sum over s = 0 .. S-1 of part[s] (in that order) + beta C.
__global__ void k_splitk_sum(float *C, int ldc, const float *__restrict__ part, int M, int N, int S, float beta)
{
    fdtd::pdl_wait();
    const long long n = (long long)M * N;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        float acc = part[e];
        for (int z = 1; z < S; ++z) acc += part[z * n + e];
        float *c = C + (e / N) * ldc + e % N;
        *c = acc + (beta != 0.0f ? beta * *c : 0.0f);
    }
}

// col[(c*9 + t)][(b*H + y)*W + x] = x[c][b][y + dy_t][x + dx_t] (zero padding).
// One thread per (c, pixel) writes the pixel's nine taps: the index
// arithmetic is done once, the nine stores of a warp are each contiguous.
__global__ void k_im2col3(const float *x, int C, int B, int H, int W, float *col)
{
    fdtd::pdl_wait();
    const int HW = H * W;
    const long long P = (long long)B * HW, n = (long long)C * P;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e / P);
        const long long p = e - (long long)c * P;
        const int b = (int)(p / HW), rem = (int)(p - (long long)b * HW);
        const int yy = rem / W, xx = rem - yy * W;
        const float *src = x + ((long long)c * B + b) * HW;
        float *dst = col + (long long)c * 9 * P + p;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int sy = yy + t / 3 - 1, sx = xx + t % 3 - 1;
            dst[(long long)t * P] = (sy >= 0 && sy < H && sx >= 0 && sx < W) ? src[sy * W + sx] : 0.0f;
        }
    }
}

// Adjoint of im2col: dx[c][b][y][x] += sum over taps of dcol at the pixels
// that read it (gathered, so no atomics).
__global__ void k_col2im3(const float *col, int C, int B, int H, int W, float *dx)
{
    fdtd::pdl_wait();
    const long long P = (long long)B * H * W, n = (long long)C * P;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e / P);
        const long long p = e % P;
        const int xx = (int)(p % W), yy = (int)((p / W) % H), b = (int)(p / ((long long)W * H));
        float s = 0.0f;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            // pixel (oy, ox) read (yy, xx) through tap t when oy + t/3 - 1 = yy
            const int oy = yy - (t / 3 - 1), ox = xx - (t % 3 - 1);
            if (oy >= 0 && oy < H && ox >= 0 && ox < W)
                s += col[((long long)c * 9 + t) * P + ((long long)b * H + oy) * W + ox];
        }
        dx[e] += s;
    }
}

__global__ void k_bias_act(float *y, const float *bias, int Cout, long long P, int relu)
{
    fdtd::pdl_wait();
    const long long n = (long long)Cout * P;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        float v = y[e] + bias[e / P];
        y[e] = relu && v < 0.0f ? 0.0f : v;
    }
}

// dy <- dy * (y > 0) where relu, then db[c] = sum over the row: one block
// of 1024 threads per row, 16-byte accesses when `vec` (P a multiple of 4,
// both arrays 16-byte aligned), a fixed summation order.
__global__ void __launch_bounds__(1024) k_relu_bwd_bias(const float *y, float *dy, float *db, long long P, int relu,
                                                        int vec)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    __shared__ float part[32];
    const int c = blockIdx.x;
    float s = 0.0f;
    const float *yr = y + (long long)c * P;
    float *dr = dy + (long long)c * P;
    if (vec) {
        const float4 *y4 = reinterpret_cast<const float4 *>(yr);
        float4 *d4 = reinterpret_cast<float4 *>(dr);
        for (long long p = threadIdx.x; p < P / 4; p += blockDim.x) {
            float4 g = d4[p];
            if (relu) {
                const float4 v = y4[p];
                if (!(v.x > 0.0f)) g.x = 0.0f;
                if (!(v.y > 0.0f)) g.y = 0.0f;
                if (!(v.z > 0.0f)) g.z = 0.0f;
                if (!(v.w > 0.0f)) g.w = 0.0f;
                d4[p] = g;
            }
            s += (g.x + g.y) + (g.z + g.w);
        }
    } else {
        for (long long p = threadIdx.x; p < P; p += blockDim.x) {
            float g = dr[p];
            if (relu && !(yr[p] > 0.0f)) g = 0.0f;
            dr[p] = g;
            s += g;
        }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0f;
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) db[c] = s;
    }
}

// The same for long rows: the 32 warps of a channel's block as a cluster of
// eight blocks.  One block per channel left 24 of 152 SMs busy on the widest
// layers (82 us for 24 x 524288 values, 150 MB; 26 us so).  Every thread adds
// the values it would have added there, in that order, and the warps' sums
// are added in theirs: the same bits.
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(128)
k_relu_bwd_bias8(const float *__restrict__ y, float *dy, float *db, long long P, int relu)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    __shared__ float part[32];
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();
    const int rank = blockIdx.x & 7, c = blockIdx.x >> 3, warp = rank * 4 + (threadIdx.x >> 5);
    const float4 *y4 = reinterpret_cast<const float4 *>(y + (long long)c * P);
    float4 *d4 = reinterpret_cast<float4 *>(dy + (long long)c * P);
    float s = 0.0f;
    for (long long p0 = rank * 128 + threadIdx.x; p0 < P / 4; p0 += 8 * 1024) {
        float4 g[8], v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (p0 + q * 1024 < P / 4) {
                g[q] = d4[p0 + q * 1024];
                if (relu) v[q] = y4[p0 + q * 1024];
            }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (p0 + q * 1024 < P / 4) {
                if (relu) {
                    if (!(v[q].x > 0.0f)) g[q].x = 0.0f;
                    if (!(v[q].y > 0.0f)) g[q].y = 0.0f;
                    if (!(v[q].z > 0.0f)) g[q].z = 0.0f;
                    if (!(v[q].w > 0.0f)) g[q].w = 0.0f;
                    d4[p0 + q * 1024] = g[q];
                }
                s += (g[q].x + g[q].y) + (g[q].z + g[q].w);
            }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    cl.barrier_wait();  // the first block has started: its shared memory can be written
    if ((threadIdx.x & 31) == 0) *cl.map_shared_rank(part + warp, 0) = s;
    cl.sync();
    if (rank == 0 && threadIdx.x < 32) {
        s = part[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) db[c] = s;
    }
}

// 2 x 2 average pooling of planes [n][H][W] -> [n][H/2][W/2] and its adjoint.
__global__ void k_pool2(const float *x, long long planes, int H, int W, float *y)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    const int h = H / 2, w = W / 2;
    const long long n = planes * h * w;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const long long pl = e / ((long long)h * w);
        const int yy = (int)((e / w) % h), xx = (int)(e % w);
        const float *s = x + (pl * H + 2 * yy) * W + 2 * xx;
        y[e] = 0.25f * (s[0] + s[1] + s[W] + s[W + 1]);
    }
}

__global__ void k_pool2_bwd(const float *dy, long long planes, int H, int W, float *dx)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    const long long n = planes * H * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const long long pl = e / ((long long)H * W);
        const int yy = (int)((e / W) % H), xx = (int)(e % W);
        dx[e] += 0.25f * dy[(pl * (H / 2) + yy / 2) * (W / 2) + xx / 2];
    }
}

// 2x nearest upsampling of planes [n][h][w] -> [n][2h][2w] and its adjoint.
__global__ void k_up2(const float *x, long long planes, int h, int w, float *y)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    const int H = 2 * h, W = 2 * w;
    const long long n = planes * H * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const long long pl = e / ((long long)H * W);
        const int yy = (int)((e / W) % H), xx = (int)(e % W);
        y[e] = x[(pl * h + yy / 2) * w + xx / 2];
    }
}

__global__ void k_up2_bwd(const float *dy, long long planes, int h, int w, float *dx)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    const long long n = planes * h * w;
    const int W = 2 * w;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const long long pl = e / ((long long)h * w);
        const int yy = (int)((e / w) % h), xx = (int)(e % w);
        const float *s = dy + (pl * 2 * h + 2 * yy) * W + 2 * xx;
        dx[e] += s[0] + s[1] + s[W] + s[W + 1];
    }
}

// The resampling passes with rows of even w and 16-byte aligned planes: a
// thread has two coarse pixels, a float2, and their 2 x 2 fine ones, two
// float4 (the passes are bound by HBM: one value per thread with its index
// divisions took 99 us instead of 19 for k_up2 to 48 x 8 planes of 256^2, 55
// instead of 15 for k_pool2_bwd).  F(coarse, fine, w4) on float2 / float4
// words: fine[0] and fine[w4] are the two rows.
template <class F>
__device__ __forceinline__ void each_pair(long long planes, int h, int w, F f)
{
    const int w2 = w / 2;
    const long long n = planes * h * w2;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        f(e, (e / w2 * 2) * w2 + e % w2, w2);  // fine rows of w2 float4
}

__global__ void k_pool2_v(const float4 *__restrict__ x, long long planes, int h, int w, float2 *y)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    each_pair(planes, h, w, [&](long long c, long long f, int w4) {
        const float4 a = x[f], b = x[f + w4];
        y[c] = make_float2(0.25f * (a.x + a.y + b.x + b.y), 0.25f * (a.z + a.w + b.z + b.w));
    });
}

__global__ void k_pool2_bwd_v(const float2 *__restrict__ dy, long long planes, int h, int w, float4 *dx)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    each_pair(planes, h, w, [&](long long c, long long f, int w4) {
        const float2 g = dy[c];
        float4 a = dx[f], b = dx[f + w4];
        a.x += 0.25f * g.x;
        a.y += 0.25f * g.x;
        a.z += 0.25f * g.y;
        a.w += 0.25f * g.y;
        b.x += 0.25f * g.x;
        b.y += 0.25f * g.x;
        b.z += 0.25f * g.y;
        b.w += 0.25f * g.y;
        dx[f] = a;
        dx[f + w4] = b;
    });
}

__global__ void k_up2_v(const float2 *__restrict__ x, long long planes, int h, int w, float4 *y)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    each_pair(planes, h, w, [&](long long c, long long f, int w4) {
        const float2 v = x[c];
        y[f] = y[f + w4] = make_float4(v.x, v.x, v.y, v.y);
    });
}

__global__ void k_up2_bwd_v(const float4 *__restrict__ dy, long long planes, int h, int w, float2 *dx)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    each_pair(planes, h, w, [&](long long c, long long f, int w4) {
        const float4 a = dy[f], b = dy[f + w4];
        float2 v = dx[c];
        v.x += a.x + a.y + b.x + b.y;
        v.y += a.z + a.w + b.z + b.w;
        dx[c] = v;
    });
}

bool pairs_ok(int w, const void *coarse, const void *fine)
{
    return w % 2 == 0 && ((uintptr_t)coarse & 7) == 0 && ((uintptr_t)fine & 15) == 0;
}

// loss = mean (y - t)^2 (FP64 accumulation into *loss, which must start at 0);
// dy = 2 (y - t) / n.
__global__ void k_mse(const float *y, const float *t, long long n, float *dy, double *loss)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    double s = 0.0;
    const float inv = 2.0f / (float)n;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const float d = y[e] - t[e];
        dy[e] = inv * d;
        s += (double)d * (double)d;
    }
    // one atomic per block: one per warp made 16384 of them on one address for 2 MB (30 us; 8 so)
    __shared__ double part[TPB / 32];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < TPB / 32; ++q) s += part[q];
        atomicAdd(loss, s / (double)n);
    }
}

// Adam on up to ADAM_T tensors in one launch: blocks of ADAM_E elements, the
// blocks of tensor i from first[i] on.  The base-24 network's 30 tensors took
// 30 launches of 4 us each, most of them a few blocks; 11 us so.
constexpr int ADAM_T = 64, ADAM_E = 1024;

struct AdamList {
    float *p[ADAM_T], *m[ADAM_T], *v[ADAM_T];
    const float *g[ADAM_T];
    long long n[ADAM_T];
    int first[ADAM_T + 1];
    int count;
};

__global__ void __launch_bounds__(TPB) k_adam(const __grid_constant__ AdamList L, float lr, float b1, float b2, float eps,
                                              float c1, float c2)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    int i = 0, hi = L.count - 1;
    while (i < hi) {
        const int mid = (i + hi + 1) / 2;
        if (L.first[mid] <= (int)blockIdx.x) i = mid;
        else hi = mid - 1;
    }
    float *p = L.p[i], *m = L.m[i], *v = L.v[i];
    const float *g = L.g[i];
    const long long n = L.n[i], step = (long long)(L.first[i + 1] - L.first[i]) * ADAM_E;
    for (long long e0 = (long long)(blockIdx.x - L.first[i]) * ADAM_E; e0 < n; e0 += step)
#pragma unroll
        for (int q = 0; q < ADAM_E / TPB; ++q) {
            const long long e = e0 + q * TPB + threadIdx.x;
            if (e >= n) break;
            const float gg = g[e];
            const float mm = b1 * m[e] + (1.0f - b1) * gg;
            const float vv = b2 * v[e] + (1.0f - b2) * gg * gg;
            m[e] = mm;
            v[e] = vv;
            p[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
        }
}

__global__ void k_zero_f(float *x, long long n)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        x[e] = 0.0f;
}

int status(cudaStream_t) { return cudaGetLastError() == cudaSuccess ? 0 : 3; }

}  // namespace

namespace {

// BF16 tensor-core GEMM (mma.sync m16n8k16, FP32 accumulation).  Block tile
// 64 (M) x 128 (N), K in slices of 32: each slice of op(A) and op(B) is read
// as FP32 from global memory (coalesced along whichever index is
// contiguous), rounded to BF16 (nearest even) and stored k-contiguous in
// shared memory, As[m][k] and Bs[n][k], rows padded to 40 elements so that
// the fragment loads of a warp hit 32 distinct banks.  Eight warps, 2 along
// M x 4 along N, each own a 32 x 32 sub-tile: 2 x 4 fragments of 16 x 8.
constexpr int BM = 64, BN = 128, BK = 32, BKP = BK + 8;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], const unsigned (&b)[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ unsigned lds32(const __nv_bfloat16 *p) { return *reinterpret_cast<const unsigned *>(p); }

// C = alpha op(A) op(B) + beta C as in k_gemm (split K over blockIdx.z).
template <bool TA, bool TB>
__global__ void __launch_bounds__(256) k_gemm_bf16(int M, int N, int K, float alpha, const float *__restrict__ A,
                                                   int lda, const float *__restrict__ B, int ldb, float beta,
                                                   float *C, int ldc, int kc, float *part)
{
    fdtd::pdl_wait();
    __shared__ __align__(16) __nv_bfloat16 As[BM][BKP];
    __shared__ __align__(16) __nv_bfloat16 Bs[BN][BKP];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = warp >> 2, wn = warp & 3;
    const int g = lane >> 2, t = lane & 3;  // fragment row / column group
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int jn = 0; jn < 4; ++jn)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][jn][r] = 0.0f;
    const int kb = blockIdx.z * kc, ke = min(K, kb + kc);
    for (int k0 = kb; k0 < ke; k0 += BK) {
        for (int e = threadIdx.x; e < BM * BK; e += 256) {
            int mm, kk;
            if (TA) { kk = e / BM; mm = e % BM; }  // A stored K x M: consecutive m
            else { mm = e / BK; kk = e % BK; }     // A stored M x K: consecutive k
            const int gm = m0 + mm, gk = k0 + kk;
            float v = 0.0f;
            if (gm < M && gk < ke) v = TA ? A[(long long)gk * lda + gm] : A[(long long)gm * lda + gk];
            As[mm][kk] = __float2bfloat16_rn(v);
        }
        for (int e = threadIdx.x; e < BN * BK; e += 256) {
            int nn, kk;
            if (TB) { nn = e / BK; kk = e % BK; }  // B stored N x K: consecutive k
            else { kk = e / BN; nn = e % BN; }     // B stored K x N: consecutive n
            const int gn = n0 + nn, gk = k0 + kk;
            float v = 0.0f;
            if (gn < N && gk < ke) v = TB ? B[(long long)gn * ldb + gk] : B[(long long)gk * ldb + gn];
            Bs[nn][kk] = __float2bfloat16_rn(v);
        }
        __syncthreads();
#pragma unroll
        for (int ks = 0; ks < BK; ks += 16) {
            unsigned a[2][4], b[4][2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = wm * 32 + i * 16 + g, c = ks + 2 * t;
                a[i][0] = lds32(&As[r][c]);
                a[i][1] = lds32(&As[r + 8][c]);
                a[i][2] = lds32(&As[r][c + 8]);
                a[i][3] = lds32(&As[r + 8][c + 8]);
            }
#pragma unroll
            for (int jn = 0; jn < 4; ++jn) {
                const int n = wn * 32 + jn * 8 + g, c = ks + 2 * t;
                b[jn][0] = lds32(&Bs[n][c]);
                b[jn][1] = lds32(&Bs[n][c + 8]);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int jn = 0; jn < 4; ++jn) mma_bf16(acc[i][jn], a[i], b[jn]);
        }
        __syncthreads();
    }
    // accumulator r of fragment (i, jn): row g (+8 for r >= 2), column 2t (+1 for odd r)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int jn = 0; jn < 4; ++jn)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int gm = m0 + wm * 32 + i * 16 + g + (r >= 2 ? 8 : 0);
                const int gn = n0 + wn * 32 + jn * 8 + 2 * t + (r & 1);
                if (gm >= M || gn >= N) continue;
                if (gridDim.z > 1) {
                    part[((long long)blockIdx.z * M + gm) * N + gn] = alpha * acc[i][jn][r];
                } else {
                    float *c = C + (long long)gm * ldc + gn;
                    *c = alpha * acc[i][jn][r] + (beta != 0.0f ? beta * *c : 0.0f);
                }
            }
}

// K = 1: C[m][n] = alpha a[m] b[n] + beta C[m][n], four columns per thread, OUTER_M rows per block.
constexpr int OUTER_M = 8;
__global__ void __launch_bounds__(TPB) k_outer_bf16(int M, int N, float alpha, const float *__restrict__ A, int as,
                                                    const float *__restrict__ B, float beta, float *C, int ldc)
{
    fdtd::pdl_wait();
    fdtd::pdl_trigger();
    const int n = (blockIdx.x * TPB + threadIdx.x) * 4, m0 = blockIdx.y * OUTER_M;
    if (n >= N) return;
    auto bf = [](float v) { return __bfloat162float(__float2bfloat16_rn(v)); };
    const float4 b = *reinterpret_cast<const float4 *>(B + n);
    const float bv[4] = {bf(b.x), bf(b.y), bf(b.z), bf(b.w)};
    float4 old[OUTER_M];
#pragma unroll
    for (int i = 0; i < OUTER_M; ++i)
        if (beta != 0.0f && m0 + i < M) old[i] = *reinterpret_cast<const float4 *>(C + (long long)(m0 + i) * ldc + n);
#pragma unroll
    for (int i = 0; i < OUTER_M; ++i) {
        if (m0 + i >= M) break;
        const float a = bf(A[(long long)(m0 + i) * as]);
        const float c[4] = {old[i].x, old[i].y, old[i].z, old[i].w};
        float o[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) o[v] = alpha * (a * bv[v]) + (beta != 0.0f ? beta * c[v] : 0.0f);
        *reinterpret_cast<float4 *>(C + (long long)(m0 + i) * ldc + n) = make_float4(o[0], o[1], o[2], o[3]);
    }
}

}  // namespace

extern "C" {

// K slices of one product: with few output tiles and a long K (weight
// gradients), enough slices to give every SM a couple of blocks, as many as
// the scratch (work_elems floats, M x N per slice) holds; kc receives the
// slice depth (a multiple of `step`).
static int splitk(int M, int N, int K, long long tiles, int step, long long work_elems, int *kc)
{
    long long splits = 1;
    if (tiles < 2 * 152 && K > 8 * step) {
        const long long want = (2 * 152 + tiles - 1) / tiles, most = (K + 4 * step - 1) / (4 * step);
        splits = want < most ? want : most;
    }
    const long long fit = work_elems / ((long long)M * N);
    if (splits > fit) splits = fit > 1 ? fit : 1;
    *kc = (int)(((K + splits - 1) / splits + step - 1) / step * step);
    return (K + *kc - 1) / *kc;
}

// The K slices nn_gemm_bf16 takes for an M x N x K product, for the kernels
// that reproduce its sums (conv.cu).
int nn_splitk_bf16(int M, long long N, long long K, long long work_elems, long long *kc)
{
    int k = 0;
    const int s = splitk(M, (int)N, (int)K, (N + BN - 1) / BN * ((M + BM - 1) / BM), BK, work_elems, &k);
    *kc = k;
    return s;
}

int nn_gemm(int transA, int transB, int M, int N, int K, float alpha, const float *A, int lda, const float *B, int ldb,
            float beta, float *C, int ldc, float *work, long long work_elems, void *stream)
{
    if (M < 0 || N < 0 || K < 0 || !C || (K > 0 && (!A || !B)) || work_elems < 0 || (work_elems > 0 && !work))
        return 1;
    if (M == 0 || N == 0) return 0;
    cudaStream_t st = (cudaStream_t)stream;
    int kc = 0;
    const int splits = splitk(M, N, K, (long long)((N + GT - 1) / GT) * ((M + GT - 1) / GT), GK, work_elems, &kc);
    dim3 grid((N + GT - 1) / GT, (M + GT - 1) / GT, splits);
    if (!transA && !transB) fdtd::launch_pdl_smem(k_gemm<false, false>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    else if (!transA && transB) fdtd::launch_pdl_smem(k_gemm<false, true>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    else if (transA && !transB) fdtd::launch_pdl_smem(k_gemm<true, false>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    else fdtd::launch_pdl_smem(k_gemm<true, true>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    if (splits > 1) fdtd::launch_pdl_smem(k_splitk_sum, blocks_for((long long)M * N), TPB, 0, st, C, ldc, work, M, N, splits, beta);
    return status(st);
}

int nn_gemm_bf16(int transA, int transB, int M, int N, int K, float alpha, const float *A, int lda, const float *B,
                 int ldb, float beta, float *C, int ldc, float *work, long long work_elems, void *stream)
{
    if (M < 0 || N < 0 || K < 0 || !C || (K > 0 && (!A || !B)) || work_elems < 0 || (work_elems > 0 && !work))
        return 1;
    if (M == 0 || N == 0) return 0;
    if (K == 0) return nn_gemm(transA, transB, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, work, work_elems, stream);
    cudaStream_t st = (cudaStream_t)stream;
    if (K == 1 && !transB && N % 4 == 0 && ldc % 4 == 0 && (((uintptr_t)B | (uintptr_t)C) & 15) == 0 &&
        M <= 65535 * OUTER_M) {
        // nothing to sum: the tiles of k_gemm_bf16 would be one thirty-second full
        // (input gradient of the 1 x 1 head, 24 x 524288: 68 us, 15 so)
        fdtd::launch_pdl_smem(k_outer_bf16, dim3((N / 4 + TPB - 1) / TPB, (M + OUTER_M - 1) / OUTER_M), TPB, 0, st, M, N,
                              alpha, A, transA ? 1 : lda, B, beta, C, ldc);
        return status(st);
    }
    int kc = 0;
    const int splits = splitk(M, N, K, (long long)((N + BN - 1) / BN) * ((M + BM - 1) / BM), BK, work_elems, &kc);
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, splits);
    if (!transA && !transB) fdtd::launch_pdl_smem(k_gemm_bf16<false, false>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    else if (!transA && transB) fdtd::launch_pdl_smem(k_gemm_bf16<false, true>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    else if (transA && !transB) fdtd::launch_pdl_smem(k_gemm_bf16<true, false>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    else fdtd::launch_pdl_smem(k_gemm_bf16<true, true>, grid, 256, 0, st, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, kc, work);
    if (splits > 1) fdtd::launch_pdl_smem(k_splitk_sum, blocks_for((long long)M * N), TPB, 0, st, C, ldc, work, M, N, splits, beta);
    return status(st);
}

int nn_im2col3(const float *x, int C, int B, int H, int W, float *col, void *stream)
{
    if (!x || !col || C <= 0 || B <= 0 || H <= 0 || W <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    fdtd::launch_pdl_smem(k_im2col3, blocks_for((long long)C * 9 * B * H * W), TPB, 0, st, x, C, B, H, W, col);
    return status(st);
}

int nn_col2im3_add(const float *col, int C, int B, int H, int W, float *dx, void *stream)
{
    if (!col || !dx || C <= 0 || B <= 0 || H <= 0 || W <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    fdtd::launch_pdl_smem(k_col2im3, blocks_for((long long)C * B * H * W), TPB, 0, st, col, C, B, H, W, dx);
    return status(st);
}

int nn_bias_act(float *y, const float *bias, int Cout, long long P, int relu, void *stream)
{
    if (!y || !bias || Cout <= 0 || P <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    fdtd::launch_pdl_smem(k_bias_act, blocks_for((long long)Cout * P), TPB, 0, st, y, bias, Cout, P, relu);
    return status(st);
}

int nn_act_bwd_bias(const float *y, float *dy, float *db, int Cout, long long P, int relu, void *stream)
{
    if (!y || !dy || !db || Cout <= 0 || P <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    const int vec = (P & 3) == 0 && (((uintptr_t)y | (uintptr_t)dy) & 15) == 0;
    if (vec && P >= 8 * 4096)  // eight values' loads in flight per thread; below, one block has them all at once
        fdtd::launch_pdl_smem(k_relu_bwd_bias8, 8 * Cout, 128, 0, st, y, dy, db, P, relu);
    else
        fdtd::launch_pdl_smem(k_relu_bwd_bias, Cout, 1024, 0, st, y, dy, db, P, relu, vec);
    return status(st);
}

int nn_pool2(const float *x, long long planes, int H, int W, float *y, void *stream)
{
    if (!x || !y || planes <= 0 || H < 2 || W < 2 || (H | W) & 1) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    if (pairs_ok(W / 2, y, x))
        fdtd::launch_pdl_smem(k_pool2_v, blocks_for(planes * (H / 2) * (W / 4)), TPB, 0, st, (const float4 *)x, planes, H / 2, W / 2, (float2 *)y);
    else
        fdtd::launch_pdl_smem(k_pool2, blocks_for(planes * (H / 2) * (W / 2)), TPB, 0, st, x, planes, H, W, y);
    return status(st);
}

int nn_pool2_bwd_add(const float *dy, long long planes, int H, int W, float *dx, void *stream)
{
    if (!dy || !dx || planes <= 0 || H < 2 || W < 2 || (H | W) & 1) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    if (pairs_ok(W / 2, dy, dx))
        fdtd::launch_pdl_smem(k_pool2_bwd_v, blocks_for(planes * (H / 2) * (W / 4)), TPB, 0, st, (const float2 *)dy, planes, H / 2, W / 2, (float4 *)dx);
    else
        fdtd::launch_pdl_smem(k_pool2_bwd, blocks_for(planes * H * W), TPB, 0, st, dy, planes, H, W, dx);
    return status(st);
}

int nn_up2(const float *x, long long planes, int h, int w, float *y, void *stream)
{
    if (!x || !y || planes <= 0 || h <= 0 || w <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    if (pairs_ok(w, x, y))
        fdtd::launch_pdl_smem(k_up2_v, blocks_for(planes * h * (w / 2)), TPB, 0, st, (const float2 *)x, planes, h, w, (float4 *)y);
    else
        fdtd::launch_pdl_smem(k_up2, blocks_for(planes * 4 * h * w), TPB, 0, st, x, planes, h, w, y);
    return status(st);
}

int nn_up2_bwd_add(const float *dy, long long planes, int h, int w, float *dx, void *stream)
{
    if (!dy || !dx || planes <= 0 || h <= 0 || w <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    if (pairs_ok(w, dx, dy))
        fdtd::launch_pdl_smem(k_up2_bwd_v, blocks_for(planes * h * (w / 2)), TPB, 0, st, (const float4 *)dy, planes, h, w, (float2 *)dx);
    else
        fdtd::launch_pdl_smem(k_up2_bwd, blocks_for(planes * h * w), TPB, 0, st, dy, planes, h, w, dx);
    return status(st);
}

int nn_mse(const float *y, const float *t, long long n, float *dy, double *loss, void *stream)
{
    if (!y || !t || !dy || !loss || n <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    fdtd::launch_pdl_smem(k_zero_f, 1, 32, 0, st, (float *)loss, 2);
    fdtd::launch_pdl_smem(k_mse, blocks_for(n, 2 * 152), TPB, 0, st, y, t, n, dy, loss);
    return status(st);
}

int nn_adam_multi(int count, float *const *p, const float *const *g, float *const *m, float *const *v, const long long *n,
                  float lr, float beta1, float beta2, float eps, int step, void *stream)
{
    if (count <= 0 || !p || !g || !m || !v || !n || step < 1) return 1;
    for (int i = 0; i < count; ++i)
        if (!p[i] || !g[i] || !m[i] || !v[i] || n[i] <= 0) return 1;
    cudaStream_t st = (cudaStream_t)stream;
    const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
    for (int i0 = 0; i0 < count; i0 += ADAM_T) {
        AdamList L;
        L.count = count - i0 < ADAM_T ? count - i0 : ADAM_T;
        int blocks = 0;
        for (int i = 0; i < L.count; ++i) {
            L.p[i] = p[i0 + i];
            L.g[i] = g[i0 + i];
            L.m[i] = m[i0 + i];
            L.v[i] = v[i0 + i];
            L.n[i] = n[i0 + i];
            L.first[i] = blocks;
            const long long b = (L.n[i] + ADAM_E - 1) / ADAM_E;
            blocks += (int)(b < 152 * 16 ? b : 152 * 16);
        }
        L.first[L.count] = blocks;
        fdtd::launch_pdl_smem(k_adam, blocks, TPB, 0, st, L, lr, beta1, beta2, eps, c1, c2);
    }
    return status(st);
}

int nn_adam(float *p, const float *g, float *m, float *v, long long n, float lr, float beta1, float beta2, float eps,
            int step, void *stream)
{
    return nn_adam_multi(1, &p, &g, &m, &v, &n, lr, beta1, beta2, eps, step, stream);
}

int nn_zero(float *x, long long n, void *stream)
{
    if (!x || n < 0) return 1;
    if (n == 0) return 0;
    cudaStream_t st = (cudaStream_t)stream;
    fdtd::launch_pdl_smem(k_zero_f, blocks_for(n), TPB, 0, st, x, n);
    return status(st);
}

}  // extern "C"
