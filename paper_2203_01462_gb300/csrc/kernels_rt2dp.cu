// Temporally blocked 2D leapfrog with E in plane (Ex, Ey, Hz + Drude Jx, Jy +
// CPML), the tile held in registers, for sm_103a.
//
// The two half-step launches per step of kernels_2dp.cu are single partial
// waves on the paper's grids (291^2, 491^2: 10 MB, resident in L2), so a step
// cost two launch and load latencies, 5.3 to 6.4 us whatever its work.  Here,
// as in kernels_rt2d.cu, a block owns tw x th nodes with a halo and advances
// up to `halo` steps per launch: a warp holds the region's width (64 columns
// in FP32, 32 in FP64) and one or two rows of Ex, Ey, Hz, Jx, Jy and the Drude
// coefficients of both edges in registers; neighbours along x come by
// shuffle; along y the H half step takes one Ex row from the warp above and
// the E half step one Hz row from the warp below, through shared memory, with
// a block barrier before each.  (Advancing the Hz row below redundantly, as
// the E_z kernel does with Hx to save a barrier, would take a second Ey row
// and its CPML terms too.)  The state goes from one buffer of a ping-pong
// pair into the other; each step spoils one layer of the region from the
// outside, so after `halo` steps the tile is exact and no block waits.
//
// Nodes outside the grid and on the walls hold zeros: an edge that is not
// updated has cb = 0, and Hz past the last cell stays zero because its four
// edges do.
//
// The adjoint run is the same kernel with the gap's source.  Its sensitivity
// sums (Eq. 25) are taken apart: inside the blocked kernel their factors,
// records and sums cost 60 registers a thread, spilled, and 3.3 us per 491^2
// step.  Instead the adjoint records its design edges' E, as the forward run
// does, and k_rt2dp_sens adds up RT2DP_CHUNK steps at a time: it reads both
// records, advances J by its own recurrence (the same operations on the same
// E, so the same bits) and touches the FP64 accumulator once.
#include <algorithm>
#include <type_traits>

#include "coef_slots.cuh"
#include "rt_common.cuh"

namespace fdtd {

namespace {

// VX columns per lane, RPW rows per warp, region width, warps per block.
template <typename R>
struct Shape {
    static constexpr int VX = sizeof(R) == 4 ? 2 : 1;
    static constexpr int RPW = sizeof(R) == 4 ? 2 : 1;
    static constexpr int W = 32 * VX;
    static constexpr int MAXW = sizeof(R) == 4 ? 16 : 24;
};

// Largest gap record (Ex and Ey values) whose adjoint source is staged.
constexpr int GAP_STAGED = 1024;

// Shared memory of one block in words of R: Ex rows to the warp below and Hz
// rows to the warp above [nw + 1][W] each, CPML tables of the columns [6][W]
// and rows [6][nw RPW], source samples, the gap's adjoint source [count][Mg].
template <typename R>
__host__ __device__ size_t smem_words(int nw, int count, int gapw)
{
    using D = Shape<R>;
    return (size_t)2 * (nw + 1) * D::W + 6 * D::W + 6 * (size_t)nw * D::RPW + RT2D_MAX + (size_t)count * gapw;
}

template <typename R, int MODE>
__global__ void __launch_bounds__(32 * Shape<R>::MAXW, 1)
    k_rt2dp(const __grid_constant__ GeoP g, const __grid_constant__ StateP<R> in,
            const __grid_constant__ StateP<R> out, int slot, const __grid_constant__ PmlP<R> pm,
            const __grid_constant__ RtP<R> w)
{
    using D = Shape<R>;
    constexpr int VX = D::VX, RPW = D::RPW, W = D::W;
    extern __shared__ __align__(16) char smem_raw[];
    const Coef<R> &c = coef_at<R>(slot);
    const int lane = threadIdx.x, wi = threadIdx.y, nw = blockDim.y, tid = wi * 32 + lane, nth = nw * 32;
    const int T = w.count, H = w.halo, nx = g.nx, ny = g.ny, np = g.npml, P = g.px, np2 = 2 * np;
    const int xr = blockIdx.x * w.tw - H, yr = blockIdx.y * w.th - H;  // region origin (grid)
    const int i0 = xr + lane * VX, j0 = yr + wi * RPW;                 // this thread's first node
    const int Mg = g.Mgc[0] + g.Mgc[1];
    const R S = c.S;

    R *sU = (R *)smem_raw;          // [nw + 1][W]: a warp's first Ex row, read by the warp below
    R *sD = sU + (nw + 1) * W;      // [nw + 1][W]: a warp's last Hz row, read by the warp above
    R *xt = sD + (nw + 1) * W;      // [6][W]: bE cE kiE bH cH kiH of the columns
    const int YT = nw * RPW;
    R *yt = xt + 6 * W;             // [6][YT]: the same of the rows
    R *ssrc = yt + 6 * YT;
    R *sgap = ssrc + RT2D_MAX;
    // the gap's adjoint source is staged by the blocks whose region holds gap edges
    const bool hasgap = xr < g.g0[0][0] + g.gn[1][0] && xr + W > g.g0[0][0] && yr < g.g0[0][1] + g.gn[0][1] &&
                        yr + nw * RPW > g.g0[0][1];
    const bool gstage = MODE == 1 && Mg <= GAP_STAGED && hasgap && w.gap;
    // The region meets the absorbing layer of the columns / rows.
    const bool xp = np > 0 && (xr < np || xr + W > nx - 1 - np);
    const bool yp = np > 0 && (yr < np || yr + nw * RPW > ny - 1 - np);

    // What the previous launch of the same run does not write is read before
    // waiting for it (see kernels_rt2d.cu).
    if (w.first) pdl_wait();
    pdl_trigger();
    for (int ax = 0; ax < 2; ++ax) {
        if (ax == 0 ? !xp : !yp) continue;
        const int len = ax == 0 ? W : YT, o = ax == 0 ? xr : yr, n = ax == 0 ? nx : ny;
        R *t = ax == 0 ? xt : yt;
        for (int q = tid; q < len; q += nth) {
            const int p = o + q;
            const bool es = (unsigned)p < (unsigned)n && slab_e(p, n, np) >= 0;
            const bool hs = (unsigned)p < (unsigned)n && slab_h(p, n, np) >= 0;
            t[q] = es ? pm.bE[ax][p] : R(0);
            t[len + q] = es ? pm.cE[ax][p] : R(0);
            t[2 * len + q] = es ? pm.kiE[ax][p] : R(1);
            t[3 * len + q] = hs ? pm.bH[ax][p] : R(0);
            t[4 * len + q] = hs ? pm.cH[ax][p] : R(0);
            t[5 * len + q] = hs ? pm.kiH[ax][p] : R(1);
        }
    }
    if (MODE == 0 && tid < T) ssrc[tid] = w.src[w.n0 + tid];
    if (gstage)  // rows n0 - T + 1 .. n0 are consecutive
        for (int q = tid; q < T * Mg; q += nth) sgap[q] = w.gap[(long long)(w.n0 - T + 1) * Mg + q];

    // ---- load the region
    const bool cin = i0 >= 0 && i0 + VX <= P;  // the row pitch is a multiple of 32 words
    const bool own_x = lane * VX >= H && lane * VX < H + w.tw && i0 < nx;
    R e[2][RPW][VX], hz[RPW][VX], jj[2][RPW][VX], ca[2][RPW][VX], cb[2][RPW][VX], bj[2][RPW][VX];
    R pe[2][RPW][VX], ph[2][RPW][VX];  // psi of Ex (y), Ey (x); of Hz along x, along y
    unsigned gapm = 0, srcm = 0, desr = 0, ownr = 0;  // bits: edge (cc RPW + r) VX + v; row r or cc RPW + r
    int d[2][RPW];  // design index of the row's first edge
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int j = j0 + r;
        if (own_x && wi * RPW + r >= H && wi * RPW + r < H + w.th && j < ny) ownr |= 1u << r;
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            zero(ca[cc][r]); zero(cb[cc][r]); zero(bj[cc][r]);
            d[cc][r] = (j - g.d0[cc][1]) * g.dp[cc] + (i0 - g.dxa[cc]);
            if (i0 >= g.dxa[cc] && i0 < g.dxa[cc] + g.dp[cc] && in_range(j, g.d0[cc][1], g.dn[cc][1])) {
                desr |= 1u << (cc * RPW + r);
                const R *q = w.coef[cc] + d[cc][r];
                ldv(q, ca[cc][r]);
                ldv(q + g.Mdi[cc], cb[cc][r]);
                ldv(q + 2 * g.Mdi[cc], bj[cc][r]);
            }
        }
    }
    if (!w.first) pdl_wait();
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int j = j0 + r;
        zero(hz[r]);
#pragma unroll
        for (int cc = 0; cc < 2; ++cc) {
            zero(e[cc][r]); zero(jj[cc][r]); zero(pe[cc][r]); zero(ph[cc][r]);
        }
        if ((unsigned)j < (unsigned)ny && cin) {
            const long long q = (long long)j * P + i0;
            ldv(in.Ex + q, e[0][r]);
            ldv(in.Ey + q, e[1][r]);
            ldv(in.Hz + q, hz[r]);
#pragma unroll
            for (int cc = 0; cc < 2; ++cc)
                if (desr >> (cc * RPW + r) & 1u) ldv(in.J[cc] + d[cc][r], jj[cc][r]);
            if (xp) {
#pragma unroll
                for (int v = 0; v < VX; ++v) {
                    const int i = i0 + v;
                    if (i >= nx) continue;
                    const int se = slab_e(i, nx, np), sh = slab_h(i, nx, np);
                    if (se >= 0) pe[1][r][v] = in.peyx[(long long)j * np2 + se];
                    if (sh >= 0) ph[0][r][v] = in.phzx[(long long)j * np2 + sh];
                }
            }
            if (yp) {
                const int te = slab_e(j, ny, np), th = slab_h(j, ny, np);
                if (te >= 0) ldv(in.pexy + (long long)te * P + i0, pe[0][r]);
                if (th >= 0) ldv(in.phzy + (long long)th * P + i0, ph[1][r]);
            }
        }
    }
    bool yph = false, ype = false;  // warp-uniform: rows in the absorbing layer
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int j = j0 + r;
        if (yp && (unsigned)j < (unsigned)ny) {
            yph |= slab_h(j, ny, np) >= 0;
            ype |= slab_e(j, ny, np) >= 0;
        }
#pragma unroll
        for (int v = 0; v < VX; ++v) {
            const int i = i0 + v;
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
                const bool upd = cc == 0 ? i >= 0 && i <= nx - 2 && j >= 1 && j <= ny - 2
                                         : j >= 0 && j <= ny - 2 && i >= 1 && i <= nx - 2;
                const bool gap = in_range(i, g.g0[cc][0], g.gn[cc][0]) && in_range(j, g.g0[cc][1], g.gn[cc][1]);
                const unsigned bit = 1u << ((cc * RPW + r) * VX + v);
                if (bj[cc][r][v] == R(0)) cb[cc][r][v] = gap ? c.inv_eps_g : c.inv_eps_s;
                if (!upd) cb[cc][r][v] = R(0);
                if (gap) gapm |= bit;
                if (MODE == 0 && cc == 0 && in_range(i, g.s0[0], g.s1[0] - g.s0[0]) &&
                    in_range(j, g.s0[1], g.s1[1] - g.s0[1]))
                    srcm |= bit;
            }
        }
    }
    const bool anysrc = __any_sync(0xffffffffu, (MODE == 0 ? srcm : gapm) != 0);
    const bool anygap = MODE == 0 && w.gap && __any_sync(0xffffffffu, gapm != 0 && ownr != 0);
    // Block-uniform: the region holds design columns (the Ex and Ey boxes
    // share their first row and column; one is a row, the other a column
    // larger).
    const bool dru = xr < g.dxa[0] + max(g.dp[0], g.dp[1]) && xr + W > g.dxa[0] &&
                     yr < g.d0[0][1] + max(g.dn[0][1], g.dn[1][1]) && yr + nw * RPW > g.d0[0][1];
    const R hJ = c.half1pkJ, kJ = c.kJ;
    __syncthreads();  // the staged tables are complete
    R tx[4][VX];  // CPML b, c of this thread's columns (E, then H); 1/kappa stays in shared memory
#pragma unroll
    for (int v = 0; v < VX; ++v)
#pragma unroll
        for (int q = 0; q < 4; ++q) tx[q][v] = xp ? xt[(q < 2 ? q : q + 1) * W + lane * VX + v] : R(0);
    R *rec = w.rec;

    // The step loop, one instance per kind of block (see kernels_rt2d.cu).
    // K1: every CPML kappa is 1 (the usual case), so that 1/kappa is not read.
    auto run = [&](auto xpc, auto ypc, auto drc, auto k1c) {
        constexpr bool XP = decltype(xpc)::value, YP = decltype(ypc)::value, DR = decltype(drc)::value,
                       K1 = decltype(k1c)::value;
#pragma unroll 1
        for (int t = 0; t < T; ++t) {
            // Rows that no own edge depends on any more are left alone.
            const int back = T - t, r0 = wi * RPW;
            const bool need = r0 + RPW - 1 >= H - back && r0 <= H + w.th - 1 + back;
            R *u = sU + wi * W + lane * VX, *dn = sD + (wi + 1) * W + lane * VX;
            stv(u, e[0][0]);
            __syncthreads();
            if (need) {
                R up[VX], dx[RPW][VX], dy[RPW][VX];
                ldv(u + W, up);  // the warp above's first Ex row
#pragma unroll
                for (int r = 0; r < RPW; ++r) {
                    const R er = __shfl_down_sync(0xffffffffu, e[1][r][0], 1);  // Ey of the column to the right
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        dx[r][v] = (v + 1 < VX ? e[1][r][v + 1 < VX ? v + 1 : v] : er) - e[1][r][v];
                        dy[r][v] = (r + 1 < RPW ? e[0][r + 1 < RPW ? r + 1 : 0][v] : up[v]) - e[0][r][v];
                    }
                }
                if (XP) {
#pragma unroll
                    for (int r = 0; r < RPW; ++r)
#pragma unroll
                        for (int v = 0; v < VX; ++v) {
                            const R p = fma(tx[2][v], ph[0][r][v], tx[3][v] * dx[r][v]);
                            ph[0][r][v] = p;
                            dx[r][v] = K1 ? dx[r][v] + p : dx[r][v] * xt[5 * W + lane * VX + v] + p;
                        }
                }
                if (YP && yph) {
#pragma unroll
                    for (int r = 0; r < RPW; ++r) {
                        const int q = wi * RPW + r;
                        const R b = yt[3 * YT + q], c2 = yt[4 * YT + q];
#pragma unroll
                        for (int v = 0; v < VX; ++v) {
                            const R p = fma(b, ph[1][r][v], c2 * dy[r][v]);
                            ph[1][r][v] = p;
                            dy[r][v] = K1 ? dy[r][v] + p : dy[r][v] * yt[5 * YT + q] + p;
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) hz[r][v] = fma(-S, dx[r][v] - dy[r][v], hz[r][v]);
            }
            stv(dn, hz[RPW - 1]);
            __syncthreads();
            if (!need) continue;
            R lo[VX], hl[RPW];
            ldv(dn - W, lo);  // the warp below's last Hz row
#pragma unroll
            for (int r = 0; r < RPW; ++r) hl[r] = __shfl_up_sync(0xffffffffu, hz[r][VX - 1], 1);  // Hz of the column to the left
            // Ex, then Ey: one component at a time, for the registers' sake
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
                R x[RPW][VX], y[RPW][VX];
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v)
                        x[r][v] = hz[r][v] - (cc == 0 ? (r > 0 ? hz[r > 0 ? r - 1 : 0][v] : lo[v])
                                                      : (v > 0 ? hz[r][v > 0 ? v - 1 : 0] : hl[r]));
                if (cc == 1 && XP) {
#pragma unroll
                    for (int r = 0; r < RPW; ++r)
#pragma unroll
                        for (int v = 0; v < VX; ++v) {
                            const R p = fma(tx[0][v], pe[1][r][v], tx[1][v] * x[r][v]);
                            pe[1][r][v] = p;
                            x[r][v] = K1 ? x[r][v] + p : x[r][v] * xt[2 * W + lane * VX + v] + p;
                        }
                }
                if (cc == 0 && YP && ype) {
#pragma unroll
                    for (int r = 0; r < RPW; ++r) {
                        const int q = wi * RPW + r;
                        const R b = yt[q], c2 = yt[YT + q];
#pragma unroll
                        for (int v = 0; v < VX; ++v) {
                            const R p = fma(b, pe[0][r][v], c2 * x[r][v]);
                            pe[0][r][v] = p;
                            x[r][v] = K1 ? x[r][v] + p : x[r][v] * yt[2 * YT + q] + p;
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        x[r][v] = (cc ? -S : S) * x[r][v];
                        if (DR) x[r][v] = fma(-hJ, jj[cc][r][v], x[r][v]);
                    }
                if (anysrc) {
#pragma unroll
                    for (int q = 0; q < RPW * VX; ++q) {
                        const int r = q / VX, v = q % VX, bit = cc * RPW * VX + q;
                        R src = R(0);
                        if (MODE == 0) {
                            if (srcm >> bit & 1u) src = ssrc[t];
                        } else if (gapm >> bit & 1u) {
                            const int gi =
                                (cc ? g.Mgc[0] : 0) + (j0 + r - g.g0[cc][1]) * g.gn[cc][0] + (i0 + v - g.g0[cc][0]);
                            src = -c.eps_g * (gstage ? sgap[(T - 1 - t) * Mg + gi] : w.gap[(long long)(w.n0 - t) * Mg + gi]);
                        }
                        x[r][v] = x[r][v] - src;
                    }
                }
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        const R eo = e[cc][r][v];
                        R en;
                        if (DR) {
                            // a Drude edge: ca E + cb x; any other: E + cb x (its J and bJ are 0)
                            const R m = ca[cc][r][v] * eo;
                            en = fma(cb[cc][r][v], x[r][v], bj[cc][r][v] != R(0) ? m : eo);
                            x[r][v] = fma(kJ, jj[cc][r][v], bj[cc][r][v] * (en + eo));
                        } else {
                            en = fma(x[r][v], cb[cc][r][v], eo);
                        }
                        y[r][v] = en;
                    }
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        e[cc][r][v] = y[r][v];
                        if (DR) jj[cc][r][v] = x[r][v];
                    }
                // records of the block's own edges
                if (DR || anygap) {
#pragma unroll
                    for (int r = 0; r < RPW; ++r)
                        if (ownr >> r & 1u) {
                            if (DR && rec && (desr >> (cc * RPW + r) & 1u))
                                stv(rec + (cc ? g.Mdi[0] : 0) + d[cc][r], e[cc][r]);
                            if (anygap) {
#pragma unroll
                                for (int v = 0; v < VX; ++v)
                                    if (gapm >> ((cc * RPW + r) * VX + v) & 1u)
                                        w.gap[(long long)(w.n0 + t + 1) * Mg + (cc ? g.Mgc[0] : 0) +
                                              (j0 + r - g.g0[cc][1]) * g.gn[cc][0] + (i0 + v - g.g0[cc][0])] = e[cc][r][v];
                            }
                        }
                }
            }
            if (DR && rec) rec += w.rec_step;
        }
    };
    using Yes = std::true_type;
    using No = std::false_type;
    if (!w.kappa1 && (xp || yp)) {
        // the tables of an axis without a layer here are not staged
        if (dru) {
            if (xp && yp) run(Yes{}, Yes{}, Yes{}, No{});
            else if (xp) run(Yes{}, No{}, Yes{}, No{});
            else run(No{}, Yes{}, Yes{}, No{});
        } else {
            if (xp && yp) run(Yes{}, Yes{}, No{}, No{});
            else if (xp) run(Yes{}, No{}, No{}, No{});
            else run(No{}, Yes{}, No{}, No{});
        }
    } else if (dru) {
        if (xp && yp) run(Yes{}, Yes{}, Yes{}, Yes{});
        else if (xp) run(Yes{}, No{}, Yes{}, Yes{});
        else if (yp) run(No{}, Yes{}, Yes{}, Yes{});
        else run(No{}, No{}, Yes{}, Yes{});
    } else {
        if (xp && yp) run(Yes{}, Yes{}, No{}, Yes{});
        else if (xp) run(Yes{}, No{}, No{}, Yes{});
        else if (yp) run(No{}, Yes{}, No{}, Yes{});
        else run(No{}, No{}, No{}, Yes{});
    }

    // ---- store the tile's own nodes into the other buffer of the pair
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        if (!(ownr >> r & 1u)) continue;
        const int j = j0 + r;
        const long long q = (long long)j * P + i0;
        stv(out.Ex + q, e[0][r]);
        stv(out.Ey + q, e[1][r]);
        stv(out.Hz + q, hz[r]);
#pragma unroll
        for (int cc = 0; cc < 2; ++cc)
            if (desr >> (cc * RPW + r) & 1u) stv(out.J[cc] + d[cc][r], jj[cc][r]);
        // (an edge that is not updated keeps its psi)
        if (xp) {
#pragma unroll
            for (int v = 0; v < VX; ++v) {
                const int i = i0 + v;
                if (i >= nx) continue;
                const int se = slab_e(i, nx, np), sh = slab_h(i, nx, np);
                if (se >= 0 && i >= 1 && i <= nx - 2 && j <= ny - 2) out.peyx[(long long)j * np2 + se] = pe[1][r][v];
                if (sh >= 0 && j <= ny - 2) out.phzx[(long long)j * np2 + sh] = ph[0][r][v];
            }
        }
        if (yp) {
            const int te = slab_e(j, ny, np), th = slab_h(j, ny, np);
            if (te >= 0 && j >= 1 && j <= ny - 2) stv(out.pexy + (long long)te * P + i0, pe[0][r]);
            if (th >= 0) stv(out.phzy + (long long)th * P + i0, ph[1][r]);
        }
    }
}

// (Blocks of two warps: with 164 registers a thread three of four fit on an SM,
// and a design box of one to two waves ended with a few blocks alone; 1 % of an
// evaluation of small boxes.)
constexpr int SENS_TPB = 64;

// Sensitivities of `count` adjoint steps of the pitched design edges (both
// components): step t went from adjoint E ae[t - 1] (t = 0: eprev) to ae[t],
// with the forward E fe[-t] of its source time.  jsens is the adjoint J
// before the first step and is advanced; eprev receives the last E.  A thread
// owns 16 bytes of adjacent edges and keeps U steps' loads in flight.
template <typename R>
__global__ void __launch_bounds__(SENS_TPB) k_rt2dp_sens(int slot, long long M0, long long M1, const R *__restrict__ coef0,
                                                    const R *__restrict__ coef1, long long step,
                                                    const R *__restrict__ ae, const R *__restrict__ fe, int count,
                                                    R *j0, R *j1, R *e0, R *e1, double *G0, double *G1, PairScale ps)
{
    constexpr int V = 16 / sizeof(R), U = 8;
    const Coef<R> &c = coef_at<R>(slot);
    // threads past the end work on the last edges and store nothing
    const long long id = min((blockIdx.x * (long long)SENS_TPB + threadIdx.x) * V, M0 + M1 - V);
    const bool inside = (blockIdx.x * (long long)SENS_TPB + threadIdx.x) * V < M0 + M1;
    const bool second = id >= M0;
    const long long q = second ? id - M0 : id, M = second ? M1 : M0;
    const R *coef = (second ? coef1 : coef0) + q;
    R *jp = (second ? j1 : j0) + q, *ep = (second ? e1 : e0) + q;
    double *Gp = (second ? G1 : G0) + q;
    const R kJ = c.kJ, te = c.t_eps;
    R bj[V], a1[V], a2[V], eo[V], jo[V];
    ld16(coef + 2 * M, bj);
    ld16(coef + 3 * M, a1);
    ld16(coef + 4 * M, a2);
    fe += id;
    pdl_wait();
    ae += id;
    ld16(ep, eo);
    ld16(jp, jo);
    double g[V];
    PairSum gp[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        g[v] = 0.0;
        gp[v] = PairSum{};
    }
    for (int t0 = 0; t0 < count; t0 += U) {
        R en[U][V], em[U][V];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int t = min(t0 + k, count - 1);
            ld16(ae + t * step, en[k]);
            ld16(fe - t * step, em[k]);
        }
        bool far = false;
        // en becomes the step's Eq. (25) bracket (steps past the last: zero)
#pragma unroll
        for (int k = 0; k < U; ++k)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const R e1v = en[k][v], jn = fma(kJ, jo[v], bj[v] * (e1v + eo[v]));
                en[k][v] = -te * (e1v - eo[v]) - a1[v] * (e1v + eo[v]) - a2[v] * (jn + jo[v]);
                if (t0 + k < count) {
                    eo[v] = e1v;
                    jo[v] = jn;
                } else {
                    en[k][v] = R(0);
                }
                if constexpr (sizeof(R) == 8) g[v] += em[k][v] * en[k][v];
                else far |= Pair::far(em[k][v], en[k][v] * ps.up);
            }
        if constexpr (sizeof(R) == 4) {
            // a uniform branch: as selects, the FP64 operations would run for
            // every step and bound the kernel
            if (__any_sync(0xffffffffu, far)) {
#pragma unroll
                for (int k = 0; k < U; ++k)
#pragma unroll
                    for (int v = 0; v < V; ++v)
                        if (Pair::far(em[k][v], en[k][v] * ps.up)) {
                            g[v] += (double)em[k][v] * (double)en[k][v];
                            en[k][v] = 0.0f;
                        }
            }
            // (steps past the last add zero)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                Pair q{};
#pragma unroll
                for (int k = 0; k < U; ++k) {
                    q.add(em[k][v], en[k][v] * ps.up);
                    if (k % 4 == 3) gp[v].errors(q);
                }
                gp[v].merge(q);
            }
        }
    }
    if (!inside) return;
    st16(ep, eo);
    st16(jp, jo);
#pragma unroll
    for (int v = 0; v < V; ++v)
        if (bj[v] != R(0)) Gp[v] += g[v] + gp[v].value(ps.down);  // not in the gap or the row padding
}

// The Drude coefficients of one component's pitched design edges, in the
// operations of the step kernels (see k_rt2d_coef).
template <typename R>
__global__ void k_rt2dp_coef(const __grid_constant__ GeoP g, int cc, int slot, const R *rho_t, R *coef)
{
    const Coef<R> &c = coef_at<R>(slot);
    const long long M = g.Mdi[cc];
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < M; q += (long long)gridDim.x * blockDim.x) {
        const int i = g.dxa[cc] + (int)(q % g.dp[cc]), j = g.d0[cc][1] + (int)(q / g.dp[cc]);
        const bool gap = in_range(i, g.g0[cc][0], g.gn[cc][0]) && in_range(j, g.g0[cc][1], g.gn[cc][1]);
        R ca = R(0), cb = R(0), bJ = R(0), a1 = R(0), a2 = R(0);
        if (in_range(i, g.d0[cc][0], g.dn[cc][0]) && !gap) {
            const R rt = rho_t[q];
            const R eps = c.eps_s + rt * c.d_eps;
            const R psi = c.psi_s + rt * (c.psi - c.psi_s);
            const R sig = c.sig_max * rt * (R(1) - rt);
            bJ = R(0.5) * psi * c.inv1g;
            const R hs = R(0.5) * (sig + bJ);
            cb = rcp(eps + hs);
            ca = (eps - hs) * cb;
            a1 = c.t_sig * (R(1) - R(2) * rt) * R(0.5);
            a2 = c.t_dpsi * rcp(psi) * R(0.5);
        }
        coef[q] = ca;
        coef[M + q] = cb;
        coef[2 * M + q] = bJ;
        coef[3 * M + q] = a1;
        coef[4 * M + q] = a2;
    }
}

}  // namespace

// A launch's fixed part is about 3 us; a row step is 0.04 us in FP32 (two
// columns per lane) and 0.4 us in FP64.
template <typename R>
Rt2DPlan rt2dp_plan(int nx, int ny, int sms)
{
    using D = Shape<R>;
    constexpr bool F64 = sizeof(R) == 8;
    return rt_tile_plan(nx, ny, sms, D::W, D::RPW, D::MAXW, F64 ? 4 : RT2D_MAX, F64 ? 8.0 : 80.0);
}

template <typename R>
bool rt2dp_ready()
{
    int dev = 0, smem = 0;
    const size_t b = smem_words<R>(Shape<R>::MAXW, sizeof(R) == 4 ? RT2D_MAX : 4, GAP_STAGED) * sizeof(R);
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        b > (size_t)smem ||
        cudaFuncSetAttribute(k_rt2dp<R, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b) != cudaSuccess ||
        cudaFuncSetAttribute(k_rt2dp<R, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

template <typename R>
int launch_rt2dp(int mode, const GeoP &g, const StateP<R> &in, const StateP<R> &out, int slot, const PmlP<R> &pm,
                 const RtP<R> &w, const Rt2DPlan &p, cudaStream_t st)
{
    const int Mg = g.Mgc[0] + g.Mgc[1];
    const size_t smem = smem_words<R>(p.nw, w.count, mode == 1 && Mg <= GAP_STAGED ? Mg : 0) * sizeof(R);
    const dim3 block(32, p.nw), grid(p.bx, p.by);
    launch_pdl_smem(mode == 0 ? k_rt2dp<R, 0> : k_rt2dp<R, 1>, grid, block, smem, st, g, in, out, slot, pm, w);
    return 1;
}

template <typename R>
int launch_rt2dp_coef(const GeoP &g, int slot, const R *const rho_t[2], R *const coef[2], cudaStream_t st)
{
    for (int cc = 0; cc < 2; ++cc) {
        const long long nb = std::max<long long>(1, std::min<long long>((g.Mdi[cc] + 255) / 256, 152 * 8));
        k_rt2dp_coef<R><<<(int)nb, 256, 0, st>>>(g, cc, slot, rho_t[cc], coef[cc]);
    }
    return 2;
}

template <typename R>
int launch_rt2dp_sens(const GeoP &g, int slot, const R *const coef[2], long long step, const R *ae, const R *fe, int count,
                      R *const jsens[2], R *const eprev[2], double *const G[2], PairScale ps, cudaStream_t st)
{
    constexpr int V = 16 / sizeof(R);
    const long long n = g.Mdi[0] + g.Mdi[1];
    launch_pdl(k_rt2dp_sens<R>, dim3((unsigned)((n + SENS_TPB * V - 1) / (SENS_TPB * V))), dim3(SENS_TPB), st, slot, (long long)g.Mdi[0],
               (long long)g.Mdi[1], coef[0], coef[1], step, ae, fe, count, jsens[0], jsens[1], eprev[0], eprev[1], G[0], G[1],
               ps);
    return 1;
}

template <typename R>
cudaError_t upload_coef_rt2dp(int slot, const Coef<R> &c, cudaStream_t st)
{
    return write_coef_slot(slot, c, st);
}

#define RT2DP_INST(R)                                                                                              \
    template Rt2DPlan rt2dp_plan<R>(int, int, int);                                                                \
    template bool rt2dp_ready<R>();                                                                                \
    template int launch_rt2dp<R>(int, const GeoP &, const StateP<R> &, const StateP<R> &, int, const PmlP<R> &,    \
                                 const RtP<R> &, const Rt2DPlan &, cudaStream_t);                                  \
    template int launch_rt2dp_sens<R>(const GeoP &, int, const R *const[2], long long, const R *, const R *, int,  \
                                      R *const[2], R *const[2], double *const[2], PairScale, cudaStream_t);                   \
    template int launch_rt2dp_coef<R>(const GeoP &, int, const R *const[2], R *const[2], cudaStream_t);            \
    template cudaError_t upload_coef_rt2dp<R>(int, const Coef<R> &, cudaStream_t);
RT2DP_INST(float)
RT2DP_INST(double)

}  // namespace fdtd
