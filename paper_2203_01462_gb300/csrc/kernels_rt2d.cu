// Temporally blocked 2D TM_z leapfrog (Ez, Hx, Hy, Jz + CPML) with the tile
// held in registers, for sm_103a.
//
// One launch advances up to `halo` steps.  A block owns a tile of tw x th
// nodes and holds it with a halo of `halo` nodes on every side: a warp spans
// the region's whole width (32 lanes of VX adjacent columns) and RPW adjacent
// rows, so every node's Ez, Hx, Hy, J and Drude coefficients stay in one
// thread's registers for the whole launch.  Neighbours along x come by warp
// shuffle.  Along y a warp needs one row of Ez from the warp above and one
// from the warp below: those two rows per warp and step go through shared
// memory (double buffered), with ONE block barrier per step.  The Hx row
// below the warp's first row, which its E update needs, is advanced by the
// warp itself (a redundant copy of the warp below's last Hx row, same inputs
// and arithmetic, so the same bits): that saves the second barrier.
//
// Measured (GB300, us per forward / adjoint step, full history): 316^2 FP32
// 1.02 / 1.28 (2.89 / 3.59 for the shared-memory tiles this replaces, 6.9 /
// 7.5 with one launch per step); 160^2 FP64 3.3 / 3.3 (12.1 / 15.1).  A 316^2
// launch of 8 steps costs about 3.2 us for its start, loads and stores and
// 0.6 us a step, bound by the latency of the step's chain at four warps per
// scheduler; in FP64 the FP64 pipe is 62 % busy, its two units per SM being
// the bound (a step's 13 needed rows x 15 operations x 16 cycles).
//
// Each half step spoils one layer of the region from the outside (what lies
// beyond is not there), so after `halo` steps the tile itself is still exact
// and no block waits for another; it writes its tile into the other buffer of
// the ping-pong pair.  Nodes outside the grid, on walls and past the last
// node load as zeros and carry zero update factors, so the step loop has no
// per-node tests: a node is updated as
//   E <- J ? ca E + cb (curl - h J - src) : E + cb (curl - src)
// with cb = 1/eps, or 0 where E is not updated.  The CPML terms (psi in
// registers, tables in shared memory) run only in blocks whose region meets
// the layer, the rows' part only in its warps.
//
// The Drude coefficients of rho~ are worked out once per pass (k_rt2d_coef):
// they cost a reciprocal per node (two in the adjoint), which a GB300's FP64
// units, two per SM, would feel on every launch.  Records, the gap's adjoint
// source, the forward source and the adjoint's forward fields of all steps of
// the launch are staged before the step loop, so no global load waits in it.
#include <algorithm>
#include <type_traits>

#include "coef_slots.cuh"
#include "rt_common.cuh"

namespace fdtd {

namespace {

// Shape per precision: VX columns per lane, RPW rows per warp.
template <typename R>
struct Shape {
    static constexpr int VX = sizeof(R) == 4 ? 2 : 1;
    static constexpr int RPW = sizeof(R) == 4 ? 2 : 1;
    static constexpr int W = 32 * VX;   // region width
    static constexpr int MAXW = sizeof(R) == 4 ? 16 : 24;  // warps per block (FP32: 128 registers a thread; the adjoint spills 88 to 128 B)
};

// Shared memory of one block (in words of R unless noted), in this order:
// Ez rows to the warp below / above [2][nw + 1][W] each, CPML tables of the
// columns [6][W] and of the rows [6][nw RPW + 1], source samples [RT2D_MAX],
// the gap's adjoint source [count][Mg] (if it fits), records [count][RPW]
// [threads][VX] (adjoint).
template <typename R>
__host__ __device__ size_t smem_words(int nw, int count, int gapw, int mode)
{
    using D = Shape<R>;
    return (size_t)4 * (nw + 1) * D::W + 6 * D::W + 6 * ((size_t)nw * D::RPW + 2) + RT2D_MAX +
           (((size_t)count * gapw + 1) & ~(size_t)1) + (mode ? (size_t)count * D::RPW * nw * D::W : 0);
}

// Largest gap whose adjoint source is staged in shared memory (nodes).
constexpr int GAP_STAGED = 256;

// FORM: which product of a Drude node's E update is rounded before the sum,
// ca E (1) or cb (curl - ...) (0).  Grids small enough for one 32 x 32 tile
// per SM, and runs with the steps per launch set by the caller, have always
// used 0, all others 1; both are kept, so that a design's results do not
// change with the kernel that computes them.
// NB: blocks per SM the registers have to leave room for; 0: one, and only
// the general kind of region (see launch_rt2d).
// FULL (FP32 adjoint): a launch's sums go into the FP64 accumulator with all
// they hold, or rounded to 2^-49, which saves one of three conversions to FP64
// per node and launch.  Against the exact sums (rt_common.cuh; ten grids, rms)
// the rounded ones are as far off as FP64 sums are, 0.6 to 1.1 times, with up
// to 6 steps a launch, and 0.7 to 1.15 times with 8: there FULL is 0.4 to 0.65
// times.  us per evaluation, not FULL / FULL: 316^2 (8 steps) 9106 / 9207, 530 x 303
// (4 steps) 4910 / 5077.
template <typename R, int MODE, int FORM, int NB, bool FULL>
__global__ void __launch_bounds__(32 * Shape<R>::MAXW, NB > 0 ? NB : 1)
    k_rt2d(const __grid_constant__ Geo2D g, const __grid_constant__ State2D<R> in,
           const __grid_constant__ State2D<R> out, int slot, const __grid_constant__ Pml1D<R> px,
           const __grid_constant__ Pml1D<R> py, const __grid_constant__ Rt2D<R> w)
{
    using D = Shape<R>;
    constexpr int VX = D::VX, RPW = D::RPW, W = D::W;
    constexpr bool F64 = sizeof(R) == 8;
    extern __shared__ __align__(16) char smem_raw[];
    const Coef<R> &c = coef_at<R>(slot);
    const int lane = threadIdx.x, wi = threadIdx.y, nw = blockDim.y, tid = wi * 32 + lane, nth = nw * 32;
    const int T = w.count, H = w.halo, nx = g.nx, ny = g.ny, np = g.npml, P = g.px, np2 = 2 * np;
    const int Mg = g.gnx * g.gny;
    const R S = c.S;

    const int xr = blockIdx.x * w.tw - H, yr = blockIdx.y * w.th - H;  // region origin (grid)
    const int i0 = xr + lane * VX, j0 = yr + wi * RPW;                 // this thread's first node
    R *sU = (R *)smem_raw;                 // [2][nw + 1][W]: a warp's first Ez row, read by the warp below
    R *sD = sU + 2 * (nw + 1) * W;         // [2][nw + 1][W]: a warp's last Ez row (FP64: last Hx row), read by the warp above
    R *xt = sD + 2 * (nw + 1) * W;         // [6][W]: bE cE kiE bH cH kiH of the columns
    const int YT = nw * RPW + 2;
    R *yt = xt + 6 * W;                    // [6][YT]: the same of the rows, entry 0 = the row below the region
    R *ssrc = yt + 6 * YT;
    R *sgap = ssrc + RT2D_MAX;
    // the gap's adjoint source is staged by the blocks whose region holds gap nodes
    const bool gstage = MODE == 1 && Mg <= GAP_STAGED && w.gap && xr < g.gx0 + g.gnx && xr + W > g.gx0 &&
                        yr < g.gy0 + g.gny && yr + nw * RPW > g.gy0;
    R *srec = sgap + (gstage ? ((T * Mg + 1) & ~1) : 0);  // [T][RPW][threads][VX], 8-byte aligned

    // The region meets the absorbing layer of the columns / rows.
    const bool xp = np > 0 && (xr < np || xr + W > nx - 1 - np);
    const bool yp = np > 0 && (yr - 1 < np || yr + nw * RPW > ny - 1 - np);

    // What the previous launch of the same run does not write is read before
    // waiting for it: tables, samples, coefficients, the adjoint's records.
    // The first launch of a run waits for the kernels before it, and only
    // then lets the next one start, so that these reads see their results.
    if (w.first) pdl_wait();
    pdl_trigger();
    if (xp)
        for (int q = tid; q < W; q += nth) {
            const int p = xr + q;
            const bool es = (unsigned)p < (unsigned)nx && slab_e(p, nx, np) >= 0;
            const bool hs = (unsigned)p < (unsigned)nx && slab_h(p, nx, np) >= 0;
            xt[q] = es ? px.bE[p] : R(0);
            xt[W + q] = es ? px.cE[p] : R(0);
            xt[2 * W + q] = es ? px.kiE[p] : R(1);
            xt[3 * W + q] = hs ? px.bH[p] : R(0);
            xt[4 * W + q] = hs ? px.cH[p] : R(0);
            xt[5 * W + q] = hs ? px.kiH[p] : R(1);
        }
    if (yp)
        for (int q = tid; q < nw * RPW + 1; q += nth) {
            const int p = yr - 1 + q;
            const bool es = (unsigned)p < (unsigned)ny && slab_e(p, ny, np) >= 0;
            const bool hs = (unsigned)p < (unsigned)ny && slab_h(p, ny, np) >= 0;
            yt[q] = es ? py.bE[p] : R(0);
            yt[YT + q] = es ? py.cE[p] : R(0);
            yt[2 * YT + q] = es ? py.kiE[p] : R(1);
            yt[3 * YT + q] = hs ? py.bH[p] : R(0);
            yt[4 * YT + q] = hs ? py.cH[p] : R(0);
            yt[5 * YT + q] = hs ? py.kiH[p] : R(1);
        }
    if (MODE == 0 && tid < T) ssrc[tid] = w.src[w.n0 + tid];
    if (gstage)  // rows n0 - T + 1 .. n0 are consecutive
        for (int q = tid; q < T * Mg; q += nth) sgap[q] = w.gap[(long long)(w.n0 - T + 1) * Mg + q];

    // Everything from the loads to the stores, one instance per kind of
    // region.  V: every node is a plain one of the background; D: of the
    // design box; both clear of walls, absorbing layer, gap and source.  On
    // large grids nearly all regions are, and the tests for anything else were
    // 600 of a launch's 1080 instructions per warp: 2048^2 22.5 -> 17.8 us per
    // forward step, 27 -> 23.5 per adjoint step, 1000^2 5.9 -> 4.9.  (Copying
    // the next tile's state into shared memory while one is stepped, in
    // persistent blocks, gained nothing on top: 18.5; a second block per SM
    // did: 13.2, see launch_rt2d.)
    auto body = [&](auto vc, auto dc) {
    constexpr bool V = decltype(vc)::value, D = decltype(dc)::value, PL = V || D;
    // ---- load the region
    const bool cin = PL || (i0 >= 0 && i0 + VX <= P);  // the row pitch is a multiple of 32 words
    const bool vdx = i0 >= g.dxa && i0 < g.dxa + g.dp;  // and the design box's columns start on a multiple of 4
    const bool own_x = lane * VX >= H && lane * VX < H + w.tw && i0 < nx;
    R ez[RPW][VX], hx[RPW][VX], hy[RPW][VX], jj[RPW][VX], ca[RPW][VX], cb[RPW][VX], bj[RPW][VX], hxd[VX];
    R a1[RPW][VX], a2[RPW][VX];
    double G[RPW][VX];
    Pair gp[RPW][VX];
    R pex[RPW][VX], phx[RPW][VX], pey[RPW][VX], phy[RPW][VX], phd[VX];  // psi of Ez, Hy (x) and Ez, Hx (y)
    unsigned gapm = 0, srcm = 0, desr = 0, ownr = 0;  // gap / source node bits; rows with design columns / own nodes
    long long d[RPW];  // design index of the row's first node
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int j = j0 + r;
        zero(ca[r]); zero(cb[r]); zero(bj[r]); zero(a1[r]); zero(a2[r]);
        if (own_x && wi * RPW + r >= H && wi * RPW + r < H + w.th && j < ny) ownr |= 1u << r;
        d[r] = (long long)(j - g.dy0) * g.dp + (i0 - g.dxa);
        if (D || (!V && vdx && in_range(j, g.dy0, g.dny))) {
            desr |= 1u << r;
            ldv(w.coef + d[r], ca[r]);
            ldv(w.coef + w.Mdi + d[r], cb[r]);
            ldv(w.coef + 2 * w.Mdi + d[r], bj[r]);
            if (MODE == 1) {
                ldv(w.coef + 3 * w.Mdi + d[r], a1[r]);
                ldv(w.coef + 4 * w.Mdi + d[r], a2[r]);
                if (ownr >> r & 1u)
                    for (int t = 0; t < T; ++t)
                        cp8(srec + ((size_t)(t * RPW + r) * nth + tid) * VX,
                            w.rec + (long long)(w.n0 - t - 1 - w.rec0) * w.Mdi + d[r]);
            }
        }
    }
    if (!w.first) pdl_wait();
    zero(hxd);
    zero(phd);
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int j = j0 + r;
        zero(ez[r]); zero(hx[r]); zero(hy[r]); zero(jj[r]);
        zero(pex[r]); zero(phx[r]); zero(pey[r]); zero(phy[r]);
#pragma unroll
        for (int v = 0; v < VX; ++v) {
            G[r][v] = 0.0;
            gp[r][v] = Pair{};
        }
        if (PL || ((unsigned)j < (unsigned)ny && cin)) {
            const long long q = (long long)j * P + i0;
            ldv(in.Ez + q, ez[r]);
            ldv(in.Hx + q, hx[r]);
            ldv(in.Hy + q, hy[r]);
            if (r == 0 && (PL || j >= 1) && !F64) ldv(in.Hx + q - P, hxd);
            if (D || desr >> r & 1u) {
                ldv(in.J + d[r], jj[r]);
                if (MODE == 1 && F64 && (ownr >> r & 1u))
#pragma unroll
                    for (int v = 0; v < VX; ++v) G[r][v] = w.G[d[r] + v];
            }
            if (!PL && xp) {
#pragma unroll
                for (int v = 0; v < VX; ++v) {
                    const int i = i0 + v;
                    if (i >= nx) continue;
                    const int se = slab_e(i, nx, np), sh = slab_h(i, nx, np);
                    if (se >= 0) pex[r][v] = in.pezx[(long long)j * np2 + se];
                    if (sh >= 0) phx[r][v] = in.phyx[(long long)j * np2 + sh];
                }
            }
            if (!PL && yp) {
                const int te = slab_e(j, ny, np), th = slab_h(j, ny, np);
                if (te >= 0) ldv(in.pezy + (long long)te * P + i0, pey[r]);
                if (th >= 0) ldv(in.phxy + (long long)th * P + i0, phy[r]);
                if (r == 0 && j >= 1 && !F64) {
                    const int td = slab_h(j - 1, ny, np);
                    if (td >= 0) ldv(in.phxy + (long long)td * P + i0, phd);
                }
            }
        }
    }
    // Update factors: cb of the nodes that are not Drude nodes, S of the H
    // components whose half-step neighbour exists.
    R Sx[VX], Sy[RPW];
#pragma unroll
    for (int v = 0; v < VX; ++v) Sx[v] = PL || (i0 + v >= 0 && i0 + v + 1 < nx) ? S : R(0);
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int j = j0 + r;
        Sy[r] = PL || (j >= 0 && j + 1 < ny) ? S : R(0);
#pragma unroll
        for (int v = 0; v < VX; ++v) {
            const int i = i0 + v;
            const bool upd = PL || (i >= 1 && i <= nx - 2 && j >= 1 && j <= ny - 2);
            const bool gap = !PL && in_range(i, g.gx0, g.gnx) && in_range(j, g.gy0, g.gny);
            if (bj[r][v] == R(0)) cb[r][v] = gap ? c.inv_eps_g : c.inv_eps_s;
            if (!upd) cb[r][v] = R(0);
            if (gap) gapm |= 1u << (r * VX + v);
            if (!PL && MODE == 0 && in_range(i, g.sx0, g.sx1 - g.sx0) && in_range(j, g.sy0, g.sy1 - g.sy0))
                srcm |= 1u << (r * VX + v);
        }
    }
    const R Syd = PL || (j0 - 1 >= 0 && j0 < ny) ? S : R(0);
    // FORM 1: nodes of the step kernel's plain vector tiles take its S / eps
    // as one factor of the unscaled curl (different bits in the denormal
    // range only, but rounding noise there outlives the front it starts in).
    R Sc = S;
    if (FORM == 1 && !D) {
        const int tx0 = i0 & ~(STEP2D_TX - 1), ty0 = j0 & ~(STEP2D_TY - 1);
        if ((PL || (i0 >= 0 && j0 >= 0)) && step2d_vector_tile(nx, ny, np, tx0, ty0) && !step2d_touches(g, MODE, tx0, ty0)) {
            Sc = R(1);
#pragma unroll
            for (int r = 0; r < RPW; ++r)
#pragma unroll
                for (int v = 0; v < VX; ++v) cb[r][v] = S * cb[r][v];
        }
    }
    // Warp-uniform facts: this warp's rows (the one below included, for H)
    // lie in the rows' absorbing layer; it holds nodes with a source term,
    // own gap nodes to record.
    bool yph = false, ype = false;
    if (!PL && yp) {
#pragma unroll
        for (int r = -1; r < RPW; ++r) {
            const int j = j0 + r;
            if ((unsigned)j < (unsigned)ny) {
                yph |= slab_h(j, ny, np) >= 0;
                if (r >= 0) ype |= slab_e(j, ny, np) >= 0;
            }
        }
    }
    const bool anysrc = !PL && __any_sync(0xffffffffu, (MODE == 0 ? srcm : gapm) != 0);
    const bool anygap = !PL && MODE == 0 && w.gap && __any_sync(0xffffffffu, gapm != 0 && ownr != 0);
    // Block-uniform: the region holds design columns.
    const bool dru = xr < g.dxa + g.dp && xr + W > g.dxa && yr < g.dy0 + g.dny && yr + nw * RPW > g.dy0;
    // Warp-uniform: it holds own rows; own Drude nodes (node bits).
    const bool ownw = wi * RPW + RPW > H && wi * RPW < H + w.th;
    unsigned sens = 0;
#pragma unroll
    for (int r = 0; r < RPW; ++r)
#pragma unroll
        for (int v = 0; v < VX; ++v)
            if ((ownr & desr) >> r & 1u && bj[r][v] != R(0)) sens |= 1u << (r * VX + v);
    const R hJ = c.half1pkJ, kJ = c.kJ;
    if (MODE == 1) {
        asm volatile("cp.async.wait_all;" ::: "memory");  // each thread reads only its own records
        if (ownw && sens != (1u << RPW * VX) - 1u)  // nodes that take no part count as zero
            for (int t = 0; t < T; ++t)
#pragma unroll
                for (int q = 0; q < RPW * VX; ++q)
                    if (!(sens >> q & 1u)) srec[((size_t)(t * RPW + q / VX) * nth + tid) * VX + q % VX] = R(0);
    }
    __syncthreads();  // the staged tables are complete
    R tx[4][VX];  // CPML b, c of this thread's columns (E, then H); 1/kappa stays in shared memory
#pragma unroll
    for (int v = 0; v < VX; ++v) {
        tx[0][v] = !PL && xp ? xt[lane * VX + v] : R(0);
        tx[1][v] = !PL && xp ? xt[W + lane * VX + v] : R(0);
        tx[2][v] = !PL && xp ? xt[3 * W + lane * VX + v] : R(0);
        tx[3][v] = !PL && xp ? xt[4 * W + lane * VX + v] : R(0);
    }
    const bool k1 = w.kappa1 != 0;
    R *rec = nullptr;
    if (MODE == 0 && w.rec) rec = w.rec + (long long)(w.n0 - w.rec0) * w.Mdi;
    R *srp = srec + (size_t)tid * VX;  // this thread's record of row 0, step 0

    // The step loop, one instance per kind of block (XP / YP: its region
    // meets the columns' / rows' absorbing layer, DR: the design box), so
    // that no test breaks up the updates of a thread's nodes: with four warps
    // per scheduler their independent chains are what hides the latency.
    auto run = [&](auto xpc, auto ypc, auto drc) {
        constexpr bool XP = decltype(xpc)::value, YP = decltype(ypc)::value, DR = decltype(drc)::value;
#pragma unroll 1
        for (int t = 0; t < T; ++t) {
            // Rows that no own node depends on any more are left alone: after
            // step t only those within T - 1 - t of the tile matter (their H
            // up to one row further, which `need` includes).
            const int back = T - t, r0 = wi * RPW;
            const bool need = r0 + RPW - 1 >= H - back && r0 <= H + w.th - 1 + back;
            R *u = sU + ((t & 1) * (nw + 1) + wi) * W + lane * VX, *dn = sD + ((t & 1) * (nw + 1) + wi + 1) * W + lane * VX;
            // ---- exchange the warp's first and last Ez rows (FP64: the first)
            stv(u, ez[0]);
            if (!F64) stv(dn, ez[RPW - 1]);
            if (need) {
                // ---- Hy (no row exchange needed)
                R dd[RPW][VX];
#pragma unroll
                for (int r = 0; r < RPW; ++r) {
                    const R ezr = __shfl_down_sync(0xffffffffu, ez[r][0], 1);  // Ez of the column to the right
#pragma unroll
                    for (int v = 0; v < VX; ++v)
                        dd[r][v] = (v + 1 < VX ? ez[r][v + 1 < VX ? v + 1 : v] : ezr) - ez[r][v];
                }
                if (XP) {
#pragma unroll
                    for (int r = 0; r < RPW; ++r)
#pragma unroll
                        for (int v = 0; v < VX; ++v) {
                            const R p = fma(tx[2][v], phx[r][v], tx[3][v] * dd[r][v]);
                            phx[r][v] = p;
                            dd[r][v] = k1 ? dd[r][v] + p : fma(dd[r][v], xt[5 * W + lane * VX + v], p);
                        }
                }
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) hy[r][v] = fma(Sx[v], dd[r][v], hy[r][v]);
            }
            __syncthreads();
            constexpr int RL = F64 ? 0 : -1;  // FP32 also advances the Hx row below the warp
            if (need) {
                R up[VX], lo[VX];
                ldv(u + W, up);             // the warp above's first Ez row
                if (!F64) ldv(dn - W, lo);  // the warp below's last Ez row
                R dd[RPW + 1][VX];
#pragma unroll
                for (int r = RL; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v)
                        dd[r + 1][v] = (r + 1 < RPW ? ez[r + 1 < RPW ? r + 1 : 0][v] : up[v]) -
                                       (r < 0 ? lo[v] : ez[r < 0 ? 0 : r][v]);
                if (YP && yph) {
#pragma unroll
                    for (int r = RL; r < RPW; ++r) {
                        const int q = wi * RPW + r + 1;
                        const R b = yt[3 * YT + q], cc = yt[4 * YT + q];
#pragma unroll
                        for (int v = 0; v < VX; ++v) {
                            R &ps = r < 0 ? phd[v] : phy[r < 0 ? 0 : r][v];
                            ps = fma(b, ps, cc * dd[r + 1][v]);
                            dd[r + 1][v] = k1 ? dd[r + 1][v] + ps : fma(dd[r + 1][v], yt[5 * YT + q], ps);
                        }
                    }
                }
#pragma unroll
                for (int r = RL; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        R &h = r < 0 ? hxd[v] : hx[r < 0 ? 0 : r][v];
                        h = fma(-(r < 0 ? Syd : Sy[r < 0 ? 0 : r]), dd[r + 1][v], h);
                    }
            }
            if (F64) {
                // FP64 units are the bound: hand the last Hx row up instead of advancing it twice
                stv(dn, hx[RPW - 1]);
                __syncthreads();
                ldv(dn - W, hxd);
            }
            if (!need) continue;
            // ---- E, J
            R x[RPW][VX], y[RPW][VX];
#pragma unroll
            for (int r = 0; r < RPW; ++r) {
                const R hyl = __shfl_up_sync(0xffffffffu, hy[r][VX - 1], 1);  // Hy of the column to the left
#pragma unroll
                for (int v = 0; v < VX; ++v) {
                    x[r][v] = hy[r][v] - (v > 0 ? hy[r][v > 0 ? v - 1 : 0] : hyl);
                    y[r][v] = hx[r][v] - (r > 0 ? hx[r > 0 ? r - 1 : 0][v] : hxd[v]);
                }
            }
            if (XP) {
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        const R p = fma(tx[0][v], pex[r][v], tx[1][v] * x[r][v]);
                        pex[r][v] = p;
                        x[r][v] = k1 ? x[r][v] + p : fma(x[r][v], xt[2 * W + lane * VX + v], p);
                    }
            }
            if (YP && ype) {
#pragma unroll
                for (int r = 0; r < RPW; ++r) {
                    const int q = wi * RPW + r + 1;
                    const R b = yt[q], cc = yt[YT + q];
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        const R p = fma(b, pey[r][v], cc * y[r][v]);
                        pey[r][v] = p;
                        y[r][v] = k1 ? y[r][v] + p : fma(y[r][v], yt[2 * YT + q], p);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < RPW; ++r)
#pragma unroll
                for (int v = 0; v < VX; ++v) {
                    x[r][v] = Sc * (x[r][v] - y[r][v]);
                    if (DR) x[r][v] = fma(-hJ, jj[r][v], x[r][v]);
                }
            if (anysrc) {
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        R src = R(0);
                        if (MODE == 0) {
                            if (srcm >> (r * VX + v) & 1u) src = ssrc[t];
                        } else if (gapm >> (r * VX + v) & 1u) {
                            const int gi = (j0 + r - g.gy0) * g.gnx + (i0 + v - g.gx0);
                            src = -c.eps_g * (gstage ? sgap[(T - 1 - t) * Mg + gi] : w.gap[(long long)(w.n0 - t) * Mg + gi]);
                        }
                        x[r][v] = x[r][v] - src;
                    }
            }
#pragma unroll
            for (int r = 0; r < RPW; ++r)
#pragma unroll
                for (int v = 0; v < VX; ++v) {
                    const R eo = ez[r][v];
                    R en;
                    if (DR) {
                        // a Drude node: ca E + cb x; any other: E + cb x (its J and bJ are 0)
                        const R jo = jj[r][v];
                        const bool nd = bj[r][v] != R(0);
                        if (FORM == 1) {
                            const R m = ca[r][v] * eo;
                            en = fma(cb[r][v], x[r][v], nd ? m : eo);
                        } else {
                            const R m = cb[r][v] * x[r][v];
                            const R ed = fma(ca[r][v], eo, m), ev = fma(x[r][v], cb[r][v], eo);
                            en = nd ? ed : ev;
                        }
                        x[r][v] = fma(kJ, jo, bj[r][v] * (en + eo));
                    } else {
                        en = fma(x[r][v], cb[r][v], eo);
                    }
                    y[r][v] = en;
                }
            if (MODE == 1 && DR && ownw) {
                R term[RPW][VX], em[RPW][VX];
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) {
                        const R en = y[r][v], eo = ez[r][v];
                        term[r][v] = -c.t_eps * (en - eo) - a1[r][v] * (en + eo) - a2[r][v] * (x[r][v] + jj[r][v]);
                        em[r][v] = srp[(size_t)(t * RPW + r) * nth * VX + v];
                    }
                if constexpr (F64) {
#pragma unroll
                    for (int r = 0; r < RPW; ++r)
#pragma unroll
                        for (int v = 0; v < VX; ++v) G[r][v] += em[r][v] * term[r][v];
                } else {
                    // products whose rounding error FP32 cannot hold go to
                    // FP64 directly
                    bool far = false;
#pragma unroll
                    for (int r = 0; r < RPW; ++r)
#pragma unroll
                        for (int v = 0; v < VX; ++v) far |= Pair::far(em[r][v], term[r][v] * w.ps.up);
                    if (__any_sync(0xffffffffu, far)) {
#pragma unroll
                        for (int r = 0; r < RPW; ++r)
#pragma unroll
                            for (int v = 0; v < VX; ++v)
                                if (Pair::far(em[r][v], term[r][v] * w.ps.up)) {
                                    if (sens >> (r * VX + v) & 1u)
                                        w.G[d[r] + v] += (double)em[r][v] * (double)term[r][v];
                                    term[r][v] = R(0);
                                }
                    }
#pragma unroll
                    for (int r = 0; r < RPW; ++r)
#pragma unroll
                        for (int v = 0; v < VX; ++v) {
                            // (two blocks per SM: no registers for the products'
                            // errors, which take the place of the step's record)
                            if constexpr (NB == 2)
                                srp[(size_t)(t * RPW + r) * nth * VX + v] = gp[r][v].add_rounded(em[r][v], term[r][v] * w.ps.up);
                            else gp[r][v].add(em[r][v], term[r][v] * w.ps.up);
                        }
                }
            }
#pragma unroll
            for (int r = 0; r < RPW; ++r)
#pragma unroll
                for (int v = 0; v < VX; ++v) {
                    ez[r][v] = y[r][v];
                    if (DR) jj[r][v] = x[r][v];
                }
            // records of the block's own nodes
            if (MODE == 0 && (DR || anygap)) {
#pragma unroll
                for (int r = 0; r < RPW; ++r)
                    if (ownr >> r & 1u) {
                        if (DR && rec && (desr >> r & 1u)) stv(rec + d[r], ez[r]);
                        if (anygap) {
#pragma unroll
                            for (int v = 0; v < VX; ++v)
                                if (gapm >> (r * VX + v) & 1u)
                                    w.gap[(long long)(w.n0 + t + 1) * Mg + (j0 + r - g.gy0) * g.gnx + (i0 + v - g.gx0)] =
                                        ez[r][v];
                        }
                    }
                if (DR && rec) rec += w.Mdi;
            }
        }
    };
    using Yes = std::true_type;
    using No = std::false_type;
    if constexpr (PL) {
        run(No{}, No{}, std::bool_constant<D>{});
    } else if (dru) {
        if (xp && yp) run(Yes{}, Yes{}, Yes{});
        else if (xp) run(Yes{}, No{}, Yes{});
        else if (yp) run(No{}, Yes{}, Yes{});
        else run(No{}, No{}, Yes{});
    } else {
        if (xp && yp) run(Yes{}, Yes{}, No{});
        else if (xp) run(Yes{}, No{}, No{});
        else if (yp) run(No{}, Yes{}, No{});
        else run(No{}, No{}, No{});
    }

    if constexpr (MODE == 1 && NB == 2 && !V) {
        if (ownw && (D || dru))
            for (int t = 0; t < T; ++t)
#pragma unroll
                for (int r = 0; r < RPW; ++r)
#pragma unroll
                    for (int v = 0; v < VX; ++v) gp[r][v].c += srp[(size_t)(t * RPW + r) * nth * VX + v];
    }
    // ---- store the tile's own nodes into the other buffer of the pair
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        if (!(ownr >> r & 1u)) continue;
        const int j = j0 + r;
        const long long q = (long long)j * P + i0;
        stv(out.Ez + q, ez[r]);
        stv(out.Hx + q, hx[r]);
        stv(out.Hy + q, hy[r]);
        if (D || (!V && desr >> r & 1u)) {
            stv(out.J + d[r], jj[r]);
            if (MODE == 1) {
#pragma unroll
                for (int v = 0; v < VX; ++v) {
                    if (!(sens >> (r * VX + v) & 1u)) continue;
                    if constexpr (F64) w.G[d[r] + v] = G[r][v];
                    else w.G[d[r] + v] += FULL ? gp[r][v].value(w.ps.down) : gp[r][v].value49(w.ps.down);
                }
            }
        }
        if (!PL && xp) {
#pragma unroll
            for (int v = 0; v < VX; ++v) {
                const int i = i0 + v;
                if (i >= nx) continue;
                const int se = slab_e(i, nx, np), sh = slab_h(i, nx, np);
                // (E is not updated on the walls, nor are its psi)
                if (se >= 0 && i >= 1 && i <= nx - 2 && j >= 1 && j <= ny - 2)
                    out.pezx[(long long)j * np2 + se] = pex[r][v];
                if (sh >= 0) out.phyx[(long long)j * np2 + sh] = phx[r][v];
            }
        }
        if (!PL && yp) {
            const int te = slab_e(j, ny, np), th = slab_h(j, ny, np);
            if (te >= 0 && j >= 1 && j <= ny - 2) {
#pragma unroll
                for (int v = 0; v < VX; ++v)
                    if (i0 + v < 1 || i0 + v > nx - 2) pey[r][v] = R(0);
                stv(out.pezy + (long long)te * P + i0, pey[r]);
            }
            if (th >= 0) stv(out.phxy + (long long)th * P + i0, phy[r]);
        }
    }
    };
    if constexpr (NB == 0) {
        body(std::false_type{}, std::false_type{});
    } else {
        const int lo = max(np, 1), xe = xr + W - 1, ye = yr + nw * RPW - 1;
        const bool inner = xr >= lo && xe <= nx - 2 - lo && yr - 1 >= lo && ye <= ny - 2 - lo &&
                           !(xr < g.gx0 + g.gnx && xe >= g.gx0 && yr < g.gy0 + g.gny && ye >= g.gy0) &&
                           !(MODE == 0 && xr < g.sx1 && xe >= g.sx0 && yr < g.sy1 && ye >= g.sy0);
        const bool invac = xr >= g.dxa + g.dp || xe < g.dxa || yr >= g.dy0 + g.dny || ye < g.dy0;
        const bool indes = xr >= g.dx0 && xe < g.dx0 + g.dnx && yr >= g.dy0 && ye < g.dy0 + g.dny;
        if (inner && invac) body(std::true_type{}, std::false_type{});
        else if (inner && indes) body(std::false_type{}, std::true_type{});
        else body(std::false_type{}, std::false_type{});
    }
}

// The Drude coefficients of the pitched design box, in the operations of
// the step kernels' drude(): ca, cb, bJ and the adjoint's a1, a2; bJ = 0
// marks the entries that are not Drude nodes (the gap, the row padding).
template <typename R>
__global__ void k_rt2d_coef(const __grid_constant__ Geo2D g, int slot, const R *rho_t, R *coef, long long Mdi)
{
    const Coef<R> &c = coef_at<R>(slot);
    for (long long d = blockIdx.x * (long long)blockDim.x + threadIdx.x; d < Mdi;
         d += (long long)gridDim.x * blockDim.x) {
        const int i = g.dxa + (int)(d % g.dp), j = g.dy0 + (int)(d / g.dp);
        const bool gap = in_range(i, g.gx0, g.gnx) && in_range(j, g.gy0, g.gny);
        R ca = R(0), cb = R(0), bJ = R(0), a1 = R(0), a2 = R(0);
        if (in_range(i, g.dx0, g.dnx) && !gap) {
            const R rt = rho_t[d];
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
        coef[d] = ca;
        coef[Mdi + d] = cb;
        coef[2 * Mdi + d] = bJ;
        coef[3 * Mdi + d] = a1;
        coef[4 * Mdi + d] = a2;
    }
}

}  // namespace

// A wave's fixed part in row steps, fitted to FP32 halos of 4, 6, 8 on seven
// grids (us per forward step, halo 4 / 6 / 8: 316^2 1.60 / 1.29 / 1.12, 530^2
// 2.77 / 2.18 / 2.47, 700^2 3.47 / 3.14 / 3.33, 1400^2 7.2 / 6.9 / 7.9, 2048^2
// 13.7 / 13.2 / 14.1: within 2 % of the best on each), and in FP64 from 3 us of
// launch against 0.24 us per row step.
template <typename R>
Rt2DPlan rt2d_plan(int nx, int ny, int sms, int steps)
{
    using D = Shape<R>;
    constexpr bool F64 = sizeof(R) == 8;
    return rt_tile_plan(nx, ny, sms, D::W, D::RPW, D::MAXW, !F64 && steps > 4 ? RT2D_MAX : 4, F64 ? 10.0 : 350.0);
}

template <typename R, int NB>
using Kernel = decltype(&k_rt2d<R, 0, 0, NB, false>);

// The instance for a mode, a rounding form and a halo.
template <typename R, int NB>
Kernel<R, NB> instance(int mode, int form, int halo)
{
    if (mode == 0) return form ? k_rt2d<R, 0, 1, NB, false> : k_rt2d<R, 0, 0, NB, false>;
    if constexpr (sizeof(R) == 4)
        if (halo > 6) return form ? k_rt2d<R, 1, 1, NB, true> : k_rt2d<R, 1, 0, NB, true>;
    return form ? k_rt2d<R, 1, 1, NB, false> : k_rt2d<R, 1, 0, NB, false>;
}

template <typename R, int NB>
bool allow(size_t b)
{
    bool ok = true;
    for (int q = 0; q < 8; ++q)
        ok = ok && cudaFuncSetAttribute(instance<R, NB>(q & 1, q >> 1 & 1, q & 4 ? RT2D_MAX : 4),
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b) == cudaSuccess;
    return ok;
}

template <typename R>
bool rt2d_ready()
{
    int dev = 0, smem = 0;
    const int Mx = Shape<R>::MAXW;
    const size_t b = std::max(smem_words<R>(Mx, RT2D_MAX, 0, 0), smem_words<R>(Mx, RT2D_MAX, GAP_STAGED, 1)) * sizeof(R);
    bool ok = cudaGetDevice(&dev) == cudaSuccess &&
              cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
              b <= (size_t)smem && allow<R, 1>(b);
    if constexpr (sizeof(R) == 4) ok = ok && allow<R, 2>(b) && allow<R, 0>(b);
    if (!ok) cudaGetLastError();
    return ok;
}

template <typename R, int NB>
void launch_nb(int mode, const Geo2D &g, const State2D<R> &in, const State2D<R> &out, int slot, const Pml1D<R> &px,
               const Pml1D<R> &py, const Rt2D<R> &w, const Rt2DPlan &p, cudaStream_t st)
{
    const int Mg = g.gnx * g.gny;
    const size_t smem = smem_words<R>(p.nw, w.count, mode == 1 && Mg <= GAP_STAGED ? Mg : 0, mode) * sizeof(R);
    const dim3 block(32, p.nw), grid(p.bx, p.by);
    launch_pdl_smem(instance<R, NB>(mode, p.form, p.halo), grid, block, smem, st, g, in, out, slot, px, py, w);
}

// Tiles whose region is plain background (V; those of the source's rows counted too).
template <typename R>
int background_tiles(const Geo2D &g, const Rt2DPlan &p)
{
    using D = Shape<R>;
    const int lo = std::max(g.npml, 1), H = p.halo, h = p.nw * D::RPW;
    int cin = 0, cdes = 0, rin = 0, rdes = 0;
    for (int b = 0; b < p.bx; ++b) {
        const int x = b * p.tw - H;
        if (x < lo || x + D::W - 1 > g.nx - 2 - lo) continue;
        ++cin;
        cdes += x < g.dxa + g.dp && x + D::W > g.dxa;
    }
    for (int b = 0; b < p.by; ++b) {
        const int y = b * p.th - H;
        if (y - 1 < lo || y + h - 1 > g.ny - 2 - lo) continue;
        ++rin;
        rdes += y < g.dy0 + g.dny && y + h > g.dy0;
    }
    return cin * rin - cdes * rdes;
}

// One wave of tiles: it ends with its slowest tile, which is a general one, and
// that one is faster alone (316^2 1.03 / 1.30 us per forward / adjoint step, with
// the instances for background and design box beside it 1.10 / 1.36).
// Two blocks per SM (64 registers a thread: the background's instance fits,
// the others spill) once there are more than four waves: one block's loads and
// stores then overlap the other's steps.  us per forward step, one and two
// blocks per SM: 700^2 (3.2 waves) 3.13 / 3.15, 850^2 (4.8) 3.87 / 3.75, 1400^2
// 8.0 / 6.9, 2048^2 17.8 / 13.2, 1500^2 nearly all design box 13.0 / 11.3.  The
// adjoint, which spills 2 kB outside the background, takes it where five
// eighths of the tiles are background: 2048^2 with a 1024^2 design box (66 %)
// 22.3 / 19.6, 2200 x 1000 with 300^2 (80 %) 9.3 / 8.5, but 1200^2 with 600^2
// (58 %) 8.3 / 8.9 and 1500^2 with 1400^2 (5 %) 20.1 / 22.5.
template <typename R>
int launch_rt2d(int mode, const Geo2D &g, const State2D<R> &in, const State2D<R> &out, int slot, const Pml1D<R> &px,
                const Pml1D<R> &py, const Rt2D<R> &w, const Rt2DPlan &p, cudaStream_t st)
{
    if constexpr (sizeof(R) == 4) {
        if (p.bx * p.by <= p.sms) {
            launch_nb<R, 0>(mode, g, in, out, slot, px, py, w, p, st);
            return 1;
        }
        if (p.bx * p.by > 4 * p.sms && (mode == 0 || 8 * background_tiles<R>(g, p) >= 5 * p.bx * p.by)) {
            launch_nb<R, 2>(mode, g, in, out, slot, px, py, w, p, st);
            return 1;
        }
    }
    launch_nb<R, 1>(mode, g, in, out, slot, px, py, w, p, st);
    return 1;
}

template <typename R>
int launch_rt2d_coef(const Geo2D &g, int slot, const R *rho_t, R *coef, long long Mdi, cudaStream_t st)
{
    const long long nb = std::min<long long>((Mdi + 255) / 256, 152 * 8);
    k_rt2d_coef<R><<<(int)nb, 256, 0, st>>>(g, slot, rho_t, coef, Mdi);
    return 1;
}

// This translation unit's copy of the coefficient slots (constant memory is
// per translation unit).
template <typename R>
cudaError_t upload_coef_rt2d(int slot, const Coef<R> &c, cudaStream_t st)
{
    return write_coef_slot(slot, c, st);
}

#define RT2D_INST(R)                                                                                              \
    template Rt2DPlan rt2d_plan<R>(int, int, int, int);                                                           \
    template bool rt2d_ready<R>();                                                                                \
    template int launch_rt2d<R>(int, const Geo2D &, const State2D<R> &, const State2D<R> &, int,                  \
                                const Pml1D<R> &, const Pml1D<R> &, const Rt2D<R> &, const Rt2DPlan &,            \
                                cudaStream_t);                                                                    \
    template int launch_rt2d_coef<R>(const Geo2D &, int, const R *, R *, long long, cudaStream_t);                \
    template cudaError_t upload_coef_rt2d<R>(int, const Coef<R> &, cudaStream_t);
RT2D_INST(float)
RT2D_INST(double)

}  // namespace fdtd
