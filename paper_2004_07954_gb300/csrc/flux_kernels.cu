// Interface-flux kernels: global Lax-Friedrichs splitting, Roe-averaged characteristic
// projection and WENO-ZN reconstruction of both split parts, one thread per interface (short
// 1D Euler lines: one per interface, field and side, the stage update in the same launch).
// The generic instantiations (GEN = 1: splittings that project the cell split fluxes, global
// LF and Steger-Warming; GEN = 2: those that split per field after the projection, per-field
// and local LF) take the weight function and the flux splitting at run
// time (WENO-Z / linear / Jiang-Shu weights; per-field LF, local LF, Steger-Warming); the
// default scheme keeps its own instantiations.
//
// A block owns a tile of TI interfaces along the sweep direction times TA grid lines.  It
// first computes, once per cell of the tile plus its 3+2 halo cells, the split fluxes
// h+- = (F +- alpha U)/2 and the Roe-average ingredients (sqrt(rho), velocities, H) into
// shared memory; then every thread turns the six cells around its interface into
// F^_{i-1/2} = R (g^+ + g^-).  No interface is computed twice (but by line_kernel, whose blocks
// share the interfaces at their edges).
#include <atomic>

#include "euler_device.cuh"
#include "launch.h"
#include "step_device.cuh"

namespace wz {

namespace {

// Tile shapes: TI interfaces along the sweep x TA lines across it, THREADS per block: one
// interface a thread, and several small blocks an SM, because the FP64 phases of one block
// (cells, Roe state) have to run beside the integer phases of others.  Both sweeps of a 2D
// tile lie alike in shared memory (cell lc of line l at lc TA + l), so one copy of the
// interface code serves both, and a warp covers a patch of 4 x 8 interfaces, which few fronts
// touch (a warp with one stencil at a front runs the weighted evaluation for all of its lanes).
// Both sweeps at 256^2 / 1024^2 / 4096^2, without the linear pass: 80 us / 0.54 / 7.5 ms with four
// blocks (32 warps, 64 registers); three blocks 86 us / 0.53 / 7.5 ms, two 97 us / 0.71 / 9.2 ms,
// 64 x 4 tiles 88 us / 0.58 / 7.55 ms, 128-thread blocks (eight) 84 us / 0.58 / 7.8 ms, a copy of the
// code per sweep (128 x 2 and 32 x 8 tiles) 98 us / 0.63 / 7.85 ms; the loop over the fields rolled
// (a quarter of the code): 77 us.  (Compared before the weights were made exactly odd and the
// linear pass unit-free; the chosen shape takes 80 us / 0.60 / 8.8 ms since.)
// The linear pass (LIN, interface_linear first, the rest compacted, three blocks): both sweeps at
// 800^2 / 1024^2 / 4096^2 310 / 440 us / 5.2 ms with it, 376 / 597 us / 8.8 ms without, on smooth
// waves and jumps; at 256^2 / 512^2 100 / 182 against 78 / 179 us.  A step of a developed flow (400
// steps on): 700^2 1.22 / 1.15 ms, 1024^2 2.01 / 2.16.  On random cells, where nearly every
// interface takes both, 1024^2 2.98 / 2.89 ms, 4096^2 45.3 / 43.3, 2^20 cells of 1D 1.13 / 1.04
// (smooth 0.50 / 0.69).  So lines of kLinearMin cells and more take it, where most interfaces of a
// resolved flow pass and the others lose 3 to 9 %; a single wave of blocks (short 1D lines) waits
// for its slowest block, which pays for both passes, and does without (a rollout at 8192 cells
// 7.7 ms without, 8.2 ms with).
// Long 1D lines use 251-interface tiles (256 cells with the halo: one full round of the cell
// and difference passes; a 2^20-cell step 0.50 ms, without the linear pass 0.69 ms); short
// ones (fewer tiles than twice the SM count) use 64-interface tiles of 64 threads so that
// every SM gets work.  GEN = 2 projects F and U (twice the difference vectors a thread) and runs
// best with two blocks and 128 registers (a 640 x 777 local-LF step 1.76 ms, 1.80 since the
// weights are exactly odd; three blocks 1.81, four 1.85 ms).
constexpr int kLinearMin = 640;
template <int NV, bool SMALL = false> struct Tile { static constexpr int TI = 251, TA = 1, THREADS = 256; };
template <int NV> struct Tile<NV, true> { static constexpr int TI = 64, TA = 1, THREADS = 64; };
template <> struct Tile<4, false> { static constexpr int TI = 32, TA = 8, THREADS = 256; };

// One tile of a sweep along dir: tile ta along the sweep direction, tile tc across it.  (The
// direction is a run-time value where one kernel holds both, so that they share one copy of
// the interface code, which fills most of the instruction cache.)
template <int NV, bool SMALL, int GEN, bool LIN>
__device__ __forceinline__ void flux_tile(const FluxArgs& a, double* Fout, int bc, const int dir, int ta, int tc,
                                          double* smem) {
    using T = Tile<NV, SMALL>;
    constexpr int TI = T::TI, TA = T::TA, kThreads = T::THREADS;
    constexpr int CL = TI + 5;            // cells per line in the tile
    constexpr int NC = CL * TA;           // cells per tile
    constexpr int kStride = TA;           // shared-index step along the sweep (cell lc of line l: lc TA + l)
    const bool x = dir == 0;
    const CellPlanes<NV> sp(smem, NC);

    const int n = x ? a.nx : a.ny;                  // cells along the sweep
    const int nlines = x ? a.ny : a.nx;
    const int j0 = ta * TI;                         // first interface of the tile
    const int l0 = tc * TA;                         // first line of the tile
    const int64_t nc = int64_t(a.nx) * a.ny;
    // cells this tile's interfaces use along the sweep (the last tile of a line may hold
    // fewer than TI interfaces, e.g. only the boundary interface n)
    const int cl_used = min(TI, n + 1 - j0) + 5;

    const double alpha = NV == 1 ? fabs(a.adv_speed) : __longlong_as_double((long long)a.alpha_bits[dir]);
    const double gm1 = a.gamma - 1.0;
    double alpha_f[3] = {0.0, 0.0, 0.0};           // per-field speeds of this direction
    if (GEN == 2 && NV > 1 && a.split == 1)
        for (int k = 0; k < 3; ++k) alpha_f[k] = __longlong_as_double((long long)a.alpha_f_bits[dir * 3 + k]);

    // ---- per-cell quantities -------------------------------------------------------
    for (int idx = threadIdx.x; idx < NC; idx += kThreads) {
        const int l = idx % TA, lc = idx / TA;
        if (lc >= cl_used) break;
        const int line = min(l0 + l, nlines - 1);
        const int gi = j0 - 3 + lc;
        const int g = ghost_src(gi, n, bc);
        const int64_t cell = x ? int64_t(line) * a.nx + g : int64_t(g) * a.nx + line;
        // direction frame: (rho, m_n, m_t, E)
        double Uc[NV];
        Uc[0] = a.U[cell];
        if (NV > 1) {
            Uc[1] = a.U[(x ? 1 : 2) * nc + cell];
            if (NV == 4) Uc[2] = a.U[(x ? 2 : 1) * nc + cell];
            Uc[NV - 1] = a.U[(NV - 1) * nc + cell];
            if (bc == 2 && ghost_mirrored(gi, n, bc)) Uc[1] = -Uc[1];   // wall mirror image
        }
        if (GEN != 0) split_cell_gen<NV>(Uc, a.split, alpha, a.adv_speed, a.gamma, sp, idx);
        else split_cell<NV>(Uc, alpha, a.adv_speed, gm1, sp, idx);
    }
    __syncthreads();
    if (NV > 1) {
        // the split-flux differences of neighbouring cells along the sweep
        for (int idx = threadIdx.x; idx < NC; idx += kThreads) {
            if (idx / TA >= cl_used - 1) break;
            cell_diffs<NV>(sp, idx, kStride);
        }
        __syncthreads();
    }

    // ---- interfaces ----------------------------------------------------------------
    const int nint = n + 1;
    auto store = [&](int idx, const double* Fh) {
        // undoing the direction frame
        const int j = j0 + idx / TA, line = l0 + idx % TA;
        const int64_t base = x ? int64_t(line) * (a.nx + 1) + j : int64_t(j) * a.nx + line;
        const int64_t plane = x ? int64_t(a.ny) * (a.nx + 1) : int64_t(a.ny + 1) * a.nx;
        Fout[base] = Fh[0];
        if (NV > 1) {
            Fout[(x ? 1 : 2) * plane + base] = Fh[1];
            if (NV == 4) Fout[(x ? 2 : 1) * plane + base] = Fh[2];
            Fout[(NV - 1) * plane + base] = Fh[NV - 1];
        }
    };
    // LIN: the interfaces with near-optimal weights first; the others are listed and share full
    // warps afterwards
    __shared__ int s_count;
    __shared__ unsigned short s_list[LIN ? TI * TA : 1];
    int count = TI * TA;
    const bool linear = LIN && n >= kLinearMin;
    if (LIN && linear) {
        if (threadIdx.x == 0) s_count = 0;
        __syncthreads();
        for (int idx = threadIdx.x; idx < TI * TA; idx += kThreads) {
            const int j = j0 + idx / TA, line = l0 + idx % TA;
            if (j >= nint || line >= nlines) continue;
            double Fh[NV];
            if (interface_linear<NV>(sp, idx, kStride, gm1, a.wide, Fh)) store(idx, Fh);
            else s_list[atomicAdd(&s_count, 1)] = (unsigned short)idx;
        }
        __syncthreads();
        count = s_count;
    }
    for (int q = threadIdx.x; q < count; q += kThreads) {
        const int idx = LIN && linear ? s_list[q] : q;
        const int j = j0 + idx / TA, line = l0 + idx % TA;
        if (j >= nint || line >= nlines) continue;
        double Fh[NV];
        interface_flux<NV, GEN>(sp, idx, kStride, gm1, a.wide, a.eps4, a.kappa, a.weights, a.split, alpha_f, Fh);
        store(idx, Fh);
    }
}

// Whether a problem takes the LIN kernels: WENO-ZN weights on split fluxes, and a line long
// enough for smooth data to be resolved well.
bool takes_linear(const FluxArgs& a, int n) { return a.weights == 0 && (a.split == 0 || a.split == 3) && n >= kLinearMin; }

// Blocks an SM: see the tile shapes
template <int NV, bool SMALL, int GEN, bool LIN>
constexpr int min_blocks() { return SMALL || GEN == 2 ? 2 : (NV == 4 && LIN ? 3 : 4); }

template <int NV, int DIR, bool SMALL, int GEN, bool LIN>
__global__ void __launch_bounds__(Tile<NV, SMALL>::THREADS, (min_blocks<NV, SMALL, GEN, LIN>())) flux_kernel(FluxArgs a) {
    extern __shared__ double smem[];
    pdl_wait();
    flux_tile<NV, SMALL, GEN, LIN>(a, a.Fout, a.bc, DIR, DIR == 0 ? blockIdx.x : blockIdx.y,
                                   DIR == 0 ? blockIdx.y : blockIdx.x, smem);
}

// Short 1D lines: too few interfaces to fill the GPU, so the time of a launch is the time of one
// thread's chain of instructions, and the launches themselves.  Euler: six warps share 32
// interfaces; after the cells, warp 0 forms the Roe states and the projection's coefficients
// while the others difference the cells, then warp (side, field) reconstructs one part of
// one field for each interface, and three warps form a flux component each.  Advection: a warp
// per part.  STAGE: the block goes on to the stage update of the cells between its
// interfaces (31 of them: neighbouring blocks both compute the interface they share) and
// their LF speeds, in the arithmetic of update_kernel, so that a stage is one launch.
// A CFL step at 200 and 8192 cells: 59 and 62 us with a thread per interface (64-thread blocks) and
// an update launch, 39 and 47 us with this flux kernel and the update launch, 29 and 32 us as one;
// advection at 160 cells 13 -> 7.6 us.
// Up to which length: as long as the blocks are one wave, six an SM (56 registers) for the default
// scheme, five (64) for the generic ones (the launch bounds hold them there).  A step as one launch a stage / by the 64-thread flux
// kernel and the update: 28,000 cells 52 / 82 us, 32,768 76 / 72, 36,864 81 / 71, 60,000 118 / 101;
// Steger-Warming 22,000 cells 60 / 90, 24,000 91 / 86; WENO-Z 45 / 72 and 73 / 70.
// (Those are 152 SMs.)  Advection's blocks hold 64 threads and more of them fit; it takes the
// same limit, on whose near side the one launch wins as well (28,000 cells 15.1 / 18.9 us).
constexpr int kLineTI = 32;
int line_max(bool gen) { return (gen ? 5 : 6) * sm_count_cached() * (kLineTI - 1); }
template <int NV> constexpr int kLineThreads = NV == 3 ? 192 : 64;

template <int NV, int GEN, bool STAGE>
__global__ void __launch_bounds__(kLineThreads<NV>, NV == 3 ? (GEN == 0 ? 6 : 5) : 1) line_kernel(FluxArgs a, UpdateArgs u) {
    constexpr int TI = kLineTI, NC = TI + 5, W = GEN == 0 ? 0 : -1, kThreads = kLineThreads<NV>;
    __shared__ double s_planes[NC * CellPlanes<NV>::kPerCellDefault];
    __shared__ double s_R[NV == 3 ? 8 : 1][TI], s_g[2][NV][TI];
    __shared__ int s_P[NV == 3 ? 13 : 1][TI];
    __shared__ int s_bad[TI];
    __shared__ double s_F[STAGE ? NV : 1][TI], s_dt;
    const CellPlanes<NV> sp(s_planes, NC);
    pdl_wait();
    const int tid = threadIdx.x, w = tid >> 5, i = tid & 31;
    const int j0 = blockIdx.x * (STAGE ? TI - 1 : TI), n = a.nx;
    const int cl_used = min(TI, n + 1 - j0) + 5;
    const double alpha = NV == 1 ? fabs(a.adv_speed) : __longlong_as_double((long long)a.alpha_bits[0]);
    const double gm1 = a.gamma - 1.0;
    // the update's own inputs: component w of cell j0 + i
    const bool mine = STAGE && w < NV && i < TI - 1 && j0 + i < n;
    double us = 0.0, un = 0.0;
    if (mine && u.mode != 0) {
        us = u.Us[w * int64_t(n) + j0 + i];
        if (u.mode > 1) un = u.Un[w * int64_t(n) + j0 + i];
    }
    if (tid < cl_used) {
        const int gi = j0 - 3 + tid, g = ghost_src(gi, n, a.bc);
        double Uc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) Uc[k] = a.U[k * int64_t(n) + g];
        if (NV > 1 && a.bc == 2 && ghost_mirrored(gi, n, a.bc)) Uc[1] = -Uc[1];   // wall mirror image
        if (GEN != 0) split_cell_gen<NV>(Uc, a.split, alpha, a.adv_speed, a.gamma, sp, tid);
        else split_cell<NV>(Uc, alpha, a.adv_speed, gm1, sp, tid);
    }
    if (STAGE && tid == kThreads - 1) {
        double dt = 0.0;
        if (u.mode == 1) {
            dt = step_dt(u, NV == 1 ? 0 : 1);
            if (blockIdx.x == 0) u.ctrl->dt = dt;
        } else if (u.mode > 1) {
            dt = u.ctrl->dt;
        }
        s_dt = dt;
    }
    __syncthreads();
    const bool live = j0 + i <= n;
    double Fw = 0.0;                           // flux component w of interface i
    if constexpr (NV == 1) {
        if (live) {
            const double* h = w == 0 ? sp.hp : sp.hm;
            const int o = w == 0 ? i : i + 5, d = w == 0 ? 1 : -1;
            const double h0 = h[o], h1 = h[o + d], h2 = h[o + 2 * d], h3 = h[o + 3 * d], h4 = h[o + 4 * d];
            s_g[w][0][i] = zn_flux_wide<W>(h0 - h1, h1 - h2, h2 - h3, h3 - h4, h2, a.wide, a.eps4, a.kappa,
                                           GEN == 0 ? 0 : a.weights);
        }
        __syncthreads();
        if (w == 0) Fw = s_g[0][0][i] + s_g[1][0][i];
    } else {
        if (w == 0) {
            s_bad[i] = 0;
            if (live) {
                const RoeState<3> R(sp, i + 2, i + 3, gm1);
                const WideProjection<3> P(R);
                const double r[8] = {R.u, R.v, R.H, R.c, R.hrc, R.hq2, R.hb1, R.hb2};
                const int q[13] = {P.z0.h, P.z0.l, P.z1.h, P.z1.l, P.zE.h, P.zE.l, P.p0.h, P.p0.l, P.p1.h, P.p1.l, P.e0, P.e1, P.eE};
#pragma unroll
                for (int m = 0; m < 8; ++m) s_R[m][i] = r[m];
#pragma unroll
                for (int m = 0; m < 13; ++m) s_P[m][i] = q[m];
            }
        } else {
            for (int c = tid - 32; c < 2 * (cl_used - 1); c += kThreads - 32) {
                const int side = c >= cl_used - 1;
                cell_diffs_side<NV>(sp, side ? c - (cl_used - 1) : c, 1, side);
            }
        }
        __syncthreads();
        const int side = w / 3, k = w % 3;
        if (live) {
            WideProjection<3> P;
            P.z0 = Limbs(s_P[0][i], s_P[1][i]);
            P.z1 = Limbs(s_P[2][i], s_P[3][i]);
            P.zE = Limbs(s_P[4][i], s_P[5][i]);
            P.p0 = Limbs(s_P[6][i], s_P[7][i]);
            P.p1 = Limbs(s_P[8][i], s_P[9][i]);
            P.e0 = s_P[10][i];
            P.e1 = s_P[11][i];
            P.eE = s_P[12][i];
            // (the scale of the field's value as in interface_flux)
            const int eb = (GEN == 0 ? exponent_of(sp.hp[i + 2]) : max_i(exponent_of(sp.hp[i + 2]), exponent_of(sp.hm[i + 3]))) - 2;
            int64_t D[4];
            int G[4];
            uint32_t xm = 0;
#pragma unroll
            for (int st = 0; st < 4; ++st) {
                int64_t d[3];
                int g[3];
                P.apply(side == 0 ? sp.dp : sp.dm, sp.ex + 2 * side * NC, NC, side == 0 ? i + st : i + 4 - st, d, g, xm);
                D[st] = k == 0 ? d[0] : (k == 1 ? d[1] : d[2]);
                G[st] = k == 0 ? g[0] : (k == 1 ? g[1] : g[2]);
            }
            double corr;
            const bool ok = wide_correction<W>(D[0], D[1], D[2], D[3], G[0], G[1], G[2], G[3], eb, a.wide, a.weights, corr);
            if (!ok || (xm & 0xffffu) == 2047u || (xm >> 16) == 2047u) s_bad[i] = 1;
            s_g[side][k][i] = corr;
        }
        __syncthreads();
        if (live && w < 3) {
            RoeState<3> R;
            R.u = s_R[0][i];
            R.v = s_R[1][i];
            R.H = s_R[2][i];
            R.c = s_R[3][i];
            R.hrc = s_R[4][i];
            R.hq2 = s_R[5][i];
            R.hb1 = s_R[6][i];
            R.hb2 = s_R[7][i];
            double gh[3], hc[3], Fh[3];
            if (s_bad[i]) {
                field_fluxes_double<3, GEN>(sp, R, i, 1, a.eps4, a.kappa, GEN == 0 ? 0 : a.weights, nullptr, gh);
            } else {
#pragma unroll
                for (int m = 0; m < 3; ++m) gh[m] = s_g[0][m][i] - s_g[1][m][i];
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) hc[m] = sp.hp[m * NC + i + 2] + sp.hm[m * NC + i + 3];
            R.back_project(gh, hc, Fh);
            Fw = w == 0 ? Fh[0] : (w == 1 ? Fh[1] : Fh[2]);
        }
    }
    if (!STAGE) {
        if (live && w < NV) a.Fout[w * int64_t(n + 1) + j0 + i] = Fw;
        return;
    }
    if (w < NV) s_F[w][i] = Fw;
    __syncthreads();
    // the stage update, as update_kernel
    bool bad = false;
    double r = 0.0;
    if (mine) {
        const double dF = s_F[w][i + 1] - s_F[w][i];
        if (u.mode == 0) {
            r = -(dF * u.rdx);
            bad = (__double2hiint(r) & 0x7ff00000) == 0x7ff00000;
        } else {
            const double wk = u.mode == 1 ? 1.0 : (u.mode == 2 ? 0.25 : 2.0 / 3.0);
            const double kx = wk * s_dt * u.rdx;
            double base = us;
            if (u.mode == 2) base = fma(0.75, un, 0.25 * us);
            else if (u.mode == 3) base = fma(1.0 / 3.0, un, (2.0 / 3.0) * us);
            r = fma(-kx, dF, base);
            if (NV == 1) bad = !isfinite(r);
        }
        u.out[w * int64_t(n) + j0 + i] = r;
    }
    if (NV == 3 && u.mode != 0 && (u.next_slot >= 0 || u.alpha_next || u.mode == 3)) {
        // (s_g is free since the last barrier but one)
        if (w < NV) s_g[0][w][i] = r;
        __syncthreads();
        if (w == 0) {
            double sx = 0.0;
            if (mine) {
                const double st[3] = {s_g[0][0][i], s_g[0][1][i], s_g[0][2][i]};
                double uu, vv, c;
                const bool adm = wave_state<3>(st, u.gamma, uu, vv, c);
                sx = __dadd_rn(fabs(uu), c);
                bad = !(adm && isfinite(sx));
            }
            const double mx = warp_max(fmax(0.0, sx));
            unsigned long long* dst = u.alpha_next ? u.alpha_next : (u.next_slot >= 0 ? u.ctrl->alpha[u.next_slot] : nullptr);
            if (i == 0 && dst) atomicMax(dst, (unsigned long long)__double_as_longlong(mx));
        }
    }
    if (bad) atomicOr(&u.ctrl->status, kStatusNonFinite);
    if (u.clear_slot >= 0 && blockIdx.x == 0 && tid < 8) {
        unsigned long long* z = tid < 2 ? &u.ctrl->alpha[u.clear_slot][tid] : &u.ctrl->alpha_f[u.clear_slot][0][tid - 2];
        *z = 0ull;
    }
}

// Both sweeps of a 2D stage in one grid, so that they share one tail: blocks [0, nbx) take
// the x tiles (along the sweep fastest, as flux_kernel<4, 0>), the others the y tiles
// (across the sweep fastest, as flux_kernel<4, 1>).
template <int GEN, bool LIN>
__global__ void __launch_bounds__(Tile<4>::THREADS, (min_blocks<4, false, GEN, LIN>()))
    flux_xy_kernel(FluxArgs ax, double* Fy, int bc_y, int x_along, int nbx, int y_across) {
    extern __shared__ double smem[];
    pdl_wait();
    const int b = int(blockIdx.x), q = b - nbx;
    const bool x = b < nbx;
    flux_tile<4, false, GEN, LIN>(ax, x ? ax.Fout : Fy, x ? ax.bc : bc_y, x ? 0 : 1, x ? b % x_along : q / y_across,
                                  x ? b / x_along : q % y_across, smem);
}

template <int NV, bool SMALL, int GEN>
constexpr size_t tile_smem() {
    return size_t((Tile<NV, SMALL>::TI + 5) * Tile<NV, SMALL>::TA) *
           (GEN != 0 ? CellPlanes<NV>::kPerCellGeneric : CellPlanes<NV>::kPerCellDefault) * sizeof(double);
}

template <int GEN, bool LIN>
cudaError_t launch_xy(const FluxArgs& ax, const FluxArgs& ay, cudaStream_t s) {
    constexpr size_t smem = tile_smem<4, false, GEN>();
    static std::atomic<unsigned long long> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(flux_xy_kernel<GEN, LIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    const int x_along = (ax.nx + 1 + Tile<4>::TI - 1) / Tile<4>::TI;
    const int nbx = x_along * ((ax.ny + Tile<4>::TA - 1) / Tile<4>::TA);
    const int y_across = (ay.nx + Tile<4>::TA - 1) / Tile<4>::TA;
    const int nby = y_across * ((ay.ny + 1 + Tile<4>::TI - 1) / Tile<4>::TI);
    return launch_pdl(flux_xy_kernel<GEN, LIN>, dim3(unsigned(nbx + nby)), dim3(Tile<4>::THREADS), smem, s, ax, ay.Fout,
                      ay.bc, x_along, nbx, y_across);
}

template <int NV, int DIR, bool SMALL, int GEN, bool LIN>
cudaError_t launch_one(const FluxArgs& a, cudaStream_t s) {
    constexpr int TI = Tile<NV, SMALL>::TI, TA = Tile<NV, SMALL>::TA;
    constexpr size_t smem = tile_smem<NV, SMALL, GEN>();
    // the dynamic shared-memory limit is a per-device function attribute
    static std::atomic<unsigned long long> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(flux_kernel<NV, DIR, SMALL, GEN, LIN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 int(smem));
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    const int n = DIR == 0 ? a.nx : a.ny;
    const int nlines = DIR == 0 ? a.ny : a.nx;
    const unsigned along = unsigned((n + 1 + TI - 1) / TI);
    const unsigned across = unsigned((nlines + TA - 1) / TA);
    dim3 grid = DIR == 0 ? dim3(along, across) : dim3(across, along);
    return launch_pdl(flux_kernel<NV, DIR, SMALL, GEN, LIN>, grid, dim3(Tile<NV, SMALL>::THREADS), smem, s, a);
}

template <int GEN>
cudaError_t launch_flux_t(int system, int dir, const FluxArgs& a, cudaStream_t s) {
    if (system != 2) {
        // 1D: short lines take the small tiles so that every SM has work
        const int64_t big_tiles = (int64_t(a.nx) + Tile<3>::TI) / Tile<3>::TI * a.ny;
        const bool small = big_tiles < 2 * sm_count_cached();
        if (system == 0)
            return small ? launch_one<1, 0, true, GEN, false>(a, s) : launch_one<1, 0, false, GEN, false>(a, s);
        if constexpr (GEN != 2)
            if (a.nx < line_max(GEN != 0))
                return launch_pdl(line_kernel<3, GEN, false>, dim3(unsigned((a.nx + kLineTI) / kLineTI)),
                                  dim3(kLineThreads<3>), 0, s, a, UpdateArgs{});
        if (small) return launch_one<3, 0, true, GEN, false>(a, s);
        if constexpr (GEN != 2)
            if (takes_linear(a, a.nx)) return launch_one<3, 0, false, GEN, true>(a, s);
        return launch_one<3, 0, false, GEN, false>(a, s);
    }
    if constexpr (GEN != 2)
        if (takes_linear(a, dir == 0 ? a.nx : a.ny))
            return dir == 0 ? launch_one<4, 0, false, GEN, true>(a, s) : launch_one<4, 1, false, GEN, true>(a, s);
    return dir == 0 ? launch_one<4, 0, false, GEN, false>(a, s) : launch_one<4, 1, false, GEN, false>(a, s);
}

}  // namespace

cudaError_t launch_flux_xy(const FluxArgs& ax, const FluxArgs& ay, cudaStream_t s) {
    const bool lin = takes_linear(ax, ax.nx > ax.ny ? ax.nx : ax.ny);
    if (ax.weights == 0 && ax.split == 0) return lin ? launch_xy<0, true>(ax, ay, s) : launch_xy<0, false>(ax, ay, s);
    if (ax.split == 0 || ax.split == 3) return lin ? launch_xy<1, true>(ax, ay, s) : launch_xy<1, false>(ax, ay, s);
    return launch_xy<2, false>(ax, ay, s);
}

bool line_stage_applies(int system, const FluxArgs& a) {
    const bool gen = a.weights != 0 || (system == 1 && a.split != 0);
    return system != 2 && a.nx < line_max(gen) && (system == 0 || a.split == 0 || a.split == 3);
}

cudaError_t launch_line_stage(int system, const FluxArgs& a, const UpdateArgs& u, cudaStream_t s) {
    const dim3 grid(unsigned((a.nx + kLineTI - 2) / (kLineTI - 1)));
    const bool gen = a.weights != 0 || (system == 1 && a.split != 0);
    if (system == 0)
        return gen ? launch_pdl(line_kernel<1, 1, true>, grid, dim3(kLineThreads<1>), 0, s, a, u)
                   : launch_pdl(line_kernel<1, 0, true>, grid, dim3(kLineThreads<1>), 0, s, a, u);
    return gen ? launch_pdl(line_kernel<3, 1, true>, grid, dim3(kLineThreads<3>), 0, s, a, u)
               : launch_pdl(line_kernel<3, 0, true>, grid, dim3(kLineThreads<3>), 0, s, a, u);
}

cudaError_t launch_flux(int system, int dir, const FluxArgs& a, cudaStream_t s) {
    if (a.weights == 0 && (system == 0 || a.split == 0)) return launch_flux_t<0>(system, dir, a, s);
    // advection ignores the splitting
    const bool diff = system == 0 || a.split == 0 || a.split == 3;
    return diff ? launch_flux_t<1>(system, dir, a, s) : launch_flux_t<2>(system, dir, a, s);
}

}  // namespace wz
