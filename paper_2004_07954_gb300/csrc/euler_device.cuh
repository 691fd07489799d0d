// Per-cell and per-interface building blocks shared by the single-problem flux kernels and
// the batched kernel: LF flux splitting of one cell (Sec. 2, Sec. 4.3) and the numerical
// flux of one interface (Roe average, characteristic projection, WENO-ZN of both split
// parts, back-projection).  Everything lives in shared memory planes of a tile.
#pragma once

#include "wenozn_device.cuh"

namespace wz {

// Shared-memory planes of one tile of NC cells: split fluxes h+ and h- (NV planes each),
// and for the Euler systems sqrt(rho), u_n, H (and u_t in 2D), the differences
// dh+-_c = h+-_c - h+-_{c+1} along the sweep (NV planes each, as signed 64-bit mantissas with
// their exponents) and, in the generic kernels, the cell's |u_n| + c.
template <int NV>
struct CellPlanes {
    static constexpr int kPerCell = NV == 1 ? 2 : 2 * NV + (NV == 4 ? 4 : 3);
    // + dh+, dh- and four exponent words (two 16-bit exponents each)
    static constexpr int kPerCellDefault = kPerCell + (NV == 1 ? 0 : 2 * NV + 2);
    static constexpr int kPerCellGeneric = kPerCellDefault + (NV == 1 ? 0 : 1);   // + |u_n| + c
    double* hp;
    double* hm;
    double* sr;
    double* un;
    double* H;
    double* ut;
    int64_t* dp;         // Euler: mantissas of dh+ and dh-
    int64_t* dm;
    uint32_t* ex;        // exponents of dh+ (0, 1), (2, 3) and dh- alike, a plane each
    double* sp;          // generic kernels: the cell's |u_n| + c (local LF)
    int NC;
    __device__ __forceinline__ CellPlanes(double* base, int nc) : NC(nc) {
        hp = base;
        hm = hp + NV * nc;
        sr = hm + NV * nc;
        un = sr + nc;
        H = un + nc;
        ut = H + nc;
        dp = reinterpret_cast<int64_t*>(base + kPerCell * nc);
        dm = dp + NV * nc;
        ex = reinterpret_cast<uint32_t*>(dm + NV * nc);
        sp = base + kPerCellDefault * nc;
    }
};

// The split-flux differences of cell si and its neighbour si + stride along the sweep, once
// per cell: the characteristic projection is linear, so the reconstructions' stencil
// differences are projections of these (no cell difference is formed per interface and field).
template <int NV>
__device__ __forceinline__ void cell_diffs_side(const CellPlanes<NV>& s, int si, int stride, int side) {
    const double* h = side == 0 ? s.hp : s.hm;
    int64_t* d = side == 0 ? s.dp : s.dm;
    int e[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < NV; ++k)
        d[k * s.NC + si] = wide_unpack(h[k * s.NC + si] - h[k * s.NC + si + stride], e[k]);
    s.ex[2 * side * s.NC + si] = uint32_t(e[0] | (e[1] << 16));
    s.ex[(2 * side + 1) * s.NC + si] = uint32_t(e[2] | (e[3] << 16));
}

template <int NV>
__device__ __forceinline__ void cell_diffs(const CellPlanes<NV>& s, int si, int stride) {
#pragma unroll
    for (int side = 0; side < 2; ++side) cell_diffs_side<NV>(s, si, stride, side);
}

// 1/sqrt(x) in integer arithmetic (correctly rounded but for 0.6 % of a last place), CUDA's where
// x is not positive and normal
__device__ __forceinline__ double inv_sqrt(double x) {
    bool ok;
    const double r = wide_rsqrt(x, ok);
    return ok ? r : rsqrt(x);
}

// sqrt(x) through it (one more rounding)
__device__ __forceinline__ double square_root(double x) {
    bool ok;
    const double r = wide_rsqrt(x, ok);
    return ok ? x * r : sqrt(x);
}

// One cell: Uc = (rho, m_n[, m_t], E) in the sweep direction's frame (or the scalar u with
// the advection speed `a`), alpha the LF speed.  Writes h+- = (F +- alpha U)/2 and the Roe
// ingredients at shared index si.
template <int NV>
__device__ __forceinline__ void split_cell(const double* Uc, double alpha, double a_adv, double gm1,
                                           const CellPlanes<NV>& s, int si) {
    const double half_a = 0.5 * alpha;
    if (NV == 1) {
        const double u = Uc[0];
        const double f = a_adv * u;
        s.hp[si] = 0.5 * fma(alpha, u, f);
        s.hm[si] = 0.5 * fma(-alpha, u, f);
        return;
    }
    const double rho = Uc[0], mn = Uc[1], E = Uc[NV - 1];
    const double mt = NV == 4 ? Uc[2] : 0.0;
    const double rs = inv_sqrt(rho);
    const double rr = rs * rs;                         // 1 / rho
    const double un = mn * rr;
    const double ut = mt * rr;
    // p/2 = (gamma-1)(E - (m_n u_n + m_t u_t)/2)/2
    const double mq = NV == 4 ? fma(mn, un, mt * ut) : mn * un;
    const double hp2 = fma(-0.25 * gm1, mq, (0.5 * gm1) * E);
    const double Ep = fma(2.0, hp2, E);
    // half the physical flux, F/2 = (m_n, m_n u_n + p, m_t u_n, u_n (E + p)) / 2
    const double hun = wide_half(un);
    double hF[NV];
    hF[0] = wide_half(mn);
    hF[1] = fma(mn, hun, hp2);
    if (NV == 4) hF[2] = mt * hun;
    hF[NV - 1] = hun * Ep;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        s.hp[k * s.NC + si] = fma(half_a, Uc[k], hF[k]);
        s.hm[k * s.NC + si] = fma(-half_a, Uc[k], hF[k]);
    }
    s.sr[si] = rho * rs;                               // sqrt(rho)
    s.un[si] = un;
    s.H[si] = Ep * rr;
    if (NV == 4) s.ut[si] = ut;
}

// The cell phase of the generic kernels, by splitting (split: 0 global LF, 1 per-field LF,
// 2 local LF, 3 Steger-Warming):
//   0     h+- = (F +- alpha U)/2, as split_cell;
//   1, 2  hp = F/2, hm = U/2 (split after the projection, per field or per interface), and
//         for 2 the cell's |u_n| + c in the speed plane;
//   3     hp = F+, hm = F- of Steger and Warming:
//         F+- = rho/(2 gamma) (2(g-1) l2 + l1 + l3, 2(g-1) l2 u + l1 (u-c) + l3 (u+c),
//                              [(2(g-1) l2 + l1 + l3) v,] (g-1) l2 q^2 + l1 ((u-c)^2 + v^2)/2
//                              + l3 ((u+c)^2 + v^2)/2 + (3-g)(l1 + l3) c^2 / (2(g-1)))
//         with l = (u-c, u, u+c) and l+- = (l +- |l|)/2, q^2 = u^2 + v^2.
// Advection ignores the splitting (every variant reduces to alpha = |a| there).
template <int NV>
__device__ __forceinline__ void split_cell_gen(const double* Uc, int split, double alpha, double a_adv,
                                               double gamma, const CellPlanes<NV>& s, int si) {
    const double gm1 = gamma - 1.0;
    if (NV == 1 || split == 0) {
        split_cell<NV>(Uc, alpha, a_adv, gm1, s, si);
        return;
    }
    const double rho = Uc[0], mn = Uc[1], E = Uc[NV - 1];
    const double mt = NV == 4 ? Uc[2] : 0.0;
    const double rs = inv_sqrt(rho);
    const double rr = rs * rs;
    const double un = mn * rr;
    const double ut = mt * rr;
    const double kin = wide_half(NV == 4 ? fma(mn, un, mt * ut) : mn * un);
    const double p = gm1 * (E - kin);
    const double Ep = E + p;
    if (split == 3) {
        const double c = square_root(gamma * p * rr);
        const double l1 = un - c, l3 = un + c;
        // (l + |l|)/2 and (l - |l|)/2: l or zero by its sign
        const double l[3] = {l1, un, l3};
        double lp[3], lm[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const bool neg = __double2hiint(l[i]) < 0;
            lp[i] = neg ? 0.0 : l[i];
            lm[i] = neg ? l[i] : 0.0;
        }
        const double k0 = rho * (1.0 / (2.0 * gamma));
        const double q2 = NV == 4 ? fma(un, un, ut * ut) : un * un;
        const double vv = NV == 4 ? ut * ut : 0.0;
        const double e1 = wide_half(fma(l1, l1, vv)), e3 = wide_half(fma(l3, l3, vv));     // ((u -+ c)^2 + v^2)/2
        const double w13 = ((3.0 - gamma) / (2.0 * gm1)) * (c * c);
        const double g2 = 2.0 * gm1;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const double* ls = side == 0 ? lp : lm;
            double* h = side == 0 ? s.hp : s.hm;
            const double s13 = ls[0] + ls[2];
            const double m0 = fma(g2, ls[1], s13);
            h[si] = k0 * m0;
            h[s.NC + si] = k0 * fma(g2 * ls[1], un, fma(ls[0], l1, ls[2] * l3));
            if (NV == 4) h[2 * s.NC + si] = k0 * (m0 * ut);
            h[(NV - 1) * s.NC + si] = k0 * fma(gm1 * ls[1], q2, fma(ls[0], e1, fma(ls[2], e3, s13 * w13)));
        }
    } else {
        const double hun = wide_half(un);
        double hF[NV];
        hF[0] = wide_half(mn);
        hF[1] = fma(mn, hun, wide_half(p));
        if (NV == 4) hF[2] = mt * hun;
        hF[NV - 1] = hun * Ep;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            s.hp[k * s.NC + si] = hF[k];
            s.hm[k * s.NC + si] = wide_half(Uc[k]);
        }
        // local LF: the cell's |u_n| + c (the interface takes the largest of its six cells;
        // the per-field splitting reads global speeds instead)
        if (split == 2) s.sp[si] = fabs(un) + square_root(gamma * p * rr);
    }
    s.sr[si] = rho * rs;
    s.un[si] = un;
    s.H[si] = Ep * rr;
    if (NV == 4) s.ut[si] = ut;
}

// Numerical flux F^ at the interface between the stencil's cells 2 and 3, the stencil being
// the six cells base + k*stride, k = 0..5 (cells i-2 .. i+3 around x_{i+1/2}), in the sweep
// direction's frame: Roe average of cells 2 and 3, projection of the split fluxes onto its left
// eigenvectors (rows, direction frame)
//   l_{u-c} = ( (b2 + u/c)/2, -(b1 u + 1/c)/2, -b1 v/2, b1/2 )
//   l_u     = ( 1 - b2, b1 u, b1 v, -b1 )
//   l_shear = ( -v, 0, 1, 0 )                          (2D only)
//   l_{u+c} = ( (b2 - u/c)/2, -(b1 u - 1/c)/2, -b1 v/2, b1/2 )
// (b1 = (gamma - 1)/c^2, b2 = q^2 b1 / 2), reconstruction of both parts per field, and
// back-projection F^ = R g^ with the right eigenvectors (columns)
//   r_{u-c} = (1, u-c, [v,] H-uc), r_u = (1, u, [v,] q^2/2), r_shear = (0, 0, 1, v),
//   r_{u+c} = (1, u+c, [v,] H+uc).
// Each field's reconstructions need only the first differences of its stencil and the centre
// value: plus side (g+ at cells 0..4) D_s = l.dh+ at cells s - 1, centre l.h+_2; minus side,
// the mirrored stencil of g- at cells 5..1, D_s = -l.dh- at cells 5 - s, centre l.h-_3.  The
// centres are not projected at all: R L = 1, so with g^ = L (h+_2 + h-_3) + gh, gh the sums of
// the fields' two f^ - c, F^ = h+_2 + h-_3 + R gh (13 FP64 instructions less, and constant data
// give equal fluxes exactly).
template <int NV>
struct RoeState {
    double u, v, H, c, hrc, hq2, hb1, hb2;   // hrc = 1/(2c), hq2 = q^2/2, hb1 = b1/2, hb2 = b2/2
    RoeState() = default;
    __device__ __forceinline__ RoeState(const CellPlanes<NV>& s, int cl, int cr, double gm1) {
        const double srl = s.sr[cl];
        const double wl = srl * wide_reciprocal(srl + s.sr[cr]);
        u = fma(wl, s.un[cl] - s.un[cr], s.un[cr]);
        v = NV == 4 ? fma(wl, s.ut[cl] - s.ut[cr], s.ut[cr]) : 0.0;
        H = fma(wl, s.H[cl] - s.H[cr], s.H[cr]);
        const double q2 = NV == 4 ? fma(u, u, v * v) : u * u;
        hq2 = wide_half(q2);
        const double c2 = gm1 * (H - hq2);
        const double rc = inv_sqrt(c2);
        c = c2 * rc;
        hrc = wide_half(rc);
        hb1 = (0.5 * gm1) * (rc * rc);
        hb2 = hq2 * hb1;
    }
    // g = L h through the rows' shared parts: with W = u h_1 + v h_2 - h_E, Z = b2 h_0 - b1 W
    // and B = (u h_0 - h_1)/(2c),
    //   l_u.h = h_0 - Z,  l_{u-+c}.h = Z/2 +- B,  l_shear.h = h_2 - v h_0.
    __device__ __forceinline__ void project(const double* h, double* g) const {
        const double h0 = h[0], h1 = h[1], hE = h[NV - 1];
        const double W = NV == 4 ? fma(u, h1, fma(v, h[2], -hE)) : fma(u, h1, -hE);
        const double Zh = fma(hb2, h0, -(hb1 * W));          // Z / 2
        const double Bi = fma(u, h0, -h1);                   // 2 c B
        g[0] = fma(hrc, Bi, Zh);
        g[1] = fma(-2.0, Zh, h0);
        if (NV == 4) g[2] = fma(-v, h0, h[2]);
        g[NV - 1] = fma(-hrc, Bi, Zh);
    }
    // Fh = hc + R gh
    __device__ __forceinline__ void back_project(const double* gh, const double* hc, double* Fh) const {
        const double uc = u * c, s = gh[0] + gh[NV - 1], d = gh[NV - 1] - gh[0], f = s + gh[1];
        Fh[0] = hc[0] + f;
        Fh[1] = fma(u, f, fma(c, d, hc[1]));
        if (NV == 3) {
            Fh[2] = fma(H, s, fma(uc, d, fma(hq2, gh[1], hc[2])));
        } else {
            Fh[2] = fma(v, f, gh[2] + hc[2]);
            Fh[3] = fma(H, s, fma(uc, d, fma(hq2, gh[1], fma(v, gh[2], hc[3]))));
        }
    }
};

// The fields' f^ - c (sum of both parts) in double arithmetic throughout, for stencils outside the
// range of the integer projection.  GEN 2: the planes hold F/2 and U/2, split per field with
// the speeds ak.
template <int NV, int GEN>
__device__ __noinline__ void field_fluxes_double(const CellPlanes<NV>& s, const RoeState<NV>& R, int base,
                                                 int stride, double eps4, double kappa, int weights,
                                                 const double* ak, double* gh) {
    double D[2][4][NV];
#pragma unroll 1
    for (int side = 0; side < 2; ++side)
#pragma unroll 1
        for (int st = 0; st < 4; ++st) {
            const int i = base + (side == 0 ? st : 4 - st) * stride;
            double g[2][NV];
#pragma unroll 1
            for (int q = 0; q < 2; ++q) {
                const double* h = q == 0 ? s.hp : s.hm;
                double dh[NV];
#pragma unroll
                for (int k = 0; k < NV; ++k) dh[k] = h[k * s.NC + i] - h[k * s.NC + i + stride];
                R.project(dh, g[q]);
            }
#pragma unroll 1
            for (int k = 0; k < NV; ++k)
                D[side][st][k] = GEN == 2 ? (side == 0 ? fma(ak[k], g[1][k], g[0][k]) : fma(ak[k], g[1][k], -g[0][k]))
                                          : (side == 0 ? g[0][k] : -g[1][k]);
        }
#pragma unroll 1
    for (int k = 0; k < NV; ++k) {
        const double fm = zn_flux_w_d(D[1][0][k], D[1][1][k], D[1][2][k], D[1][3][k], 0.0, eps4, kappa, weights);
        gh[k] = zn_flux_w_d(D[0][0][k], D[0][1][k], D[0][2][k], D[0][3][k], fm, eps4, kappa, weights);
    }
}

// The stencil differences projected in integer arithmetic: Z/2, B and v h_0 of each difference
// vector are sums of products of the vector's mantissas and the coefficients', brought to the
// exponent of the sum's largest term at that point (so every point keeps its own relative
// accuracy; an error of 2^-55 of that term, where the double projection rounds by 2^-54 in each
// of its steps).
template <int NV>
struct WideProjection {
    // Z/2 = z0 h_0 + z1 h_1 + [z2 h_2 +] zE h_E, B = p0 h_0 + p1 h_1, shear: h_2 + w0 h_0; the
    // coefficients of h_0 (and of h_1) in Z/2 and B share an exponent
    Limbs z0, z1, z2, zE, p0, p1, w0;
    int e0, e1, e2, eE, ew;
    __device__ __forceinline__ WideProjection() : z0(0), z1(0), z2(0), zE(0), p0(0), p1(0), w0(0), e0(0), e1(0), e2(0), eE(0), ew(0) {}
    __device__ __forceinline__ explicit WideProjection(const RoeState<NV>& R)
        : z0(0), z1(0), z2(0), zE(0), p0(0), p1(0), w0(0), e2(0), ew(0) {
        int a, b;
        const int64_t c0 = wide_unpack(R.hb2, a), b0 = wide_unpack(R.hrc * R.u, b);
        e0 = max_i(a, b);
        z0 = Limbs(shr_s64(c0, e0 - a));
        p0 = Limbs(shr_s64(b0, e0 - b));
        const int64_t c1 = wide_unpack(-R.hb1 * R.u, a), b1 = wide_unpack(-R.hrc, b);
        e1 = max_i(a, b);
        z1 = Limbs(shr_s64(c1, e1 - a));
        p1 = Limbs(shr_s64(b1, e1 - b));
        zE = Limbs(wide_unpack(R.hb1, eE));
        if (NV == 4) {
            z2 = Limbs(wide_unpack(-R.hb1 * R.v, e2));
            w0 = Limbs(wide_unpack(-R.v, ew));
        }
    }
    // D[k] 2^(G[k] - 1082), |D[k]| < 2^60, of the vector at index i of the mantissa planes pl and
    // exponent planes ex; xm: running maximum of the exponents
    __device__ __forceinline__ void apply(const int64_t* pl, const uint32_t* ex, int NC, int i, int64_t* D, int* G,
                                          uint32_t& xm) const {
        const uint32_t xa = ex[i], xb = ex[NC + i];
        xm = __vimax3_u16x2(xm, xa, xb);
        const int x0 = int(xa & 0xffffu), x1 = int(xa >> 16), x2 = int(xb & 0xffffu);
        const int xE = NV == 4 ? int(xb >> 16) : x2;
        const int64_t h0 = pl[i], h1 = pl[NC + i], h2 = NV == 4 ? pl[2 * NC + i] : 0, hE = pl[(NV - 1) * NC + i];
        // a term's exponent, as of the double of its largest value (+ 1022)
        const int t0 = e0 + x0, t1 = e1 + x1, tE = eE + xE, t2 = NV == 4 ? e2 + x2 : 0;
        const int t = max_i(max_i(t0, t1), max_i(t2, tE));
        const Limbs l0(shr_s64(h0, t - t0)), l1(shr_s64(h1, t - t1)), lE(shr_s64(hE, t - tE));
        int64_t zm = wide_mul(z0.h, l0.h) + wide_mul(z1.h, l1.h) + wide_mul(zE.h, lE.h);
        int64_t zc = wide_mul(z0.h, l0.l) + wide_mul(z0.l, l0.h) + wide_mul(z1.h, l1.l) + wide_mul(z1.l, l1.h) +
                     wide_mul(zE.h, lE.l) + wide_mul(zE.l, lE.h);
        if (NV == 4) {
            const Limbs l2(shr_s64(h2, t - t2));
            zm += wide_mul(z2.h, l2.h);
            zc += wide_mul(z2.h, l2.l) + wide_mul(z2.l, l2.h);
        }
        const int64_t Z = zm + (zc >> 32);                               // units 2^(g - 1082)
        const int64_t B = wide_mul(p0.h, l0.h) + wide_mul(p1.h, l1.h) +
                          ((wide_mul(p0.h, l0.l) + wide_mul(p0.l, l0.h) + wide_mul(p1.h, l1.l) +
                            wide_mul(p1.l, l1.h)) >> 32);
        const int g = t - 1018;
        D[0] = Z + B;
        D[NV - 1] = Z - B;
        G[0] = G[NV - 1] = g;
        // h_0 - 2 Z/2 at its own scale
        const int gu = max_i(g + 2, x0 + 1);
        D[1] = shr_s64(h0, gu - x0) - (shr_s64(Z, gu - g) << 1);
        G[1] = gu;
        if (NV == 4) {
            const int gp = ew + x0 - 1018, gw = max_i(gp + 1, x2 + 1);  // w0 h_0 / 2^64 in units 2^(gp - 1082)
            const Limbs m0(h0);
            const int64_t P = wide_mul(w0.h, m0.h) + ((wide_mul(w0.h, m0.l) + wide_mul(w0.l, m0.h)) >> 32);
            D[2] = shr_s64(h2, gw - x2) + shr_s64(P, gw - gp);
            G[2] = gw;
        }
    }
};

// The interface flux where every field's weights are close to the optimal ones; false where that
// is not shown.  With the optimal weights the reconstruction is the same linear combination
// in every field, and R L = 1 takes the projection out: F^ = h+_2 + h-_3 + lin(dh+) - lin(dh-)
// per component, lin = (2 D1 - 11 D2 - 24 D3 + 3 D4)/60, sums of integers here, without an FP64
// Roe state.  What the fields add to it, R times the sum of their
//   Delta = sum c_k r_k (g_k - lin) / (1 + sum c_k r_k)   (wide_linear),
// is evaluated in float with float eigenvectors: each field's D2, D3, their difference, the
// second differences delta_0, delta_1 and d4 are projections of vectors differenced exactly in
// integers, so each is off by at most rel times the sum M of its own projection's terms (rel
// from the coefficients: 2^-19, more where c^2 is a small difference of H and u^2/2).  The
// errors of r and of Delta follow from these, and the interface is accepted if they stay below
// 2^-57 of every field's value.  Smooth data of some 40 cells a wave pass.
//
// Units.  Velocities are taken in units of 2^q, 2^(2q) the scale of H, and a difference of the
// momenta's fluxes in units 2^q, of the energy's 2^(2q) times larger than the mass flux's, so
// u, c, H and every field are of order one or less whatever the units of the data.  A small
// float counts as proof only where nothing it came from can have been rounded away: variables
// more than 2^126 below the largest enter with their scale raised to that (an error below 2^-120
// in every magnitude), and a field's r is used only where every 1/b_k is below 2^84, with 2^-62
// added to its error: products that fall below the float range then move r by less, and so does
// R, held at 2^100 from there on (r < 4 (K d4)^2 / R there).  Elsewhere Delta counts as
// unknown, |Delta| <= 0.34 (|delta_0| + |delta_1|) whatever the weights.
template <int NV>
struct FieldMagnitudes {                     // sums of the projections' terms: acoustic, entropy, shear
    float a, e, s;
    __device__ __forceinline__ FieldMagnitudes(const float* w, float hb1, float hrc, float um, float vm) {
        float z = fmaf(um, um, vm * vm) * w[0];
        z = fmaf(um, w[1], z + w[NV - 1]);
        if (NV == 4) z = fmaf(vm, w[2], z);
        z *= hb1;
        a = fmaf(hrc, fmaf(um, w[0], w[1]), z);
        e = fmaf(2.0f, z, w[0]);
        s = NV == 4 ? fmaf(vm, w[0], w[2]) : 0.0f;
    }
    __device__ __forceinline__ float of(int k) const { return k == 0 || k == NV - 1 ? a : (k == 1 ? e : s); }
};

// The float evaluation behind it, for the fields k0 <= k < k1.  ADJ: whether the flux is the optimal
// linear combination to rounding with all its first derivatives (the adjoint's use): Delta
// below 2^-54 of the value and sum_i |d Delta / d D_i| below 2^-53, from
//   |dr| <= r (2 |dQ/Q| + 2 |dT/T| + 2 |dh/h| + |db/b|), |dQ| <= 8, |dT| <= 100 F, |dh|, |db| <= 50 F
// summed over the stencil, F its largest difference, in Delta's derivative 0.07 A |dr| + 2 r.
template <int NV, bool ADJ>
struct NearLinear {
    int X[4], E, q;                            // the variables' exponents over both sides' vectors; the units' (below)
    int64_t S[NV];                             // 60 (lin(dh+) - lin(dh-)) per component, 2^(X_k - 1078)
    float dl[NV];                              // 60 Delta of the fields, plus side - minus side, 2^(E - 1022) (shear: times 2^q)
    float val[2];                              // 2^-57 of the fields' values in the same units
    float u, v, H, c2, rc, hq2;                // the Roe state in units of 2^q
    bool ok;

    __device__ __forceinline__ NearLinear(const CellPlanes<NV>& s, int base, int stride, double gm1,
                                          const WideConst& wc, int k0, int k1) {
        const int NC = s.NC, cl = base + 2 * stride, cr = cl + stride;
        // the variables' exponents over both sides' vectors
        uint32_t xa = 0, xb = 0;
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            const int i = base + st * stride;
            xa = __vimax3_u16x2(xa, s.ex[i], s.ex[2 * NC + i + stride]);
            xb = __vimax3_u16x2(xb, s.ex[NC + i], s.ex[3 * NC + i + stride]);
        }
        X[0] = int(xa & 0xffffu);
        X[1] = int(xa >> 16);
        X[2] = int(xb & 0xffffu);
        X[3] = int(xb >> 16);
        // the unit of velocity 2^q from the larger H; variables' exponents in units of 1, 2^q, 2^(2q)
        q = (max_i(exponent_of(s.H[cl]), exponent_of(s.H[cr])) - 1023) >> 1;
        ok = unsigned(q + 400) < 800u;
        int Y[NV];
        E = -4096;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            Y[k] = X[k] == 0 ? -8192 : X[k] - (k == 0 ? 0 : (k == NV - 1 ? 2 * q : q));
            E = max_i(E, Y[k]);
            // (infinities, NaN; differences whose linear part would leave the normal range)
            ok = ok && (X[k] == 0 || unsigned(X[k] - 64) < unsigned(kWideMaxExp - 64));
        }
        // powers of two of the variables against the largest
        float sc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) sc[k] = bits_float(uint32_t(max_i(Y[k] - E + 127, 1)) << 23);
        // the Roe state in float
        const float sl = wide_truncate(s.sr[cl]), wl = sl * float_rcp(sl + wide_truncate(s.sr[cr]));
        const float ul = wide_scaled(s.un[cl], q), ur = wide_scaled(s.un[cr], q);
        const float vl = NV == 4 ? wide_scaled(s.ut[cl], q) : 0.0f, vr = NV == 4 ? wide_scaled(s.ut[cr], q) : 0.0f;
        const float Hl = wide_scaled(s.H[cl], 2 * q), Hr = wide_scaled(s.H[cr], 2 * q);
        u = fmaf(wl, ul - ur, ur);
        v = fmaf(wl, vl - vr, vr);
        H = fmaf(wl, Hl - Hr, Hr);
        const float um = fabsf(ul) + fabsf(ur), vm = fabsf(vl) + fabsf(vr);
        const float g1 = wide_truncate(gm1);
        hq2 = 0.5f * fmaf(u, u, v * v);
        c2 = g1 * (H - hq2);
        rc = rsqrtf(c2);
        const float hrc = 0.5f * rc, hb1 = 0.5f * g1 * rc * rc, hb2 = hq2 * hb1;
        const float rel = 0x1p-21f * fmaf(2.0f * hb1, fabsf(H), 4.0f);
        // R in the units of the fields' squares (density's and shear's), 0 below 2^-126
        float R[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int er = wc.eR - 57 - 2 * (m == 0 ? E : E + q);
            R[m] = er < -126 ? 0.0f : wc.Rf * bits_float(uint32_t((er > 100 ? 100 : er) + 127) << 23);
        }
        const int e0 = max_i(exponent_of(s.hp[cl]), exponent_of(s.hm[cr]));
        const int ew = NV == 4 ? max_i(exponent_of(s.hp[2 * NC + cl]), exponent_of(s.ut[cl]) + e0 - 1024) - q : 0;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int ef = (m == 0 ? e0 - 2 : ew) - E + 126;
            val[m] = 0x1p-57f * bits_float(uint32_t(ef < 0 ? 0 : (ef > 250 ? 250 : ef)) << 23);
        }
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            S[k] = 0;
            dl[k] = 0.0f;
        }
        // (a thread whose interface is refused is done: warps at fronts and in rough data leave early)
#pragma unroll 1
        for (int side = 0; side < 2 && ok; ++side) {
            const int64_t* pl = side == 0 ? s.dp : s.dm;
            const uint32_t* ex = s.ex + 2 * side * NC;
            const int step = side == 0 ? stride : -stride;
            const int i0 = side == 0 ? base : base + 4 * stride;
            // the vectors D2, D2 - D3, delta_0, delta_1 (floats, variable units against 2^E)
            float w[4][NV];
            uint32_t da[4], db[4];
#pragma unroll
            for (int st = 0; st < 4; ++st) {
                da[st] = xa - ex[i0 + st * step];
                db[st] = xb - ex[NC + i0 + st * step];
            }
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                int64_t x[4];
#pragma unroll
                for (int st = 0; st < 4; ++st) {
                    const uint32_t d = k < 2 ? da[st] : db[st];
                    x[st] = shr_s64(pl[k * NC + i0 + st * step], int((k & 1) ? d >> 16 : d & 0xffffu) + 4);
                }
                const int64_t t = 2 * x[0] - 11 * x[1] - 24 * x[2] + 3 * x[3];
                S[k] += side == 0 ? t : -t;
                const int64_t s1 = x[1] - x[2], d0 = (x[0] - x[1]) - s1, d1 = s1 - (x[2] - x[3]);
                w[0][k] = wide_float(x[1]) * sc[k];
                w[1][k] = wide_float(s1) * sc[k];
                w[2][k] = wide_float(d0) * sc[k];
                w[3][k] = wide_float(d1) * sc[k];
            }
            float P[4][NV];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float* h = w[q];
                const float W = fmaf(u, h[1], NV == 4 ? fmaf(v, h[2], -h[NV - 1]) : -h[NV - 1]);
                const float Z = fmaf(hb2, h[0], -(hb1 * W)), B = hrc * fmaf(u, h[0], -h[1]);
                P[q][0] = Z + B;
                P[q][NV - 1] = Z - B;
                P[q][1] = fmaf(-2.0f, Z, h[0]);
                if (NV == 4) P[q][2] = fmaf(-v, h[0], h[2]);
            }
            // magnitudes of the projections' terms, of D2 and D3, their difference and the delta's
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                w[1][k] = fabsf(w[1][k]);
                w[0][k] = 2.0f * fabsf(w[0][k]) + w[1][k];
                w[2][k] = fabsf(w[2][k]) + fabsf(w[3][k]);
            }
            const FieldMagnitudes<NV> Mf(w[0], hb1, hrc, um, vm), Ms(w[1], hb1, hrc, um, vm), Md(w[2], hb1, hrc, um, vm);
            // (a rolled loop: the code of the interface phases is larger than the instruction cache's
            // first level as it is)
#pragma unroll 1
            for (int k = k0; k < k1 && ok; ++k) {
                float f2 = P[0][0], s1 = P[1][0], d0 = P[2][0], d1 = P[3][0];
#pragma unroll
                for (int m = 1; m < NV; ++m) {
                    f2 = k == m ? P[0][m] : f2;
                    s1 = k == m ? P[1][m] : s1;
                    d0 = k == m ? P[2][m] : d0;
                    d1 = k == m ? P[3][m] : d1;
                }
                const float f3 = f2 - s1, s0 = s1 + d0, s2 = s1 - d1, Q = d0 - d1;
                const float A = fabsf(d0) + fabsf(d1), As = fabsf(s0) + fabsf(s2), Af = fabsf(f2) + fabsf(f3);
                const float ef = fmaf(rel, Mf.of(k), 0x1p-120f);
                const float es = fmaf(rel, Ms.of(k), fmaf(0x1p-22f, Af, 0x1p-120f));
                const float ed = fmaf(rel, Md.of(k), fmaf(0x1p-22f, A, 0x1p-120f));
                const float Rk = R[NV == 4 && k == 2 ? 1 : 0];
                const float b0 = fmaf(4.0f * s0, s0, fmaf(3.0f * f2, f2 - s0, Rk)), b1 = fmaf(4.0f * s1, s1, fmaf(3.0f * f2, f3, Rk));
                const float b2 = fmaf(4.0f * s2, s2, fmaf(3.0f * f3, f3 + s2, Rk));
                const float T = fabsf(fmaf(4.0f * Q + 8.0f * d1, s0 + s2, 3.0f * fmaf(f3, d1, -(f2 * d0)))) + Rk;
                // (an error common to D2 and D3 enters f3 delta_1 - f2 delta_0 with delta_1 - delta_0 only)
                const float ET = fmaf(ed, fmaf(8.0f, As + A, 6.0f * Af), fmaf(3.0f * ef, fabsf(Q) + ed, 11.0f * A * es));
                const float i0f = float_rcp(b0), i1f = float_rcp(b1), i2f = float_rcp(b2), im = fmaxf(fmaxf(i0f, i1f), i2f);
                // relative error of the b's, from their derivatives by the two differences
                const float F1 = f2 + s0, F4 = f3 - s2;
                const float g0 = (fabsf(fmaf(8.0f, F1, -11.0f * f2)) + fabsf(fmaf(20.0f, f2, -11.0f * F1))) * i0f;
                const float g1 = (fabsf(fmaf(8.0f, f2, -5.0f * f3)) + fabsf(fmaf(8.0f, f3, -5.0f * f2))) * i1f;
                const float g2 = (fabsf(fmaf(20.0f, f3, -11.0f * F4)) + fabsf(fmaf(8.0f, F4, -11.0f * f3))) * i2f;
                const float rho = 2.0f * (ef + es + ed) * fmaxf(fmaxf(g0, g1), g2);
                const float x = wc.Kf * float_rcp(fminf(b0, b2) - 0.5f * Rk);
                const float z = x * Q * T, rr = z * z;
                // r's error (x, im: b's and h to within rho < 1/8; d4 to within 2 ed)
                const float za = fabsf(z), ze = fabsf(x) * fmaf(fabsf(Q) + 2.0f * ed, ET, 2.0f * ed * T);
                const float err = fmaf(2.0f * im, fmaf(ze, fmaf(2.0f, za, ze), rr * fmaf(8.0f, rho, 0x1p-13f)), 0x1p-62f);
                const bool known = rho < 0.125f && im <= 0x1p84f;
                const float r0 = rr * i0f, r1 = 6.0f * rr * i1f, r2 = 3.0f * rr * i2f;
                const float num = fmaf(r0, fmaf(18.0f, d0, -3.0f * d1),
                                       fmaf(r1, fmaf(-2.0f, d0, -3.0f * d1), r2 * fmaf(-2.0f, d0, 7.0f * d1)));
                const bool zero = Mf.of(k) + Md.of(k) == 0.0f;
                const float del = zero || !known ? 0.0f : num * float_rcp(10.0f + (r0 + r1 + r2));
                // |error of Delta| <= 0.07 (A + 2 ed) err + rounding of Delta and of R Delta
                const float bound = fmaf(A + 2.0f * ed, known ? fminf(0.125f * err, 0.34f) : 0.34f,
                                         0x1p-22f * fabsf(del) + rel * fabsf(del));
                const float vk = NV == 4 && k == 2 ? val[1] : val[0];
                ok = ok && (zero || bound <= vk);
                if (ADJ) {
                    const float xb = 2.0f * fabsf(x) * (T + ET), qb = xb * (fabsf(Q) + 2.0f * ed), rb = 2.0f * qb * qb * im;
                    const float F = Af + As + A, B = 0.07f * A * im * (xb * qb * 32.0f + qb * qb * F * 400.0f * float_rcp(T + ET) +
                                                                       rb * F * 300.0f) + 2.0f * rb;
                    ok = ok && (zero || (known && B <= 0x1p-53f && fabsf(del) <= 480.0f * vk));
                }
                const float sd = side == 0 ? del : -del;
#pragma unroll
                for (int m = 0; m < NV; ++m) dl[m] += k == m ? sd : 0.0f;
            }
        }
    }
};

template <int NV>
__device__ __forceinline__ bool interface_linear(const CellPlanes<NV>& s, int base, int stride, double gm1,
                                                 const WideConst& wc, double* Fh) {
    const NearLinear<NV, false> L(s, base, stride, gm1, wc, 0, NV);
    if (!L.ok) return false;
    const int NC = s.NC, cl = base + 2 * stride, cr = cl + stride;
#pragma unroll
    for (int k = 0; k < NV; ++k)
        Fh[k] = (s.hp[k * NC + cl] + s.hm[k * NC + cr]) + (L.X[k] == 0 ? 0.0 : wide_sixtieth(L.S[k], L.X[k]));
    // R Delta, where it reaches the last places of the fluxes
    bool add = false;
#pragma unroll
    for (int k = 0; k < NV; ++k) add = add || fabsf(L.dl[k]) > 2.0f * L.val[NV == 4 && k == 2 ? 1 : 0];
    if (add) {
        const float c = L.c2 * L.rc, t = L.dl[0] + L.dl[NV - 1], d = L.dl[NV - 1] - L.dl[0], f = t + L.dl[1];
        float dF[NV];
        dF[0] = f;
        dF[1] = fmaf(L.u, f, c * d);
        if (NV == 4) dF[2] = fmaf(L.v, f, L.dl[2]);
        dF[NV - 1] = fmaf(L.H, t, fmaf(L.u * c, d, fmaf(L.hq2, L.dl[1], NV == 4 ? L.v * L.dl[2] : 0.0f)));
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            // dF 2^(E - 1022) / 60 in the variable's units as a double, from the bits of dF/60
            const uint32_t b = float_bits(dF[k] * (1.0f / 60.0f));
            const int e = int((b >> 23) & 0xffu), ex = e + L.E - 126 + (k == 0 ? 0 : (k == NV - 1 ? 2 * L.q : L.q));
            if (e != 0 && unsigned(ex - 1) < 2046u)
                Fh[k] += bits_double(join((b & 0x80000000u) | (((b & 0x7fffffu) >> 3) + (uint32_t(ex) << 20)), b << 29));
        }
    }
    return true;
}

// The interface flux.  GEN 0: WENO-ZN on the split fluxes of global Lax-Friedrichs; 1: any weight
// function on the split fluxes the planes hold (global LF, Steger-Warming); 2: the planes
// hold F/2 and U/2 and each field is split with its own speed after the projection,
// g+-_c = l.F_c/2 +- a_k l.U_c/2, a_k = alpha_f[kind of field k] (split 1; kinds 0 u-c, 1 u, 2
// u+c) or the largest |u_n| + c of the six cells (split 2).  The planes dh+- must be filled.
template <int NV, int GEN>
__device__ __forceinline__ void interface_flux(const CellPlanes<NV>& s, int base, int stride, double gm1,
                                               const WideConst& wc, double eps4, double kappa, int weights, int split,
                                               const double* alpha_f, double* Fh) {
    constexpr int W = GEN == 0 ? 0 : -1;
    if (NV == 1) {
        Fh[0] = zn_split_flux<W>(s.hp[base], s.hp[base + stride], s.hp[base + 2 * stride],
                                 s.hp[base + 3 * stride], s.hp[base + 4 * stride],
                                 s.hm[base + stride], s.hm[base + 2 * stride], s.hm[base + 3 * stride],
                                 s.hm[base + 4 * stride], s.hm[base + 5 * stride], wc, eps4, kappa,
                                 GEN == 0 ? 0 : weights);
        return;
    }
    const int NC = s.NC, cl = base + 2 * stride;
    const RoeState<NV> R(s, cl, cl + stride, gm1);
    double ak[NV];
    int64_t xk[NV];
    int ek[NV];
    int ebl = 0;
    if (GEN == 2) {
        if (split == 2) {
            // (non-negative doubles order like their bit patterns)
            long long m = __double_as_longlong(s.sp[base]);
#pragma unroll
            for (int st = 1; st < 6; ++st) m = max(m, __double_as_longlong(s.sp[base + st * stride]));
#pragma unroll
            for (int k = 0; k < NV; ++k) ak[k] = __longlong_as_double(m);
        } else {
            ak[0] = alpha_f[0];
            ak[1] = alpha_f[1];
            if (NV == 4) ak[2] = alpha_f[1];
            ak[NV - 1] = alpha_f[2];
        }
#pragma unroll
        for (int k = 0; k < NV; ++k) xk[k] = wide_unpack(ak[k], ek[k]);
        ebl = exponent_of(s.hm[cl]) + ek[0] - 1024;            // |a U/2|, U the density
    }
    // scales of the fields' values (the centre's terms), below which an error does not count:
    // for the fields of the density's dimension h+-_0 (h+_0 > c rho / 2 for Lax-Friedrichs)
    const int eb0 = GEN == 0 ? exponent_of(s.hp[cl]) : max_i(max_i(exponent_of(s.hp[cl]), ebl),
                                                             GEN == 1 ? exponent_of(s.hm[cl + stride]) : 0);
    const int ebw = NV == 4 ? max_i(exponent_of(s.hp[2 * NC + cl]), exponent_of(R.v) + eb0 - 1024) : 0;
    double gh[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) gh[k] = 0.0;
    const WideProjection<NV> P(R);
    uint32_t xm = 0;
    bool ok = true;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        int64_t D[4][NV];
        int G[4][NV];
        const int step = side == 0 ? stride : -stride;
        const int first = side == 0 ? base : base + 4 * stride;
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            if (GEN != 2) {
                P.apply(side == 0 ? s.dp : s.dm, s.ex + 2 * side * NC, NC, first + st * step, D[st], G[st], xm);
            } else {
                // plus side l.dF/2 + a_k l.dU/2, minus side its negative l.dF/2 - a_k l.dU/2
                int64_t u[NV];
                int gu[NV];
                P.apply(s.dp, s.ex, NC, first + st * step, D[st], G[st], xm);
                P.apply(s.dm, s.ex + 2 * NC, NC, first + st * step, u, gu, xm);
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    const Limbs A(xk[k]), B(u[k]);
                    const int64_t v = wide_mul(A.h, B.h) + ((wide_mul(A.h, B.l) + wide_mul(A.l, B.h)) >> 32);
                    const int gv = gu[k] + ek[k] - 1018, g = max_i(gv, G[st][k]) + 1;
                    const int64_t w = shr_s64(v, g - gv);
                    D[st][k] = shr_s64(D[st][k], g - G[st][k]) + (side == 0 ? w : -w);
                    G[st][k] = g;
                }
            }
        }
        // (rolled as interface_linear's loop, for the instruction cache: 1501 x 999 cells between walls
        // 3.06 ms a step instead of 3.12 unrolled)
#pragma unroll 1
        for (int k = 0; k < NV; ++k) {
            double corr;
            ok = wide_correction<W>(D[0][0], D[1][0], D[2][0], D[3][0], G[0][0], G[1][0], G[2][0], G[3][0],
                                    NV == 4 && k == 2 ? ebw : eb0 - 2, wc, weights, corr) && ok;
            const double g = side == 0 ? corr : gh[0] - corr;
#pragma unroll
            for (int m = 0; m + 1 < NV; ++m) {
#pragma unroll
                for (int st = 0; st < 4; ++st) {
                    D[st][m] = D[st][m + 1];
                    G[st][m] = G[st][m + 1];
                }
                gh[m] = gh[m + 1];
            }
            gh[NV - 1] = g;
        }
    }
    if (!ok || (xm & 0xffffu) == 2047u || (xm >> 16) == 2047u) {
        // out of the integer evaluation's range, infinite or not a number (copies, so that the
        // kept values need no address)
        const RoeState<NV> Rc = R;
        double gd[NV], ac[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) ac[k] = GEN == 2 ? ak[k] : 0.0;
        field_fluxes_double<NV, GEN>(s, Rc, base, stride, eps4, kappa, GEN == 0 ? 0 : weights, ac, gd);
#pragma unroll
        for (int k = 0; k < NV; ++k) gh[k] = gd[k];
    }
    double hc[NV];
    if (GEN != 2) {
#pragma unroll
        for (int k = 0; k < NV; ++k) hc[k] = s.hp[k * NC + cl] + s.hm[k * NC + cl + stride];
    } else {
        // the centres (F_2 + F_3)/2 + R diag(a_k) L (U_2 - U_3)/2
        double du[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            hc[k] = s.hp[k * NC + cl] + s.hp[k * NC + cl + stride];
            du[k] = s.hm[k * NC + cl] - s.hm[k * NC + cl + stride];
        }
        if (split == 2) {
#pragma unroll
            for (int k = 0; k < NV; ++k) hc[k] = fma(ak[k], du[k], hc[k]);
        } else {
            double gu[NV];
            R.project(du, gu);
#pragma unroll
            for (int k = 0; k < NV; ++k) gh[k] = fma(ak[k], gu[k], gh[k]);
        }
    }
    R.back_project(gh, hc, Fh);
}

}  // namespace wz
