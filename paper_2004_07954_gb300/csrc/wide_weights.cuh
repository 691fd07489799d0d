// The WENO-ZN reconstruction of wenozn_device.cuh in 64-bit integer arithmetic.
//
// Why.  GB300 issues one FP64 instruction per SM sub-partition every 64 cycles, and its 32-bit
// integer and FMA pipes one every 2: a 64 x 64-bit product of which only the top half is kept
// is three 32 x 32 multiply-adds, an addition two instructions.  A reconstruction is 46 FP64
// instructions (2,944 cycles of a sub-partition's FP64 unit) or some 650 ALU and multiply-add
// ones, on pipes that otherwise idle; where the weights hardly differ from the
// optimal ones (wide_linear) about 150 in all.  Measured with the FP64 weights before and these
// after (with the integer projection of euler_device.cuh in the solver): wenozn_reconstruct
// 1.24 -> 0.24 ms per side of 2^24 points, the 2D Euler step 99.9 -> 19.0 ms at 4096^2 and 6.5 ->
// 1.54 ms at 1024^2, the 1D step 2.63 -> 0.50 ms at 2^20 cells.
//
// Precision.  Every quantity carries a 64-bit mantissa (block floating point: integers with a
// common exponent), every truncation stays below that of a 53-bit one, so the result is
// closer to the exact value than the double evaluation's: against binary128, over 3 10^5
// stencils each, the rms error of f^ - c relative to the largest difference is 6.3e-18 on random
// differences (double 3.3e-17), 4.7e-18 on smooth data (4.7e-17), the largest 1.3e-16 and 1.1e-16
// (3.4e-16, 2.3e-16).  Nothing overflows or underflows on the way: the exponents are integers of
// their own (a result below the normal range becomes 0).
//
// Derivation, from the first differences D1..D4 of the stencil (see wenozn_device.cuh for
// the scheme).  With s_k the second differences, 3 IS_k is a binary form in the two differences
// of sub-stencil k,
//   beta_0 = 4 s_0^2 + 3 D2 (2 D2 - D1),  beta_1 = 4 s_1^2 + 3 D2 D3,  beta_2 = 4 s_2^2 + 3 D3 (2 D3 - D4),
// positive definite: 0.73 (Di^2 + Dj^2) <= beta_k <= 25 max(Di^2, Dj^2), so with Di, Dj scaled
// by the larger one's exponent beta_k is known to within six bits beforehand.  With R = 3 eps,
// b_k = beta_k + R, T = |b_0 - b_2| + R, h = min(b_0, b_2) - R/2 and K = sqrt(3 / (4 A)) the weights are
//   a_k = h^2 b_0 b_1 b_2 + (K d4 T)^2 b_i b_j   (i, j the other two),
// and f^ - c = (a_0 g_0 + 6 a_1 g_1 + 3 a_2 g_2) / (6 (a_0 + 6 a_1 + 3 a_2)) with
//   g_0 = 2 D1 - 5 D2,  g_1 = -(D2 + 2 D3),  g_2 = D4 - 4 D3.
//
// Signs.  f^ - c is odd in the differences and every step here is exactly odd or even in them:
// shifts and products drop the low bits of magnitudes, never of two's complement values.  So a
// stencil mirrored about its centre cell (D4 = -D1, D3 = -D2) has b_0 = b_2 to the last bit and
// tau5 = 0 exactly: near a flat top a last bit of tau5 alone would decide the weights.
//
// Scales.  Each D_i comes with an exponent of its own.  A sub-stencil's pair takes the scale of
// its larger difference, each weight a_k and each product a_k g_k an exponent of its own too,
// so a flat sub-stencil beside a jump keeps its full relative accuracy (the result there is
// its small difference, whatever the jump).  d4 takes the largest difference's scale.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define WZ_HD __device__ __forceinline__
#else
#define WZ_HD inline
#endif

namespace wz {

// eps and A in the form the integer evaluation takes them (host side, once per launch).
struct WideConst {
    uint64_t RM, KM;      // mantissas in [2^63, 2^64) of R = 3 eps and K = sqrt(3 / (4 A))
    int eR, eK;           // R = RM 2^(eR - 2164), K = KM 2^eK
    int e_min;            // smallest pair exponent: that of sqrt(eps)
    float Rf, Kf;         // R = Rf 2^(eR - 2101), Rf in [1, 2); K
};

inline WideConst wide_const(double eps, double A) {
    WideConst w;
    int e = 0;
    const double r = std::frexp(3.0 * eps, &e);                    // [1/2, 1)
    w.RM = uint64_t(std::ldexp(r, 53)) << 11;
    w.eR = e - 64 + 2164;
    const double k = std::frexp(std::sqrt(0.75 / A), &e);
    w.KM = uint64_t(std::ldexp(k, 53)) << 11;
    w.eK = e - 64;
    w.e_min = (w.eR - 57) >> 1;
    w.Rf = float(2.0 * r);
    w.Kf = float(std::sqrt(0.75 / A));
    return w;
}

// Differences of magnitude [2^-300, 2^400) take the integer evaluation (biased exponents).
constexpr int kWideMinExp = 1023 - 300, kWideMaxExp = 1023 + 400;

WZ_HD uint64_t shr_u64(uint64_t x, int n) {          // n >= 0, zero from 64 on
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return n > 63 ? 0 : x >> n;
#endif
}

WZ_HD int64_t shr_s64(int64_t x, int n) {            // n >= 0, the sign from 63 on
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return x >> (n > 63 ? 63 : n);
#endif
}

// x, or ~|x| of a negative x, so that shifting drops bits of the magnitude; and x >> n from it,
// toward zero
WZ_HD int64_t ones(int64_t x) { return x - int64_t(uint64_t(x) >> 63); }

WZ_HD int64_t shr_ones(int64_t o, int n) {
    const int64_t r = shr_s64(o, n);
    return r + int64_t(uint64_t(r) >> 63);
}

WZ_HD int clz_u32(uint32_t x) {                      // x > 0
#ifdef __CUDA_ARCH__
    int r;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(r) : "r"(x));
    return r;
#else
    return __builtin_clz(x);
#endif
}

WZ_HD uint32_t funnel_l(uint32_t lo, uint32_t hi, int n) {      // high word of (hi:lo) << n, 0 <= n < 32
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, n);
#else
    return n ? (hi << n) | (lo >> (32 - n)) : hi;
#endif
}

WZ_HD int max_i(int a, int b) { return a > b ? a : b; }

WZ_HD int leading_zeros4(uint64_t x) {               // of x, at most 4
    const int n = clz_u32(uint32_t(x >> 32) | 1u);
    return n < 4 ? n : 4;
}

WZ_HD uint64_t join(uint32_t hi, uint32_t lo) { return (uint64_t(hi) << 32) | lo; }

// floor(a b / 2^64), at most 2 too small
WZ_HD uint64_t mul_hi(uint64_t a, uint64_t b) {
    const uint32_t ah = uint32_t(a >> 32), al = uint32_t(a), bh = uint32_t(b >> 32), bl = uint32_t(b);
    const uint64_t x = uint64_t(al) * bh, y = uint64_t(ah) * bl;
    return uint64_t(ah) * bh + (x >> 32) + (y >> 32);
}

WZ_HD uint64_t sqr_hi(uint64_t a) {
    const uint32_t ah = uint32_t(a >> 32), al = uint32_t(a);
    return uint64_t(ah) * ah + ((uint64_t(al) * ah) >> 31);
}

// x = h 2^32 + l with a signed low limb, so that products of limbs are signed 32 x 32 ones
struct Limbs {
    int32_t h, l;
    WZ_HD Limbs(int32_t high, int32_t low) : h(high), l(low) {}
    WZ_HD explicit Limbs(int64_t x) {
        const uint32_t lo = uint32_t(x);
        l = int32_t(lo);
        h = int32_t(uint32_t(uint64_t(x) >> 32) + (lo >> 31));
    }
};

WZ_HD int64_t wide_mul(int32_t a, int32_t b) { return int64_t(a) * b; }

WZ_HD int32_t wide_mul_hi(int32_t a, int32_t b) {    // floor(a b / 2^32)
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return int32_t((int64_t(a) * b) >> 32);
#endif
}

// b_k = beta_k + R of a sub-stencil: its second difference s and the factors p w of beta's
// other part (beta = 4 s^2 + 3 p w) at the pair's scale, e its exponent: |2 s| <= 2^62,
// |3 p|, |w| <= 3 2^60.  B in [2^63, 2^64), b = B 2^eb.  (The low limbs' product counts with its
// floor, so that the sum does not depend on which way p and w were split: it is even in them.)
WZ_HD uint64_t wide_indicator(int64_t s, int64_t p, int64_t w, int e, const WideConst& c, int& eb) {
    const Limbs S(s + s), P(p + p + p), Wl(w);
    const int64_t main = wide_mul(S.h, S.h) + wide_mul(P.h, Wl.h);
    const int64_t cross = wide_mul(S.h, S.l) + wide_mul(S.h, S.l) + wide_mul(P.h, Wl.l) + wide_mul(P.l, Wl.h) + wide_mul_hi(P.l, Wl.l);
    const uint64_t m = uint64_t(main + (cross >> 32)) + shr_u64(c.RM, 64 + 2 * e - c.eR);
    const int n = clz_u32(uint32_t(m >> 32));
    eb = 2 * e + 64 - n;
    return join(funnel_l(uint32_t(m), uint32_t(m >> 32), n), funnel_l(uint32_t(cross), uint32_t(m), n));
}

// 2^127 / d for d in [2^63, 2^64), a few units too small at most: the float reciprocal and two
// Newton steps
WZ_HD uint64_t wide_rcp(uint64_t d) {
    const uint32_t dh = uint32_t(d >> 32), dl = uint32_t(d);
#ifdef __CUDA_ARCH__
    float f;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint2float_rz(dh)));
    const uint32_t r0 = __float2uint_rz(f * 9223369837831520256.0f);      // 2^63 (1 - 2^-22)
#else
    const uint32_t r0 = uint32_t((1.0f / float(dh)) * 9223369837831520256.0f);
#endif
    const uint64_t e0 = (uint64_t(1) << 63) - uint64_t(dh) * r0 - ((uint64_t(dl) * r0) >> 32);     // < 2^43
    const uint64_t r1 = (uint64_t(r0) << 32) + ((uint64_t(r0) * uint32_t(e0 >> 11)) >> 20);
    const uint32_t e1 = uint32_t((uint64_t(1) << 63) - mul_hi(d, r1));
    return r1 + ((uint64_t(uint32_t(r1 >> 32)) * e1) >> 31);
}

// A double as a signed mantissa x, |x| in [2^59, 2^60), and its biased exponent e: the value is
// x 2^(e - 1082).  Zeros and subnormals have e = 0 (a zero x = 0).  wide_unpack_ones gives ones(x)
// (of -0.0: -1, which every shift takes to 0).
WZ_HD int64_t wide_unpack_ones(double v, int& e) {
#ifdef __CUDA_ARCH__
    const uint64_t u = uint64_t(__double_as_longlong(v));
#else
    uint64_t u;
    std::memcpy(&u, &v, 8);
#endif
    const uint32_t hi = uint32_t(u >> 32), sg = uint32_t(int32_t(hi) >> 31);
    e = int((hi >> 20) & 0x7ffu);
    const uint64_t m = join((hi & 0xfffffu) | (e ? 0x100000u : 0u), uint32_t(u)) << 7;
    return int64_t(m ^ join(sg, sg));
}

WZ_HD int64_t wide_unpack(double v, int& e) {
    const int64_t o = wide_unpack_ones(v, e);
    return o + int64_t(uint64_t(o) >> 63);
}

WZ_HD int64_t shl_s64(int64_t x, int n) {            // 0 <= n < 64
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return int64_t(uint64_t(x) << n);
#endif
}

// D 2^(G - 1082), |D| <= 2^60, as x 2^(e - 1082) with |x| in [2^59, 2^60]; e = 0 for D = 0.
WZ_HD int64_t wide_normalise(int64_t D, int G, int& e) {
    const uint32_t s = uint32_t(uint64_t(D >> 63)), h = uint32_t(uint64_t(D) >> 32) ^ s, l = uint32_t(D) ^ s;
    const bool low = h == 0;
    const int n = max_i(clz_u32((low ? l : h) | 1u) + (low ? 28 : -4), 0);
    e = D == 0 ? 0 : G - n;
    return shl_s64(D, n);
}

// f^ - c from the differences x_i 2^(e_i - 1082), |x_i| in [2^59, 2^60] (or x_i = 0, e_i = 0),
// given as o_i = ones(x_i).
// weights: 0 WENO-ZN, as above; 1 WENO-Z (q = 1), a_k = b_0 b_1 b_2 + |b_0 - b_2| b_i b_j; 3
// Jiang-Shu, a_k = (b_i b_j)^2 (the linear weights, 2, are wide_linear's).
WZ_HD double wide_weighted(int64_t o0, int64_t o1, int64_t o2, int64_t o3, int e0, int e1, int e2, int e3,
                           const WideConst& c, int weights) {
    // the sub-stencils' pairs at their own scales
    const int g01 = max_i(e0, e1), g12 = max_i(e1, e2), g23 = max_i(e2, e3);
    const int E = max_i(g01, g23);
    const int64_t p0 = shr_ones(o0, g01 - e0), q0 = shr_ones(o1, g01 - e1);
    const int64_t p1 = shr_ones(o1, g12 - e1), q1 = shr_ones(o2, g12 - e2);
    const int64_t p2 = shr_ones(o2, g23 - e2), q2 = shr_ones(o3, g23 - e3);

    // the indicators; a pair below the scale of eps enters at that scale (b_k is then R to
    // within rounding, and never loses its leading bits)
    uint64_t b0, b1, b2;
    int n0, n1, n2;                                           // exponents of b_k
    {
        int64_t u0 = p0, v0 = q0, u1 = p1, v1 = q1, u2 = p2, v2 = q2;
        int h01 = g01, h12 = g12, h23 = g23;
        if (g01 < c.e_min || g12 < c.e_min || g23 < c.e_min) {
            h01 = max_i(g01, c.e_min);
            h12 = max_i(g12, c.e_min);
            h23 = max_i(g23, c.e_min);
            u0 = shr_ones(ones(u0), h01 - g01);
            v0 = shr_ones(ones(v0), h01 - g01);
            u1 = shr_ones(ones(u1), h12 - g12);
            v1 = shr_ones(ones(v1), h12 - g12);
            u2 = shr_ones(ones(u2), h23 - g23);
            v2 = shr_ones(ones(v2), h23 - g23);
        }
        b0 = wide_indicator(u0 - v0, v0, v0 + v0 - u0, h01, c, n0);
        b1 = wide_indicator(u1 - v1, u1, v1, h12, c, n1);
        b2 = wide_indicator(u2 - v2, u2, u2 + u2 - v2, h23, c, n2);
    }

    // a_k = X 2^eX + Y_k 2^(f_k), exponents relative to that of b_0 b_1 b_2
    const uint64_t b01 = mul_hi(b0, b1), b12 = mul_hi(b1, b2), b02 = mul_hi(b0, b2);
    uint64_t X = 0, Y0, Y1, Y2;
    int eX = -(1 << 20), f0, f1, f2;
    if (weights == 3) {
        Y0 = sqr_hi(b12);
        Y1 = sqr_hi(b02);
        Y2 = sqr_hi(b01);
        const int eS = n0 + n1 + n2 + 192;
        f0 = eS - 2 * n0;
        f1 = eS - 2 * n1;
        f2 = eS - 2 * n2;
    } else {
        // T = |b_0 - b_2|, normalised (zero: exponent far below), then + R: R at its own scale, since
        // on a tie T is R alone
        const bool lt = n0 < n2 || (n0 == n2 && b0 < b2);
        const uint64_t mx = lt ? b2 : b0, mn = lt ? b0 : b2;
        const int nx = lt ? n2 : n0, nn = lt ? n0 : n2;
        uint64_t T = mx - shr_u64(mn, nx - nn);
        const bool lowT = (T >> 32) == 0;
        T = lowT ? T << 32 : T;
        const int nT = clz_u32(uint32_t(T >> 32) | 1u);
        int eT = T == 0 ? -(1 << 20) : nx - (lowT ? 32 : 0) - nT;
        T <<= nT;
        if (weights == 0) {
            const int e = max_i(eT, c.eR) + 1;
            T = shr_u64(T, e - eT) + shr_u64(c.RM, e - c.eR);
            eT = e;
        }
        uint64_t Y;
        int eY;
        if (weights == 1) {
            X = mul_hi(b01, b2);
            eX = 128;
            Y = T;
            eY = eT + 128;
        } else {
            // z = K |d4| T from normalised factors (T to within a bit);
            // X = h^2 b_0 b_1 b_2 with h = min - R/2, Y = z^2
            const int64_t c1 = shr_ones(o0, E - e0), c2 = shr_ones(o1, E - e1), c3 = shr_ones(o2, E - e2),
                          c4 = shr_ones(o3, E - e3);
            const int64_t d23 = c2 - c3;
            const int64_t d4 = (c1 - c4) - (d23 + d23 + d23);
            uint64_t ad = uint64_t(d4 < 0 ? -d4 : d4);
            const bool low = (ad >> 32) == 0;
            ad = low ? ad << 32 : ad;
            const int na = clz_u32(uint32_t(ad >> 32) | 1u);
            ad <<= na;
            uint64_t z = mul_hi(mul_hi(ad, T), c.KM);
            const int nz = clz_u32(uint32_t(z >> 32) | 1u);
            z <<= nz;
            const int ez = E + eT + c.eK + 128 - na - (low ? 32 : 0) - nz;
            const uint64_t h = mn - shr_u64(c.RM, nn - c.eR + 1);
            X = mul_hi(sqr_hi(h), mul_hi(b01, b2));
            eX = 2 * nn + 256;
            Y = sqr_hi(z);
            eY = z == 0 ? -(1 << 20) : 2 * ez + 192;
        }
        Y0 = mul_hi(Y, b12);
        Y1 = mul_hi(Y, b02);
        Y2 = mul_hi(Y, b01);
        f0 = eY - n0;
        f1 = eY - n1;
        f2 = eY - n2;
    }
    // a_k below 2^61 with the exponent of its larger term's leading bit (at most four zeros counted)
    const int tX = eX - leading_zeros4(X);
    const int m0 = max_i(tX, f0 - leading_zeros4(Y0)) + 4;
    const int m1 = max_i(tX, f1 - leading_zeros4(Y1)) + 4;
    const int m2 = max_i(tX, f2 - leading_zeros4(Y2)) + 4;
    // with the optimal weights 1 : 6 : 3
    const uint64_t a0 = shr_u64(X, m0 - eX) + shr_u64(Y0, m0 - f0);
    const uint64_t a1 = (shr_u64(X, m1 - eX) + shr_u64(Y1, m1 - f1)) * 6;
    const uint64_t a2 = (shr_u64(X, m2 - eX) + shr_u64(Y2, m2 - f2)) * 3;

    // numerator: products a_k g_k / 2^64, each with its own exponent, summed at the largest
    // (|g_k| <= 7 2^60, 3 2^60, 5 2^60: the sum stays below 2^62.4)
    auto product = [](uint64_t a, int64_t g, int n) {
        const int32_t s = int32_t(uint64_t(g) >> 32) >> 31;
        const int64_t m = int64_t(shr_u64(mul_hi(a, uint64_t((g + s) ^ s)), n));
        return (m ^ s) - s;
    };
    const int k0 = m0 + g01, k1 = m1 + g12, k2 = m2 + g23, km = max_i(max_i(k0, k1), k2);
    const int64_t S = product(a0, p0 + p0 - 5 * q0, km - k0) - product(a1, p1 + q1 + q1, km - k1) +
                      product(a2, q2 - 4 * p2, km - k2);
    // denominator
    const int dm = max_i(max_i(m0, m1), m2);
    uint64_t d = (shr_u64(a0, dm + 2 - m0) + shr_u64(a1, dm + 2 - m1) + shr_u64(a2, dm + 2 - m2)) * 3;
    const int nd = clz_u32(uint32_t(d >> 32));
    d <<= nd;
    // |S|, normalised, times the reciprocal
    const uint32_t sign = uint32_t(uint64_t(S) >> 32) & 0x80000000u;
    uint64_t N = uint64_t(S < 0 ? -S : S);
    const bool up = (N >> 32) == 0;
    N = up ? N << 32 : N;
    const int nt = clz_u32(uint32_t(N >> 32) | 1u);
    uint64_t q = mul_hi(N << nt, wide_rcp(d));
    const int nq = clz_u32(uint32_t(q >> 32) | 1u);
    q <<= nq;
    // round to 53 bits; a carry out of the mantissa raises the exponent by itself
    const uint64_t r = ((q >> 10) + 1) >> 1;
    // (an exponent below the normal range: every product of weight vanished against a flat pair's)
    const int ex = km - dm + 1 - nt - (up ? 32 : 0) + nd - nq;
    const uint64_t bits = N == 0 || ex < 0 ? 0 : r + join((uint32_t(ex) << 20) | sign, 0);
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)bits);
#else
    double corr;
    std::memcpy(&corr, &bits, 8);
    return corr;
#endif
}

WZ_HD float bits_float(uint32_t b) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    std::memcpy(&f, &b, 4);
    return f;
#endif
}

WZ_HD uint32_t float_bits(float f) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(f);
#else
    uint32_t b;
    std::memcpy(&b, &f, 4);
    return b;
#endif
}

WZ_HD int exponent_of(double v) {                    // biased
#ifdef __CUDA_ARCH__
    return (__double2hiint(v) >> 20) & 0x7ff;
#else
    uint64_t u;
    std::memcpy(&u, &v, 8);
    return int(u >> 52) & 0x7ff;
#endif
}

WZ_HD float float_rcp(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;
#endif
}

WZ_HD float wide_float(int64_t x) {                  // x 2^-56 to 24 bits
    const Limbs l(x);
    return fmaf(float(l.h), 0x1p-24f, float(l.l) * 0x1p-56f);
}

WZ_HD uint64_t double_bits(double v) {
#ifdef __CUDA_ARCH__
    return uint64_t(__double_as_longlong(v));
#else
    uint64_t u;
    std::memcpy(&u, &v, 8);
    return u;
#endif
}

WZ_HD double bits_double(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double v;
    std::memcpy(&v, &u, 8);
    return v;
#endif
}

// x / 2 (exact) on the exponent field; by multiplication only where that underflows
WZ_HD double wide_half(double x) {
    const uint64_t u = double_bits(x);
    const uint32_t e = uint32_t(u >> 52) & 0x7ffu;
    if (e - 2u < 2045u) return bits_double(u - (uint64_t(1) << 52));
    return (u << 1) == 0 ? x : 0.5 * x;
}

// 1 / x of a positive normal x below 2^1021, rounded to 53 bits from an error below 2^-60
WZ_HD double wide_reciprocal(double x) {
    const uint64_t u = double_bits(x);
    const uint64_t r = wide_rcp((u << 11) | (uint64_t(1) << 63));
    return bits_double((((r >> 10) + 1) >> 1) + (uint64_t(2044 - int(u >> 52)) << 52));
}

// 1 / sqrt(x) of a positive normal x: the float approximation Y0 of y = 1/sqrt(t), t in [1/4, 1)
// the mantissa with an even exponent, and one step of Householder's third-order iteration,
// y = y0 (1 + h/2 + 3/8 h^2 + ...), h = 1 - t y0^2 < 2^-19 in units of 2^-62, so the truncated terms
// are below 2^-59 and the result is within 2^-59 before its rounding to 53 bits.  Where x is not
// positive and normal: ok = false.
WZ_HD double wide_rsqrt(double x, bool& ok) {
    const uint64_t u = double_bits(x);
    const int e = int(u >> 52);                                // the sign included
    ok = unsigned(e - 1) < 2046u;
    const uint64_t m = ((u << 11) | (uint64_t(1) << 63)) >> ((e & 1) ? 1 : 0);   // t = m / 2^64
#ifdef __CUDA_ARCH__
    float f;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint2float_rz(uint32_t(m >> 32))));
    const uint32_t y0 = __float2uint_rz(f * 140737421246464.0f);         // 2^47 (1 - 2^-21)
#else
    const uint32_t y0 = uint32_t((1.0f / std::sqrt(float(uint32_t(m >> 32)))) * 140737421246464.0f);
#endif
    const uint64_t hh = (uint64_t(1) << 62) - mul_hi(m, uint64_t(y0) * y0);
    const uint64_t h = hh > 2 ? hh - 2 : 0;
    const uint32_t hs = uint32_t(h >> 12);
    const uint64_t q = h + ((uint64_t(uint32_t((uint64_t(hs) * hs) >> 32)) * 3) >> 8);
    const uint64_t y = (uint64_t(y0) << 32) + ((uint64_t(y0) * uint32_t(q)) >> 31) + ((uint64_t(y0) * uint32_t(q >> 32)) << 1);
    // x = t 2^(e - 1022) with e odd after the shift's adjustment: y 2^((1022 - e') / 2)
    const int ee = e + (e & 1);                                // even exponent field of t
    return bits_double((((y >> 10) + 1) >> 1) + (uint64_t(1022 - ((ee - 1022) >> 1)) << 52));
}

// S 2^(G - 1078) / 60 as a double, |S| < 2^63
WZ_HD double wide_sixtieth(int64_t S, int G) {
    const uint32_t sign = uint32_t(uint64_t(S) >> 32) & 0x80000000u;
    uint64_t N = uint64_t(S < 0 ? -S : S);
    const bool up = (N >> 32) == 0;
    N = up ? N << 32 : N;
    const int nt = clz_u32(uint32_t(N >> 32) | 1u);
    uint64_t q = mul_hi(N << nt, 9838263505978427528ull);     // 2^69 / 60
    const int nq = clz_u32(uint32_t(q >> 32) | 1u);
    q <<= nq;
    const uint64_t r = ((q >> 10) + 1) >> 1;
    const int ex = G + 2 - nt - (up ? 32 : 0) - nq;           // (below 0: below the normal range)
    return bits_double(N == 0 || ex < 0 ? 0 : r + join((uint32_t(ex) << 20) | sign, 0));
}

// A double to float by truncation of its bits; not a number outside [2^-126, 2^127) but for 0.
WZ_HD float wide_truncate(double v) {
    const uint64_t u = double_bits(v);
    const uint32_t hi = uint32_t(u >> 32), a = (hi & 0x7fffffffu) - (897u << 20);
    const uint32_t f = funnel_l(uint32_t(u), a + (1u << 20), 3) | (hi & 0x80000000u);
    return bits_float(a < (253u << 20) ? f : ((u << 1) == 0 ? 0u : 0x7fffffffu));
}

// v 2^-n as a float by truncation, |n| < 897; 0 below 2^-126, not a number from 2^127 on
WZ_HD float wide_scaled(double v, int n) {
    const uint64_t u = double_bits(v);
    const uint32_t hi = uint32_t(u >> 32), a = (hi & 0x7fffffffu) - (uint32_t(897 + n) << 20);
    const uint32_t f = funnel_l(uint32_t(u), a + (1u << 20), 3) | (hi & 0x80000000u);
    return bits_float(a < (253u << 20) ? f : (int32_t(a) < 0 ? 0u : 0x7fffffffu));
}

// f^ - c where the weights hardly differ from the optimal ones; false where that is not shown.
// With r_k = (K d4 T)^2 / (h^2 b_k) the weights are c_k (1 + r_k) (the other weight functions alike
// with their own r_k), so f^ - c is the optimal
// linear combination of the differences, formed exactly in integers, plus
//   sum c_k r_k (g_k - lin) / (1 + sum c_k r_k),
// a combination of the second differences delta_0 = D1 - 2 D2 + D3 and delta_1 = D2 - 2 D3 + D4.
// This part is evaluated in float from integers (each converted with 24 bits of its own: T is
// formed from the delta's, without the cancellation in b_0 - b_2), and accepted only where the
// bound on its error, from the bound ET on T's, is below 2^-56 of the differences and the value
// they are added to: a quarter of a last place of the result.  Smooth data resolved by some 30
// cells a wave are accepted (r falls like the twelfth power of the spacing), as are constant
// data and differences at the rounding level of the value itself.  2^(eb - 1023) bounds that
// value from below (eb <= 0: nothing is known of it).
// About 150 instructions instead of 600 for a warp whose lanes are all accepted.
// ODD: the differences come as ones(D_i), as wide_weighted's, for a result exactly odd in them;
// else as D_i, rounded down (the bound holds either way).
template <bool ODD>
WZ_HD bool wide_linear(int64_t o1, int64_t o2, int64_t o3, int64_t o4, int G1, int G2, int G3, int G4, int eb, const WideConst& c, int weights, double& corr) {
    const int G = max_i(max_i(G1, G2), max_i(G3, G4));
    auto shifted = [](int64_t o, int n) { return ODD ? shr_ones(o, n) : shr_s64(o, n); };
    const int64_t c1 = shifted(o1, G - G1 + 4), c2 = shifted(o2, G - G2 + 4);      // |c_i| <= 2^56
    const int64_t c3 = shifted(o3, G - G3 + 4), c4 = shifted(o4, G - G4 + 4);
    const int64_t c12 = c1 - c2, c23 = c2 - c3, c34 = c3 - c4, d0 = c12 - c23, d1 = c23 - c34;
    const float f2 = wide_float(c2), f3 = wide_float(c3), S1 = wide_float(c23), E0 = wide_float(d0),
                E1 = wide_float(d1), Q = wide_float(d0 - d1);
    const float S0 = S1 + E0, S2 = S1 - E1;
    const int er = c.eR - 57 - 2 * G;                         // R in the floats' units
    const float R = c.Rf * bits_float(uint32_t((er < -126 ? -126 : (er > 60 ? 60 : er)) + 127) << 23);
    const float be0 = fmaf(4.0f * S0, S0, 3.0f * f2 * (f2 - S0)), be2 = fmaf(4.0f * S2, S2, 3.0f * f3 * (f3 + S2));
    const float be1 = fmaf(4.0f * S1, S1, 3.0f * f2 * f3);
    const float b0 = be0 + R, b1 = be1 + R, b2 = be2 + R;
    const float A = fabsf(E0) + fabsf(E1), M = fabsf(f2) + fabsf(S1) + A;
    const float T = fabsf(fmaf(4.0f * (E0 + E1), S0 + S2, 3.0f * fmaf(f3, E1, -(f2 * E0)))) + R;
    const float ET = 0x1p-18f * A * M;
    const float i0 = float_rcp(b0), i1 = float_rcp(b1), i2 = float_rcp(b2);
    const float im = fmaxf(fmaxf(i0, i1), i2);
    float r0, r1, r2, err;
    if (weights == 0) {
        const float u = c.Kf * Q * float_rcp(fminf(be0, be2) + 0.5f * R);
        const float w = (u * T) * (u * T);
        r0 = w * i0;
        r1 = w * i1;
        r2 = w * i2;
        err = fmaf(fabsf(u) * ET * im, fabsf(u) * fmaf(2.0f, T, ET), 0x1p-14f * (w * im));
    } else if (weights == 1) {
        // WENO-Z: r_k = |b_0 - b_2| / b_k
        r0 = (T - R) * i0;
        r1 = (T - R) * i1;
        r2 = (T - R) * i2;
        err = fmaf(ET, im, 0x1p-14f * (T * im));
    } else if (weights == 3) {
        // Jiang-Shu: r_k = (b_1 - b_k)(b_1 + b_k) / b_k^2, the differences of the b's from the delta's
        r0 = E0 * fmaf(3.0f, f2, -4.0f * (S0 + S1)) * (b1 + b0) * i0 * i0;
        r1 = 0.0f;
        r2 = E1 * fmaf(3.0f, f3, 4.0f * (S1 + S2)) * (b1 + b2) * i2 * i2;
        err = ET * (b0 + b1 + b2) * im * im + 0x1p-14f * (fabsf(r0) + fabsf(r2));
    } else {
        r0 = r1 = r2 = err = 0.0f;
    }
    const int ef = eb - G + 126;                              // 2^(eb - 1023) in the floats' units
    const float fb = bits_float(uint32_t(ef < 0 ? 0 : (ef > 250 ? 250 : ef)) << 23);
    if (!(A * err <= 0x1p-53f * (fabsf(f2) + fabsf(f3) + fb)) ||
        unsigned(G - kWideMinExp) >= unsigned(kWideMaxExp - kWideMinExp))
        return false;
    // 60 (f^ - c) = lin + sum 10 c_k r_k (10 g_k - lin) / (10 + sum 10 c_k r_k)
    r1 *= 6.0f;
    r2 *= 3.0f;
    const float num = fmaf(r0, fmaf(18.0f, E0, -3.0f * E1),
                           fmaf(r1, fmaf(-2.0f, E0, -3.0f * E1), r2 * fmaf(-2.0f, E0, 7.0f * E1)));
    const uint32_t v = float_bits(num * float_rcp(10.0f + (r0 + r1 + r2)));
    const int ve = int((v >> 23) & 0xffu);
    // (below 2^7: the float is an average of 18 delta_0 - 3 delta_1 and the like, |delta| <= 4)
    const int64_t vm = int64_t(shr_u64(join(((v & 0x7fffffu) | (ve ? 0x800000u : 0u)) << 7, 0), 133 - ve));
    const int64_t S = 2 * c1 - 11 * c2 - 24 * c3 + 3 * c4 + (int32_t(v) < 0 ? -vm : vm);
    corr = wide_sixtieth(S, G);
    return true;
}

// The weighted evaluation as a call of its own: the warps of smooth data pass it by, and one copy
// of its code serves every field (inlined four times it does not fit the instruction cache).
// The projected differences of a stencil mirrored about its centre cell (a plateau of three cells
// between equal neighbours) are so but for their truncations, five of the last places of
// D_i: within eight (2^-57 of the projection's terms, its accuracy) they are made so exactly, or
// tau5 would be noise where it is zero, and decide the weights ("Signs" above).
// W: the weight function, -1 for the run-time value.
template <int W>
#ifdef __CUDACC__
static __device__ __noinline__
#else
inline
#endif
double wide_weighted_call(int64_t D1, int64_t D2, int64_t D3, int64_t D4, int G1, int G2, int G3, int G4, WideConst c,
                          int weights) {
    if (G1 == G4 && G2 == G3 && uint64_t(D1 + D4 + 8) <= 16 && uint64_t(D2 + D3 + 8) <= 16) {
        D4 = -D1;
        D3 = -D2;
    }
    int e0, e1, e2, e3;
    const int64_t x0 = wide_normalise(D1, G1, e0), x1 = wide_normalise(D2, G2, e1), x2 = wide_normalise(D3, G3, e2),
                  x3 = wide_normalise(D4, G4, e3);
    return wide_weighted(ones(x0), ones(x1), ones(x2), ones(x3), e0, e1, e2, e3, c, W < 0 ? weights : W);
}

// Whether the largest difference lies in the range of the integer evaluation (E its exponent).
WZ_HD bool wide_in_range(int E) { return unsigned(E - kWideMinExp) < unsigned(kWideMaxExp - kWideMinExp); }

// f^ - c from D_i 2^(G_i - 1082), |D_i| <= 2^60, to be added to a value of exponent eb.  False
// where the caller has to take the double evaluation (the largest difference outside the range
// above).  W: the weight function, -1 for the run-time value.
template <int W>
WZ_HD bool wide_correction(int64_t D1, int64_t D2, int64_t D3, int64_t D4, int G1, int G2, int G3, int G4, int eb,
                           const WideConst& c, int weights, double& corr) {
    if (wide_linear<false>(D1, D2, D3, D4, G1, G2, G3, G4, eb, c, W < 0 ? weights : W, corr)) return true;
    corr = 0.0;
    int e0, e1, e2, e3;
    wide_normalise(D1, G1, e0);
    wide_normalise(D2, G2, e1);
    wide_normalise(D3, G3, e2);
    wide_normalise(D4, G4, e3);
    const int E = max_i(max_i(e0, e1), max_i(e2, e3));
    // (constant data; other differences below 2^-1022 are not zero)
    if (!wide_in_range(E) || (W < 0 && weights == 2)) return (D1 | D2 | D3 | D4) == 0;
    corr = wide_weighted_call<W>(D1, D2, D3, D4, G1, G2, G3, G4, c, weights);
    return true;
}

// The same from the first differences as doubles (infinities and NaN return false).
template <int W>
WZ_HD bool wide_correction(double D1, double D2, double D3, double D4, int eb, const WideConst& c, int weights,
                           double& corr) {
    int e0, e1, e2, e3;
    const int64_t o0 = wide_unpack_ones(D1, e0), o1 = wide_unpack_ones(D2, e1), o2 = wide_unpack_ones(D3, e2),
                  o3 = wide_unpack_ones(D4, e3);
    const int E = max_i(max_i(e0, e1), max_i(e2, e3));
    corr = 0.0;
    if (!wide_in_range(E)) return ((double_bits(D1) | double_bits(D2) | double_bits(D3) | double_bits(D4)) << 1) == 0;
    if (wide_linear<true>(o0, o1, o2, o3, e0, e1, e2, e3, eb, c, W < 0 ? weights : W, corr)) return true;
    if (W < 0 && weights == 2) return false;
    corr = wide_weighted(o0, o1, o2, o3, e0, e1, e2, e3, c, W < 0 ? weights : W);
    return true;
}

}  // namespace wz
