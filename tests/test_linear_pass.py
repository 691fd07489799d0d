"""The linear pass of the Euler fluxes (NearLinear and interface_linear in csrc/euler_device.cuh)
over data of any units: an interface it accepts has to be right whatever the scales of density
and velocity, since it is taken without the weights.  And the flux with its weights on mirrored
stencils, where tau5 = 0.

On the host the device code is compiled as plain C++ and every interface (of the linear pass, every
accepted one) is compared with a binary128 evaluation of the scheme from the same split fluxes.  Tolerance, from the
operations: the two sides' linear parts are integer sums of differences truncated at 2^-56 of the
largest (2 x 40/60 units), rounded once to 53 bits, the centre sum, the correction and R Delta
are added with one rounding each, and Delta is off by less than 2^-57 of a field's value:
|error| <= 2^-51 sum_k |R_mk| (|g_k| + max |D_k|), both sides' fields g_k and differences D_k."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_07954_gb300", "csrc")
SHIM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
#define __shared__ static
static struct { unsigned x; } threadIdx, blockDim;
using std::isfinite; using std::max;
static long long __double_as_longlong(double d) { long long u; std::memcpy(&u, &d, 8); return u; }
static double __longlong_as_double(long long u) { double d; std::memcpy(&d, &u, 8); return d; }
static int __double2hiint(double d) { return int(__double_as_longlong(d) >> 32); }
static double __ddiv_rn(double a, double b) { return a / b; }
static double __dmul_rn(double a, double b) { return a * b; }
static double __dadd_rn(double a, double b) { return a + b; }
static double __dsqrt_rn(double a) { return std::sqrt(a); }
static double rsqrt(double a) { return 1.0 / std::sqrt(a); }
static float rsqrtf(float a) { return float(1.0 / std::sqrt(double(a))); }
static double __shfl_xor_sync(unsigned, double v, int) { return v; }
static void __syncthreads() {}
static void atomicMax(unsigned long long* p, unsigned long long v) { if (v > *p) *p = v; }
static uint32_t __vimax3_u16x2(uint32_t a, uint32_t b, uint32_t c) {
    return max(max(a & 0xffffu, b & 0xffffu), c & 0xffffu) | (max(max(a >> 16, b >> 16), c >> 16) << 16);
}
#include "euler_device.cuh"
using namespace wz;
#ifdef __aarch64__
typedef long double Q;
#else
typedef __float128 Q;
#endif
static Q mag(Q a) { return a < 0 ? -a : a; }
static Q root(Q a) { Q y = std::sqrt(double(a)); for (int i = 0; i < 4; ++i) y = (y + a / y) / 2; return y; }
static Q weno(const Q* D, Q eps, Q A) {
    const Q s0 = D[0] - D[1], s1 = D[1] - D[2], s2 = D[2] - D[3], t0 = D[0] - 3 * D[1], t1 = D[1] + D[2], t2 = 3 * D[2] - D[3];
    const Q k = Q(13) / 12, i0 = k * s0 * s0 + t0 * t0 / 4, i1 = k * s1 * s1 + t1 * t1 / 4, i2 = k * s2 * s2 + t2 * t2 / 4;
    const Q tau = mag(i0 - i2), d4 = t0 + t2, c = (i0 + i2 - tau + eps) / (tau + eps), C = A * c * c;
    const Q a0 = C + d4 * d4 / (i0 + eps), a1 = 6 * (C + d4 * d4 / (i1 + eps)), a2 = 3 * (C + d4 * d4 / (i2 + eps));
    return (a0 * (2 * D[0] - 5 * D[1]) - a1 * (D[1] + 2 * D[2]) + a2 * (D[3] - 4 * D[2])) / (6 * (a0 + a1 + a2));
}
// the interface flux F of the six cells' split fluxes, and the scale of the tolerance
template <int NV> void exact(const CellPlanes<NV>& s, Q gm1, Q eps, Q A, Q* F, Q* scale) {
    const int NC = s.NC, E = NV - 1;
    const Q w = Q(s.sr[2]) / (Q(s.sr[2]) + Q(s.sr[3])), u = w * s.un[2] + (1 - w) * s.un[3];
    const Q v = NV == 4 ? w * s.ut[2] + (1 - w) * s.ut[3] : Q(0), H = w * s.H[2] + (1 - w) * s.H[3];
    const Q q2 = u * u + v * v, c2 = gm1 * (H - q2 / 2), c = root(c2), b1 = gm1 / c2, b2 = q2 * b1 / 2;
    auto project = [&](const Q* h, Q* g) {
        const Q W = u * h[1] - h[E] + (NV == 4 ? v * h[2] : Q(0)), Z = b2 * h[0] - b1 * W, B = (u * h[0] - h[1]) / (2 * c);
        if (NV == 4) g[2] = h[2] - v * h[0];
        g[0] = Z / 2 + B; g[1] = h[0] - Z; g[E] = Z / 2 - B;
    };
    Q gh[NV] = {}, gs[NV] = {};
    for (int side = 0; side < 2; ++side) {
        const double* h = side == 0 ? s.hp : s.hm;
        Q D[NV][4], d[NV], g[NV];
        for (int st = 0; st < 4; ++st) {
            const int i = side == 0 ? st : 5 - st, n = side == 0 ? i + 1 : i - 1;
            for (int m = 0; m < NV; ++m) d[m] = Q(h[m * NC + i]) - Q(h[m * NC + n]);
            project(d, g);
            for (int k = 0; k < NV; ++k) D[k][st] = g[k];
        }
        for (int m = 0; m < NV; ++m) d[m] = h[m * NC + 2 + side];
        project(d, g);
        for (int k = 0; k < NV; ++k) {
            gh[k] += g[k] + weno(D[k], eps, A);
            gs[k] += max(max(mag(D[k][0]), mag(D[k][1])), max(mag(D[k][2]), mag(D[k][3]))) + mag(g[k]);
        }
    }
    for (int abs = 0; abs < 2; ++abs) {
        const Q* g = abs ? gs : gh;
        Q* o = abs ? scale : F;
        auto r = [&](Q x) { return abs ? mag(x) : x; };
        const Q a = g[0] + g[1] + g[E];
        o[0] = a;
        o[1] = r(u - c) * g[0] + r(u) * g[1] + r(u + c) * g[E];
        o[E] = r(H - u * c) * g[0] + q2 / 2 * g[1] + r(H + u * c) * g[E];
        if (NV == 4) { o[2] = r(v) * a + g[2]; o[E] += r(v) * g[2]; }
    }
}
// U: n x 6 cells x NV; out: the accepted interfaces' error over the tolerance's scale, -1 refused
template <int NV> void all(const double* U, long n, double gamma, double eps, double A, double* out) {
    static double buf[CellPlanes<NV>::kPerCellGeneric * 6];
    const CellPlanes<NV> s(buf, 6);
    const WideConst wc = wide_const(eps, A);
    for (long t = 0; t < n; ++t, U += 6 * NV) {
        double al = 0.0, F[NV];
        for (int c = 0; c < 6; ++c) {
            const double* q = U + c * NV;
            const double m2 = q[1] * q[1] + (NV == 4 ? q[2] * q[2] : 0.0), p = (gamma - 1.0) * (q[NV - 1] - 0.5 * m2 / q[0]);
            al = std::max(al, std::fabs(q[1] / q[0]) + std::sqrt(gamma * p / q[0]));
        }
        for (int c = 0; c < 6; ++c) split_cell<NV>(U + c * NV, al, 0.0, gamma - 1.0, s, c);
        for (int c = 0; c < 5; ++c) cell_diffs<NV>(s, c, 1);
        out[t] = -1.0;
        if (!interface_linear<NV>(s, 0, 1, gamma - 1.0, wc, F)) continue;
        Q G[NV], scale[NV];
        exact<NV>(s, gamma - 1.0, eps, A, G, scale);
        out[t] = 0.0;
        for (int m = 0; m < NV; ++m) out[t] = F[m] == F[m] ? std::max(out[t], double(mag(F[m] - G[m]) / scale[m])) : 1.0;
    }
}
template <int NV> void general(const double* U, long n, double gamma, double eps, double A, double* out) {
    static double buf[CellPlanes<NV>::kPerCellGeneric * 6];
    const CellPlanes<NV> s(buf, 6);
    const WideConst wc = wide_const(eps, A);
    for (long t = 0; t < n; ++t, U += 6 * NV) {
        double F[NV];
        for (int c = 0; c < 6; ++c) split_cell<NV>(U + c * NV, 3.0, 0.0, gamma - 1.0, s, c);
        for (int c = 0; c < 5; ++c) cell_diffs<NV>(s, c, 1);
        interface_flux<NV, 0>(s, 0, 1, gamma - 1.0, wc, 4.0 * eps, 2.0 / std::sqrt(A), 0, 0, nullptr, F);
        Q G[NV], scale[NV];
        exact<NV>(s, gamma - 1.0, eps, A, G, scale);
        out[t] = 0.0;
        for (int m = 0; m < NV; ++m) out[t] = std::max(out[t], double(mag(F[m] - G[m]) / scale[m]));
    }
}
extern "C" void general_errors(int nv, const double* U, long n, double eps, double A, double* out) {
    if (nv == 3) general<3>(U, n, 1.4, eps, A, out);
    else general<4>(U, n, 1.4, eps, A, out);
}
extern "C" void linear_errors(int nv, const double* U, long n, double eps, double A, double* out) {
    if (nv == 3) all<3>(U, n, 1.4, eps, A, out);
    else all<4>(U, n, 1.4, eps, A, out);
}
"""


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    d = tmp_path_factory.mktemp("linear")
    src, so = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as fh:
        fh.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-w", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, src, "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    P = ctypes.c_void_p

    def run(U, eps=1e-40, A=10.0, entry=L.linear_errors):
        U = np.ascontiguousarray(U)
        out = np.empty(U.shape[0])
        entry.argtypes = [ctypes.c_int, P, ctypes.c_long, ctypes.c_double, ctypes.c_double, P]
        entry(U.shape[2], U.ctypes.data, U.shape[0], eps, A, out.ctypes.data)
        return out

    run.general = L.general_errors

    return run


def _stencils(kind, nv, n=1500, seed=1):
    """n six-cell stencils of order-one states: (n, 6) arrays rho, u, v, p."""
    g = np.random.default_rng(seed + nv)
    c = np.arange(6)[None, :, None]
    if kind == "random":
        q = g.uniform(-0.8, 0.8, size=(n, 6, 4))
    else:
        amp = 10.0 ** g.uniform(-12, -0.5, size=(n, 1, 4 if kind == "unlike" else 1)) * np.ones((1, 1, 4))
        q = amp * np.sin(g.uniform(0, 6.28, size=(n, 1, 4)) + c * 10.0 ** g.uniform(-3, -0.5, size=(n, 1, 1)))
        if kind == "jumps":
            q = q + 0.4 * (c >= g.integers(0, 6, size=(n, 1, 1)))
    base = g.uniform(-2, 2, size=(n, 1, 2))
    return 1 + q[..., 0], base[..., 0] + q[..., 1], (base[..., 1] + q[..., 2]) * (nv == 4), 1 + q[..., 3]


def _cons(rho, u, v, p, nv):
    E = p / 0.4 + 0.5 * rho * (u * u + v * v)
    return np.stack([rho, rho * u] + ([rho * v] if nv == 4 else []) + [E], axis=-1)


@pytest.mark.parametrize("nv", [3, 4])
@pytest.mark.parametrize("kind", ["random", "jumps", "smooth", "unlike"])
def test_accepted_interfaces_are_right_in_any_units(errors, kind, nv):
    rho, u, v, p = _stencils(kind, nv)
    taken = 0
    for r in (1.0, 2.0 ** -40, 2.0 ** 40):
        for f in (1.0, 2.0 ** -60, 2.0 ** -20, 2.0 ** 20, 2.0 ** 34, 2.0 ** 36, 2.0 ** 38, 2.0 ** 60, 2.0 ** 90):
            e = errors(_cons(r * rho, f * u, f * v, r * f * f * p, nv))
            assert e.max() <= 2.0 ** -51, (r, f, int((e > 2.0 ** -51).sum()))
            taken += int((e >= 0).sum())
    assert taken > 0 or kind == "random"


@pytest.mark.parametrize("kind", ["random", "jumps", "smooth", "unlike"])
def test_accepted_interfaces_beside_fast_tangential_flow(errors, kind):
    rho, u, v, p = _stencils(kind, 4)
    for t in (1e2, 1e4, 1e6):
        for f in (1.0, 2.0 ** 20, 2.0 ** 24):
            assert errors(_cons(rho, f * u, f * t * v, f * f * p, 4)).max() <= 2.0 ** -51, (t, f)


@pytest.mark.parametrize("nv", [3, 4])
@pytest.mark.parametrize("eps,A", [(1e-6, 10.0), (1.0, 1e-6), (1.0, 1e6), (1e-60, 1e-6), (1e-60, 1e6), (1e-20, 10.0)])
def test_accepted_interfaces_with_other_constants(errors, eps, A, nv):
    for kind in ("random", "jumps", "smooth", "unlike"):
        rho, u, v, p = _stencils(kind, nv, 600)
        for r, f in ((1.0, 1.0), (2.0 ** -27, 2.0 ** 10), (2.0 ** -60, 2.0 ** -40), (2.0 ** 30, 2.0 ** 30)):
            assert errors(_cons(r * rho, f * u, f * v, r * f * f * p, nv), eps, A).max() <= 2.0 ** -51, (kind, r, f)


@pytest.mark.parametrize("nv", [3, 4])
@pytest.mark.parametrize("eps,A", [(1e-40, 10.0), (1e-6, 10.0), (1e-60, 1e-6)])
def test_plateaus_between_equal_neighbours(errors, eps, A, nv):
    """Cells a, b, b, b, a, c and their mirror image: tau5 of every field is zero exactly, and b_1 is
    eps alone, so a last bit between the two ends' projections would decide the weights."""
    g = np.random.default_rng(nv)
    q = g.uniform(-0.8, 0.8, size=(400, 3, 4))
    S = _cons(1 + q[..., 0], q[..., 1], q[..., 2] * (nv == 4), 1 + q[..., 3], nv)
    for order in ((0, 1, 1, 1, 0, 2), (2, 0, 1, 1, 1, 0), (0, 1, 1, 1, 0, 0)):
        assert errors(S[:, order], eps, A, errors.general).max() <= 2.0 ** -51, order


def _line(n):
    """Smooth waves with jumps, (3, n)."""
    x = (np.arange(n) + 0.5) / n
    w = lambda m, a, s: a * np.sin(2 * np.pi * m * x + s)
    rho = 1.0 + w(n // 150, 0.2, 0.3) + (x > 0.3) + 2.0 * (x > 0.7)
    u, p = 0.4 + w(n // 120, 0.2, 1.0), 1.0 + w(n // 90, 0.2, 2.0) + 3.0 * ((x > 0.5) & (x < 0.9))
    return np.stack([rho, rho * u, p / 0.4 + 0.5 * rho * u * u])


def _same(got, want, f, tol=1e-13):
    """got = want with velocities in units 1/f: momentum f, energy f^2; both with `want`'s other units taken out."""
    for k in range(len(want)):
        g = got[k] / (1.0 if k == 0 else (f if k < len(want) - 1 else f * f))
        assert np.abs(g - want[k]).max() <= tol * np.abs(want[k]).max(), k


@pytest.mark.gpu
@pytest.mark.parametrize("f", [2.0 ** 20, 2.0 ** 36, 2.0 ** 40, 2.0 ** 60])
def test_gpu_velocity_units(f):
    """Sizes that take the linear pass (a long line, 2D sweeps of 700 cells, batch instances of 1024
    and more): with velocities f times larger the RHS is that of the order-one data, f times
    larger in density, f^2 in momentum, f^3 in energy (eps plays no part), to the rounding of
    powers of two through the same operations."""
    import torch
    from paper_2004_07954_gb300 import build, wenozn as W
    build.build()
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def rhs(U, nx, ny, system, h):
        p = W.wenozn_problem_init(system, nx, ny, h, h, bc_x=W.WENOZN_BC_PERIODIC, bc_y=W.WENOZN_BC_PERIODIC)
        return W.Solver(p).rhs(dev(U)).cpu().numpy()

    U = _line(40001)
    S = U * np.array([1.0, f, f * f])[:, None]
    one, big = (rhs(a[:, None], 40001, 1, 1, 1e-3)[:, 0] for a in (U, S))
    _same(big / f, one, f)
    U = _line(700)
    for axis in (0, 1):
        Z = np.zeros((4, 16, 700))
        Z[0], Z[1 + axis], Z[2 - axis], Z[3] = U[0], U[1], 0.7 * U[0], U[2] + 0.5 * 0.49 * U[0]
        Z = Z if axis == 0 else Z.transpose(0, 2, 1)
        nx, ny = (700, 16) if axis == 0 else (16, 700)
        one, big = (rhs(a, nx, ny, 2, 1e-3) for a in (Z, Z * np.array([1.0, f, f, f * f])[:, None, None]))
        _same(big / f, one, f)
    off, dx = np.array([0, 1024, 2100, 3600]), np.full(3, 1e-3)
    U = np.concatenate([_line(1024), _line(1076), _line(1500)], 1)
    out = []
    for a in (U, U * np.array([1.0, f, f * f])[:, None]):
        t = dev(a)
        W.Batch(off, dx, t).step(t)
        out.append(t.cpu().numpy())
    _same(out[1], out[0], f)


@pytest.mark.gpu
@pytest.mark.parametrize("system,nx,ny,split,weights", [
    (1, 200, 1, 0, 0), (1, 200, 1, 3, 0), (1, 200, 1, 0, 1), (1, 200, 1, 2, 0), (1, 40000, 1, 0, 0), (1, 40000, 1, 3, 1),
    (2, 96, 40, 0, 0), (2, 700, 16, 0, 0), (2, 16, 700, 0, 0), (2, 700, 16, 3, 0), (2, 96, 40, 2, 0), (2, 96, 40, 1, 1)])
def test_gpu_plateaus_between_equal_neighbours(orc, system, nx, ny, split, weights):
    """Two states alternating in pieces of three cells along both axes, through every Euler flux
    kernel: the RHS against the oracle in binary128, at 1e-14 of the flux over dx.  (The oracle's own
    tau5 is not exactly zero on every such stencil: in double that shows in its result, in binary128
    only where tau5 is divided by eps, so WENO-Z takes eps = 1e-6.)"""
    import torch
    from paper_2004_07954_gb300 import build, inputs, wenozn as W
    build.build()
    i = (np.arange(nx) // 3 % 2)[None, :] ^ (np.arange(ny) // 3 % 2)[:, None]
    pick = lambda a, b: np.where(i == 0, a, b)
    rho, u, v, pr = pick(1.0, 0.6), pick(0.3, 0.2), pick(-0.1, 0.25), pick(1.0, 0.7)
    U = inputs.cons_from_prim(rho, u, pr, v) if system == 2 else inputs.cons_from_prim(rho, u, pr).reshape(3, 1, nx)
    U, h, nv = np.ascontiguousarray(U), 1.0 / 96, 3 if system == 1 else 4
    opt = dict(split=split, weights=weights, eps=1e-6 if weights == 1 else 1e-40)
    got = W.Solver(W.wenozn_problem_init(system, nx, ny, h, h, **opt)).rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    want, _ = orc.rhs_jvp_quad(orc.problem(system, nx, ny, dx=h, dy=h, **opt), U, U)
    for k in range(nv):
        assert np.abs(got[k] - want[k]).max() <= 1e-14 * 10.0 / h, k


@pytest.mark.gpu
def test_gpu_plateaus_in_a_batch(orc):
    import torch
    from paper_2004_07954_gb300 import build, inputs, wenozn as W
    build.build()
    U = []
    for n in (150, 1500):                      # below and in the linear pass
        i = np.arange(n) // 3 % 2
        U.append(inputs.cons_from_prim(np.where(i, 0.6, 1.0), np.where(i, 0.2, 0.3), np.where(i, 0.7, 1.0)))
    t = torch.from_numpy(np.ascontiguousarray(np.concatenate(U, 1))).cuda()
    W.Batch(np.array([0, 150, 1650]), np.full(2, 0.01), t).step(t)
    got = t.cpu().numpy()
    for o, a in ((0, U[0]), (150, U[1])):
        n, a = a.shape[1], a.reshape(3, 1, -1)
        P = orc.problem(1, n, 1, dx=0.01)
        want, _ = orc.rollout_jvp_quad(P, a, a, orc.cfl_dt(P, a), 1)
        assert np.abs(got[:, o:o + n] - want[:, 0]).max() <= 1e-12 * np.abs(want).max()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2000, 20001])
@pytest.mark.parametrize("f", [2.0 ** 20, 2.0 ** 36, 2.0 ** 40])
def test_gpu_adjoint_in_velocity_units(n, f):
    """The reverse makes the same check, in both its kernels: with S = diag(1, f, f^2) the RHS of S U is
    f S L(U), so J(S U)^T S^-1 lam = f S^-1 J(U)^T lam, to 1e-10 (the adjoint tests' figure)."""
    import torch
    from paper_2004_07954_gb300 import build, wenozn as W
    build.build()
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    p = W.wenozn_problem_init(W.WENOZN_EULER_1D, n, dx=1e-3, bc_x=W.WENOZN_BC_PERIODIC)
    ws, S = W.vjp_workspace(p), np.array([1.0, f, f * f])[:, None, None]
    U, lam = _line(n)[:, None], np.random.default_rng(3).normal(size=(3, 1, n))
    one, big = torch.empty_like(dev(U)), torch.empty_like(dev(U))
    W.wenozn_rhs_vjp(p, dev(U), dev(lam), one, ws)
    W.wenozn_rhs_vjp(p, dev(U * S), dev(lam / S), big, ws)
    got, want = big.cpu().numpy() * S / f, one.cpu().numpy()
    assert np.abs(got - want).max() <= 1e-10 * np.abs(want).max()
