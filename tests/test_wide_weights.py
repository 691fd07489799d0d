"""The integer evaluation of the reconstruction (csrc/wide_weights.cuh): compiled for the host
against the binary128 oracle, and on the GPU at the edges of its range.

Tolerance, from the operations: the numerator's operands are exact or off by 2^-58 of the
largest difference Dmax, every weight a_k by less than 2^-53 relative, so f^ - c is off by less
than 2^-52 Dmax before its rounding to 53 bits (|f^ - c| <= 7/6 Dmax), and the centre value is
added with one more rounding: |error| <= 2^-51 (Dmax + |f^|)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_07954_gb300", "csrc")
SHIM = """
#include "wide_weights.cuh"
extern "C" long wide_line(const double* f, long n, int side, double eps, double A, int weights,
                          double* out) {
    const wz::WideConst c = wz::wide_const(eps, A);
    long refused = 0;
    for (long j = 0; j <= n; ++j) {
        const double* s = f + j;
        double v[5], corr;
        for (int k = 0; k < 5; ++k) v[k] = side > 0 ? s[k] : s[5 - k];
        if (!wz::wide_correction<-1>(v[0] - v[1], v[1] - v[2], v[2] - v[3], v[3] - v[4], wz::exponent_of(v[2]), c, weights, corr))
            ++refused, corr = 0.0;
        out[j] = v[2] + corr;
    }
    return refused;
}
"""


@pytest.fixture(scope="module")
def wide(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide")
    src, so = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as fh:
        fh.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, src, "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    P = ctypes.c_void_p
    L.wide_line.argtypes = [P, ctypes.c_long, ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int, P]
    L.wide_line.restype = ctypes.c_long

    def line(f, side, eps=1e-40, A=10.0, weights=0):
        out = np.empty(f.size - 5)
        refused = L.wide_line(f.ctypes.data, f.size - 6, side, eps, A, weights, out.ctypes.data)
        return out, refused

    return line


def _lines(n=600):
    g = np.random.default_rng(7)
    x = np.arange(n + 6) / n
    smooth = np.sin(2 * np.pi * x) + 0.3 * np.cos(17 * x)
    jumps = smooth + (x > 0.3) - 2.0 * (x > 0.31) + 1e3 * (x > 0.7)
    return {
        "random": g.normal(size=n + 6),
        "smooth": smooth,
        "jumps": jumps,
        "steps": np.round(g.normal(size=n + 6)),                       # flat pieces, exact zeros
        "noise beside jumps": np.where(x < 0.5, 1.0, -2.0) + 1e-15 * g.normal(size=n + 6),
        "ranges": g.normal(size=n + 6) * 10.0 ** g.uniform(-30, 0, size=n + 6),
        "flat": np.full(n + 6, 0.7),
        "zeros": np.where(g.random(n + 6) < 0.5, 0.0, -0.0),
    }


def _bound(f, ref, side):
    d = np.abs(np.diff(f))
    win = np.lib.stride_tricks.sliding_window_view(d, 4).max(axis=1)
    dmax = win[:-1] if side > 0 else win[1:]
    return 2.0 ** -51 * (dmax + np.abs(ref))


@pytest.mark.parametrize("eps,A", [(1e-40, 10.0), (1e-6, 10.0), (1e-60, 1e6), (1.0, 0.1)])
@pytest.mark.parametrize("name", list(_lines()))
def test_integer_evaluation_against_binary128(wide, orc, name, eps, A):
    f = np.ascontiguousarray(_lines()[name])
    for scale in (1.0, 2.0 ** -200, 2.0 ** 390):
        fs = f * scale
        for side in (1, -1):
            got, refused = wide(fs, side, eps, A)
            assert refused == 0 or scale != 1.0
            ref = orc.reconstruct_quad(fs, side, eps=eps, A=A)
            if refused == 0:
                assert np.all(np.abs(got - ref) <= _bound(fs, ref, side)), (scale, side)


@pytest.mark.parametrize("weights,eps", [(1, 1e-40), (1, 1e-6), (2, 1e-40), (3, 1e-6), (3, 1e-40)])
@pytest.mark.parametrize("name", list(_lines()))
def test_integer_evaluation_of_the_other_weights(wide, orc, name, weights, eps):
    """WENO-Z, linear and Jiang-Shu weights, the same bound."""
    f = np.ascontiguousarray(_lines()[name])
    for side in (1, -1):
        got, refused = wide(f, side, eps, 10.0, weights)
        ref = orc.reconstruct_quad(f, side, eps=eps, kind=weights)
        assert refused == 0
        assert np.all(np.abs(got - ref) <= _bound(f, ref, side)), side


@pytest.mark.parametrize("eps,A", [(1e-40, 10.0), (1e-6, 1e-6), (1.0, 1e-6), (1e-6, 0.1)])
def test_a_tie_leaves_eps_alone_in_the_weights(wide, orc, eps, A):
    """b_0 = b_2 far above eps: tau5 + eps is eps, which has to keep its own precision (the module's
    bound), for every size of the differences."""
    for x in 10.0 ** np.arange(-12.0, 13.0):
        for f in ([-x, 0.0, 0.0, 0.0, -x, 0.0], [-x, 0.0, 0.0, 0.0, -x, 0.4 * x], [3.0 * x, x, 0.0, x, 3.0 * x, 0.0]):
            for side in (1, -1):
                g = np.array(f if side > 0 else f[::-1])
                got, refused = wide(g, side, eps, A)
                ref = orc.reconstruct_quad(g, side, eps=eps, A=A)
                assert refused == 0 and abs(got[0] - ref[0]) <= _bound(g, ref, side)[0], (x, f, side)


@pytest.mark.parametrize("scale", [2.0 ** -320, 2.0 ** -300, 2.0 ** -290, 1.0, 2.0 ** 390, 2.0 ** 399])
@pytest.mark.parametrize("name", list(_lines()))
def test_every_stencil_is_right_or_refused_by_its_range(wide, orc, name, scale):
    """Stencil by stencil: refused exactly where the largest difference leaves [2^-300, 2^400), unless
    all are zero; every other one within the bound."""
    f = np.ascontiguousarray(_lines()[name] * scale)
    for side in (1, -1):
        ref = orc.reconstruct_quad(f, side)
        bound = _bound(f, ref, side)
        d = np.abs(np.diff(f))
        for j in range(ref.size):
            dmax = d[j:j + 4].max() if side > 0 else d[j + 1:j + 5].max()
            got, refused = wide(f[j:j + 6].copy(), side)
            assert bool(refused) == (dmax != 0.0 and not 2.0 ** -300 <= dmax < 2.0 ** 400), (j, side)
            assert refused or abs(got[0] - ref[j]) <= bound[j], (j, side)


@pytest.mark.parametrize("A", [10.0, 1e-6])
def test_stencils_mirrored_about_their_centre(wide, orc, A):
    """D4 = -D1, D3 = -D2: tau5 = 0 exactly, however flat the top is (the module's bound)."""
    y = np.concatenate([10.0 ** -np.arange(1.0, 17.0), 2.0 ** -np.arange(1.0, 50.0), [0.0]])
    for D1, D2 in ((y - 1.0, y), (-np.ones_like(y), y), (1.0 + y, -y)):
        for sixth in (0.0, 0.3):
            for a, b in zip(D1, D2):
                f = np.array([a + b, b, 0.0, b, a + b, sixth])
                for side in (1, -1):
                    g = f if side > 0 else f[::-1].copy()
                    got, refused = wide(g, side, 1e-40, A)
                    ref = orc.reconstruct_quad(g, side, eps=1e-40, A=A)
                    assert refused == 0 and abs(got[0] - ref[0]) <= _bound(g, ref, side)[0], (a, b, side)


@pytest.mark.parametrize("weights", [0, 1, 2, 3])
@pytest.mark.parametrize("name", list(_lines()) + ["single precision"])
def test_odd_in_the_data_and_mirrored_between_the_sides(wide, name, weights):
    """f^(-f) = -f^(f), and the plus side is the minus side of the reversed line, bit for bit."""
    f = _lines()[name] if name in _lines() else np.random.default_rng(3).normal(size=3006).astype(np.float32).astype(np.float64)
    for scale in (1.0, 2.0 ** -100):
        g = np.ascontiguousarray(f * scale)
        got = wide(g, 1, weights=weights)[0]
        assert np.array_equal(wide(-g, 1, weights=weights)[0], -got)
        assert np.array_equal(wide(g[::-1].copy(), -1, weights=weights)[0][::-1], got)


def test_constant_data_are_exact_and_other_values_refused(wide):
    for c in (0.0, -0.0, 0.1, -3.7e200):
        got, refused = wide(np.full(40, c), 1)
        assert refused == 0 and np.array_equal(got, np.full(35, c))
    for bad in (np.nan, np.inf, 2.0 ** 402):
        f = np.zeros(40)
        f[20] = bad
        assert wide(f, 1)[1] > 0


def test_differences_below_the_normal_range_are_refused(wide):
    """They are no zeros: the double evaluation has to take them."""
    f = np.random.default_rng(1).integers(-2 ** 40, 2 ** 40, size=46) * 5e-324
    for side in (1, -1):
        assert wide(f, side)[1] == 41
        assert wide(np.where(np.arange(46) < 23, f, f[22]), side)[1] < 41


def test_integer_reciprocal_square_root_and_halves(tmp_path):
    """wide_reciprocal and wide_rsqrt to 0.506 of a last place over their ranges (the comments' figure,
    with the host's seeds), wide_half and wide_truncate to the bit."""
    src, so = str(tmp_path / "f.cpp"), str(tmp_path / "f.so")
    with open(src, "w") as fh:
        fh.write("""#include "wide_weights.cuh"
extern "C" void f(const double* x, long n, double* r, double* q, double* h, float* t) {
    bool ok;
    for (long i = 0; i < n; ++i) {
        r[i] = wz::wide_reciprocal(x[i]);
        q[i] = wz::wide_rsqrt(x[i], ok);
        h[i] = wz::wide_half(x[i]);
        t[i] = wz::wide_truncate(x[i]);
    }
}""")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    g = np.random.default_rng(2)
    p = 2.0 ** np.arange(-1000.0, 1001.0)
    x = np.concatenate([p, np.nextafter(p, 0), np.nextafter(p, np.inf), g.uniform(1, 4, 20000) * 2.0 ** g.integers(-1000, 999, 20000)])
    r, q, h, t = np.empty_like(x), np.empty_like(x), np.empty_like(x), np.empty(x.size, np.float32)
    P = ctypes.c_void_p
    L = ctypes.CDLL(so)
    L.f.argtypes = [P, ctypes.c_long, P, P, P, P]
    L.f(x.ctypes.data, x.size, r.ctypes.data, q.ctypes.data, h.ctypes.data, t.ctypes.data)
    from fractions import Fraction as F
    for xi, ri, qi in zip(x[::7].tolist(), r[::7].tolist(), q[::7].tolist()):
        ulp = F(float(np.spacing(ri)))
        assert abs(F(ri) - 1 / F(xi)) <= F(506, 1000) * ulp, xi
        # |q - 1/sqrt(x)| <= e  <=>  (q - e)^2 x <= 1 <= (q + e)^2 x
        e = F(506, 1000) * F(float(np.spacing(qi)))
        assert (F(qi) - e) ** 2 * F(xi) <= 1 <= (F(qi) + e) ** 2 * F(xi), xi
    assert np.array_equal(h, 0.5 * x)
    y = (x.view(np.uint64) & np.uint64(0xFFFFFFFFE0000000)).view(np.float64)          # 24 bits kept
    inside = (x >= 2.0 ** -126) & (x < 2.0 ** 127)
    assert np.array_equal(t[inside].astype(np.float64), y[inside]) and np.all(np.isnan(t[~inside]))


@pytest.mark.gpu
@pytest.mark.parametrize("weights", [0, 1, 2, 3])
def test_gpu_reconstruction_of_subnormal_data(orc, weights):
    """Against the binary128 evaluation, to the last places of the subnormal range: the double
    evaluation's differences are exact there, its weights off by 1e-12 at most."""
    import torch
    from paper_2004_07954_gb300 import build, wenozn as W
    build.build()
    f = np.random.default_rng(1).integers(-2 ** 50, 2 ** 50, size=606) * 5e-324
    out = torch.empty(601, dtype=torch.float64, device="cuda")
    for side in (1, -1):
        W.wenozn_reconstruct_weights(torch.from_numpy(f).cuda(), out, side, weights)
        ref = orc.reconstruct_quad(f, side, kind=weights)
        # (in units of the smallest double, which 1e-12 of the data is about a thousandth of)
        assert np.abs((out.cpu().numpy() - ref) / 5e-324).max() <= 4 + 1e-12 * 2 ** 50


@pytest.mark.gpu
@pytest.mark.parametrize("k", [-320, -301, -300, -299, 0, 398, 399, 400])
def test_gpu_reconstruction_across_the_range_switch(orc, k):
    """Differences on both sides of the exponents where the double evaluation takes over, block
    and warp remainders, a NaN reaching exactly the stencils that hold it."""
    import torch
    from paper_2004_07954_gb300 import build, wenozn as W
    build.build()
    for n in (1, 31, 255, 256, 257, 600):
        f = np.random.default_rng(n).normal(size=n + 6) * 2.0 ** k
        t = torch.from_numpy(f).cuda()
        out = torch.empty(n + 1, dtype=torch.float64, device="cuda")
        for side in (1, -1):
            W.wenozn_reconstruct(t, out, side)
            ref = orc.reconstruct_quad(f, side)
            # (the double evaluation's own bound in this suite is 1e-12 of the data's scale)
            assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * np.abs(f).max()
    f[n // 2] = np.nan
    W.wenozn_reconstruct(torch.from_numpy(f).cuda(), out, 1)
    bad = np.isnan(out.cpu().numpy())
    assert np.array_equal(np.flatnonzero(bad), np.arange(n // 2 - 4, n // 2 + 1))


def _state_2d(kind, nx, ny):
    """2D Euler states that put the integer projection at its limits."""
    from paper_2004_07954_gb300 import inputs
    g = np.random.default_rng(5)
    one = np.ones((ny, nx))
    rho, u, v, p = 1.0 + 0.2 * g.random((ny, nx)), 0.3 * g.random((ny, nx)), 0.2 * g.random((ny, nx)), 1.0 + 0.1 * g.random((ny, nx))
    if kind == "rest":                       # every difference zero, momenta zero
        rho, u, v, p = one, 0 * one, 0 * one, one
    elif kind == "signed zeros":
        rho, u, v, p = one, -0.0 * one, 0 * one, one
    elif kind == "tiny shear":               # transverse differences below the scale of eps
        v = 1e-30 * g.normal(size=(ny, nx))
    elif kind == "blast":                    # neighbouring cells 10^5 apart in pressure, along a front
        p = p * np.where(np.arange(nx) < nx // 2, 1000.0, 0.01)
    elif kind == "low Mach":
        u, v = 1e-6 * u, 1e-6 * v
    elif kind == "units":                    # c = 340, E = 2.5e5: variables of unlike magnitude
        rho, u, v, p = 1.2 * rho, 300.0 * u, 200.0 * v, 1.0e5 * p
    elif kind == "supersonic":
        u = u - 8.0
    elif kind == "one jump":
        rho, u, v, p = np.where(np.arange(nx) < nx // 2, 1.0, 0.125) * one, 0 * one, 0 * one, np.where(np.arange(nx) < nx // 2, 1.0, 0.1) * one
    return np.ascontiguousarray(inputs.cons_from_prim(rho, u, p, v))


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["rest", "signed zeros", "tiny shear", "blast", "low Mach", "units", "supersonic", "one jump"])
def test_gpu_integer_projection(orc, kind):
    """The RHS at the suite's bound (1e-12 of its largest value, per variable), tile remainders."""
    import torch
    from paper_2004_07954_gb300 import build, wenozn as W
    build.build()
    for nx, ny in ((131, 9), (5, 35), (64, 33)):
        U = _state_2d(kind, nx, ny)
        p = W.wenozn_problem_init(2, nx, ny, 1.0 / nx, 1.0 / ny)
        got = W.Solver(p).rhs(torch.from_numpy(U).cuda()).cpu().numpy()
        want = orc.rhs(orc.problem(2, nx, ny, dx=1.0 / nx, dy=1.0 / ny), U)
        if kind in ("rest", "signed zeros"):
            assert np.abs(got).max() == 0.0
            continue
        for k in range(4):
            # rounding of the fluxes whose differences the RHS is: 1e-12 of the largest flux / dx
            scale = max(np.abs(want[k]).max(), 1e-3 * np.abs(want).max())
            assert np.abs(got[k] - want[k]).max() <= 1e-12 * scale, k


def _smooth_line(kind, n, dx):
    """Periodic 1D Euler states around the linear pass's acceptance: waves from well to badly
    resolved, alone, with jumps, with constant pieces, nearly incompressible, supersonic."""
    from paper_2004_07954_gb300 import inputs
    x = (np.arange(n) + 0.5) * dx
    g = np.random.default_rng(3)
    wave = lambda m, a: a * np.sin(2 * np.pi * m * x / (n * dx) + g.uniform(0, 6.28))
    m = {"waves": n // 200, "short waves": n // 20, "all waves": None}.get(kind, n // 100)
    if m is None:                            # every resolution from 1000 to 4 cells a wave
        rho = 1.0 + sum(wave(q, 0.02) for q in (n // 1000 + 1, n // 300, n // 100, n // 50, n // 30, n // 15, n // 4))
        u, p = 0.3 + wave(n // 80, 0.05), 1.0 + wave(n // 60, 0.05)
    else:
        rho, u, p = 1.0 + wave(m, 0.2), 0.4 + wave(m + 1, 0.2), 1.0 + wave(m + 2, 0.2)
    if kind == "jumps":
        rho, p = rho + (x > 0.3 * n * dx) + 2.0 * (x > 0.7 * n * dx), p + 3.0 * ((x > 0.5 * n * dx) & (x < 0.9 * n * dx))
    elif kind == "pieces":
        rho, u, p = np.where(np.sin(3e-3 * np.arange(n)) > 0, rho, 1.0), np.where(np.sin(3e-3 * np.arange(n)) > 0, u, 0.0), 1.0 + 0 * p
    elif kind == "entropy":
        u, p = 0.7 + 0 * u, 1.0 + 0 * p
    elif kind == "low Mach":
        u = 1e-4 * u
    elif kind == "supersonic":
        u = u + 6.0
    return np.ascontiguousarray(inputs.cons_from_prim(rho, u, p).reshape(3, 1, n))


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["waves", "short waves", "all waves", "jumps", "pieces", "entropy", "low Mach", "supersonic"])
def test_gpu_linear_pass(orc, kind):
    """Lines long enough for the linear pass (2^17 + 13 cells; the same states at 900 cells take the
    other kernels): the RHS against the oracle at the suite's 1e-12 of the flux scale over dx
    that the differences of the fluxes can carry, and the 2D sweeps of a repeated line."""
    import torch
    from paper_2004_07954_gb300 import build, wenozn as W
    build.build()
    dev = lambda a: torch.from_numpy(a).cuda()
    for n in (900, 131085):
        dx = 1.0 / 900
        U = _smooth_line(kind, n, dx)
        p = W.wenozn_problem_init(1, n, 1, dx, 1.0, bc_x=W.WENOZN_BC_PERIODIC)
        got = W.Solver(p).rhs(dev(U)).cpu().numpy()
        want = orc.rhs(orc.problem(1, n, 1, dx=dx, bc_x=W.WENOZN_BC_PERIODIC), U)
        for k in range(3):
            # (alpha U and, in the momentum's, the pressure) / dx, alpha < 10
            flux = (np.abs(U[k]).max() * 10.0 + (np.abs(U[2]).max() if k == 1 else 0.0)) / dx
            assert np.abs(got[k] - want[k]).max() <= 1e-14 * flux, (n, k)
    # both sweeps in 2D (1100 cells along, the line repeated across): the same values as in 1D
    n, m = 1100, 40
    U1 = _smooth_line(kind, n, 1.0 / n)
    p1 = W.wenozn_problem_init(1, n, 1, 1.0 / n, 1.0, bc_x=W.WENOZN_BC_PERIODIC)
    L1 = W.Solver(p1).rhs(dev(U1)).cpu().numpy()[:, 0]
    for axis in (0, 1):
        U = np.zeros((4, m, n))
        U[0], U[1 + axis], U[3] = U1[0], U1[1], U1[2]
        U = np.ascontiguousarray(U if axis == 0 else U.transpose(0, 2, 1))
        nx, ny = (n, m) if axis == 0 else (m, n)
        p = W.wenozn_problem_init(2, nx, ny, 1.0 / n, 1.0 / n, bc_x=W.WENOZN_BC_PERIODIC, bc_y=W.WENOZN_BC_PERIODIC)
        L = W.Solver(p).rhs(dev(U)).cpu().numpy()
        L = L if axis == 0 else L.transpose(0, 2, 1)
        for k, q in ((0, 0), (1 + axis, 1), (3, 2)):
            flux = (np.abs(U1[q]).max() * 10.0 + (np.abs(U1[2]).max() if q == 1 else 0.0)) * n
            assert np.abs(L[k] - L1[q]).max() <= 1e-14 * flux, (axis, k)


@pytest.mark.gpu
@pytest.mark.parametrize("split,weights,n", [(0, 0, 28271), (0, 0, 28272), (3, 0, 23559), (3, 0, 23560), (0, 1, 23559), (0, 1, 23560)])
def test_gpu_line_kernel_limits(orc, split, weights, n):
    """The longest lines of the one-launch stage kernel and the shortest beyond it: the RHS against
    the oracle, at the tolerance of test_gpu_linear_pass."""
    import torch
    from paper_2004_07954_gb300 import build, inputs, wenozn as W
    build.build()
    dx = 10.0 / n
    U = inputs.euler1d_ic(n, seed=5)
    p = W.wenozn_problem_init(1, n, 1, dx, 1.0, split=split, weights=weights)
    got = W.Solver(p).rhs(torch.from_numpy(U).cuda()).cpu().numpy()
    want = orc.rhs(orc.problem(1, n, 1, dx=dx, split=split, weights=weights), U)
    for k in range(3):
        flux = (np.abs(U[k]).max() * 10.0 + (np.abs(U[2]).max() if k == 1 else 0.0)) / dx
        assert np.abs(got[k] - want[k]).max() <= 1e-14 * flux, k
