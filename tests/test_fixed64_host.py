"""The fixed-point arithmetic of FP64 storage (csrc/fixed64.cuh), compiled for
the host, against the method's equations in extended precision.

Tolerance of an update: FP64 instructions make a chain of about ten roundings
of terms of at most 4 rho (the e and eps rows of Eq. 15), below 10 * 2^-53 *
4 rho = 4.4e-15 rho, and the fixed-point update is to be no worse.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_05110_gb300", "csrc")
UPDATE_TOL = 4.4e-15

SHIM = r"""
#include "fixed64.cuh"
using namespace vplbm;

// n nodes f[9]: the update into out (a node that is out of range: done = 0)
extern "C" int fx_host_update(const double *s, double rho0, double gx, double gy, double pen_k, long n, int chi,
                              const double *f, const double *us, double *out, double *acc, int *done)
{
    FixedConsts k;
    fold_fixed(k, s, rho0, gx, gy, pen_k);
    for (long m = 0; m < n; ++m) {
        uint64_t b[9];
        for (int a = 0; a < 9; ++a) b[a] = fx_bits(f[9 * m + a]);
        long long rho = 0, ax = 0, ay = 0;
        done[m] = k.ok && fx_update(k, b, chi != 0, llrint(ldexp(us[2 * m], 61)), llrint(ldexp(us[2 * m + 1], 61)), out + 9 * m,
                                    rho, ax, ay);
        acc[2 * m] = ldexp((double)ax, -60);
        acc[2 * m + 1] = ldexp((double)ay, -60);
    }
    return k.ok;
}

// n nodes (rho, ux, uy): the equilibrium's populations, or (dev) their deviations from w rho0
extern "C" void fx_host_equilibrium(double rho0, int dev, long n, const double *m, double *out, int *done)
{
    const double s[9] = {1, 1, 1, 1, 1, 1, 1, 1, 1};
    FixedConsts k;
    fold_fixed(k, s, rho0, 0.0, 0.0, 0.0);
    for (long q = 0; q < n; ++q) {
        long long v[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        done[q] = k.ok && fx_equilibrium(k, fx_bits(m[3 * q]), fx_bits(m[3 * q + 1]), fx_bits(m[3 * q + 2]), dev != 0, v);
        for (int a = 0; a < 9; ++a) out[9 * q + a] = ldexp((double)v[a], k.e - (dev ? 62 : 59));
    }
}

// the same deviations as floats; done: none is left to the FP64 instructions
extern "C" void fx_host_equilibrium_f32(double rho0, long n, const double *m, float *out, int *done)
{
    const double s[9] = {1, 1, 1, 1, 1, 1, 1, 1, 1};
    FixedConsts k;
    fold_fixed(k, s, rho0, 0.0, 0.0, 0.0);
    for (long q = 0; q < n; ++q) {
        long long v[9];
        bool near_tie = false;
        done[q] = k.ok && fx_equilibrium(k, fx_bits(m[3 * q]), fx_bits(m[3 * q + 1]), fx_bits(m[3 * q + 2]), true, v);
        for (int a = 0; a < 9 && done[q]; ++a) out[9 * q + a] = fx_signed_to_float(v[a], k.e - 62, near_tie);
        done[q] = done[q] && !near_tie;
    }
}

// the momentum that n nodes gain in an update, less rho g, per direction: its mean
extern "C" int fx_host_gain(const double *s, double gx, double gy, long n, const double *f, double *mean)
{
    FixedConsts k;
    fold_fixed(k, s, 1.0, gx, gy, 0.0);
    static const int cx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, cy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    long double px = 0, py = 0;
    for (long m = 0; m < n; ++m) {
        uint64_t b[9];
        double out[9];
        for (int a = 0; a < 9; ++a) b[a] = fx_bits(f[9 * m + a]);
        long long rho = 0, ax = 0, ay = 0;
        long double ex = 0, ey = 0, mass = 0;
        if (!k.ok || !fx_update(k, b, false, 0, 0, out, rho, ax, ay)) return 0;
        for (int a = 0; a < 9; ++a) {
            const long double d = (long double)out[a] - f[9 * m + a];
            ex += cx[a] * d;
            ey += cy[a] * d;
            mass += f[9 * m + a];
        }
        px += ex - mass * gx;
        py += ey - mass * gy;
    }
    mean[0] = (double)(px / n);
    mean[1] = (double)(py / n);
    return 1;
}

// n nodes of deviations d[9]: rho, u_x, u_y
extern "C" void fx_host_moments_dev(double rho0, long n, const float *d, double *out, int *done)
{
    const double s[9] = {1, 1, 1, 1, 1, 1, 1, 1, 1};
    FixedConsts k;
    fold_fixed(k, s, rho0, 0.0, 0.0, 0.0);
    for (long q = 0; q < n; ++q) done[q] = k.ok && fx_moments_dev(k, d + 9 * q, out[3 * q], out[3 * q + 1], out[3 * q + 2]);
}
"""

M = np.array([[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
              [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
              [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]])
C = np.array([[0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1]])
W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
LD = np.longdouble


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed64")
    src, lib = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    # arithmetic on the integers wraps, as it does on the device
    subprocess.run(["g++", "-O1", "-std=c++17", "-fwrapv", "-ffp-contract=off", "-fPIC", "-shared", f"-I{CSRC}", "-o", str(lib),
                    str(src)], check=True)
    return ctypes.CDLL(str(lib))


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _rates(tau=0.7, **other):
    s = [1 / tau, 1.1, 1.25, 1 / tau, 1.8, 1 / tau, 1.8, 1 / tau, 1 / tau]
    for k, v in other.items():
        s[int(k[1:])] = v
    return np.array(s)


def _nodes(n, rho0, seed, amp=0.1):
    rng = np.random.default_rng(seed)
    u = rng.uniform(-amp, amp, (2, n))
    rho = rho0 * (1 + 0.02 * rng.uniform(-1, 1, n))
    cu = C.T @ u
    f = W[:, None] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0)) * (1 + 1e-3 * rng.uniform(-1, 1, (9, n)))
    return np.ascontiguousarray(f.T), np.ascontiguousarray(rng.uniform(-0.05, 0.05, (n, 2)))


def _update(host, f, us, s, rho0=1.0, g=(0.0, 0.0), eta=None):
    n = len(f)
    out, acc, done = np.zeros((n, 9)), np.zeros((n, 2)), np.zeros(n, np.int32)
    pen = 0.0 if eta is None else 1.0 / (eta + 0.5)
    host.fx_host_update(_ptr(s), ctypes.c_double(rho0), ctypes.c_double(g[0]), ctypes.c_double(g[1]), ctypes.c_double(pen),
                        ctypes.c_long(n), int(eta is not None), _ptr(f), _ptr(us), _ptr(out), _ptr(acc), _ptr(done))
    return out, acc, done.astype(bool)


def _exact(f, us, s, g=(0.0, 0.0), eta=None):
    """Collision with forcing (Eqs. 14-17, 22) of each node in extended precision."""
    f = f.T.astype(LD)
    m = M.astype(LD) @ f
    rho, j = m[0], m[[3, 5]]
    g = np.array(g, LD)[:, None]
    u = j / rho + g / 2
    a = np.zeros_like(u)
    if eta is not None:
        a = (us.T.astype(LD) - u) / (LD(eta) + LD(0.5))
        u = u + a / 2
    G = rho * (g + a)
    u2, uG = (u * u).sum(0), (u * G).sum(0)
    eq = np.array([rho, -2 * rho + 3 * rho * u2, rho - 3 * rho * u2, m[3], -rho * u[0], m[5], -rho * u[1],
                   rho * (u[0] ** 2 - u[1] ** 2), rho * u[0] * u[1]])
    F = np.array([0 * rho, 6 * uG, -6 * uG, G[0], -G[0], G[1], -G[1], 2 * (u[0] * G[0] - u[1] * G[1]), u[0] * G[1] + u[1] * G[0]])
    sk = s.astype(LD)[:, None].copy()
    sk[[0, 3, 5]] = 0
    d = sk * (eq - m) + (1 - sk / 2) * F
    return (f + (M / (M * M).sum(1)[:, None].astype(LD)).T.astype(LD) @ d).T, a.T


@pytest.mark.parametrize("eta", [1e-3, 1e-9, 1.2e-10, 1.1e-10, 1e-12, 1e-20])
@pytest.mark.parametrize("rho0", [1.0, 0.7])
def test_penalization_factor_of_every_eta(host, eta, rho0):
    f, us = _nodes(500, rho0, 1)
    out, acc, done = _update(host, f, us, _rates(), rho0, eta=eta)
    assert done.all()   # in fixed point, at any eta
    want, a = _exact(f, us, _rates(), eta=eta)
    assert np.max(np.abs(acc - a)) < 1e-15
    assert np.max(np.abs(out - want)) < UPDATE_TOL * 1.1 * rho0


@pytest.mark.parametrize("rates", [{"s7": 2 - 1e-10}, {"s8": 2 - 1e-10}, {"s7": 1e-10}, {"s8": 1e-10}, {"s7": 2 - 1e-9},
                                   {"s7": 1e-9}, {"s1": 2 - 1e-15, "s4": 1e-15}])
@pytest.mark.parametrize("g", [(0.0, 0.0), (1e-3, -2e-3)])
@pytest.mark.parametrize("eta", [None, 1e-3])
def test_rates_at_the_ends_of_their_range(host, rates, g, eta):
    """Rates in (0, 2) up to its ends: the right update, or left to the FP64 instructions."""
    f, us = _nodes(500, 1.0, 2)
    s = _rates(**rates)
    out, _, done = _update(host, f, us, s, g=g, eta=eta)
    want, _ = _exact(f, us, s, g=g, eta=eta)
    assert np.max(np.abs(out - want)[done], initial=0.0) < UPDATE_TOL * 1.1


@pytest.mark.parametrize("dev", [False, True])
@pytest.mark.parametrize("rho0", [1.0, 0.99, 0.7, 0.51])
def test_equilibrium_over_the_accepted_velocities(host, dev, rho0):
    """All of |u_x|, |u_y| < 1/4 and densities around rho0: the right value, or left to the FP64 instructions.  FP64
    instructions round terms of at most 4 rho about ten times."""
    u = np.linspace(-0.2499, 0.2499, 41)
    rho = rho0 * np.array([0.9, 0.95, 0.999, 1.0, 1.003, 1.04])
    m = np.array([(r, x, y) for r in rho for x in u for y in u])
    out, done = np.zeros((len(m), 9)), np.zeros(len(m), np.int32)
    host.fx_host_equilibrium(ctypes.c_double(rho0), int(dev), ctypes.c_long(len(m)), _ptr(m), _ptr(out), _ptr(done))
    r, ux, uy = m.T.astype(LD)
    cu = C[0][:, None] * ux + C[1][:, None] * uy
    w = np.array([LD(4) / 9] + [LD(1) / 9] * 4 + [LD(1) / 36] * 4)[:, None]
    want = w * ((r - LD(rho0) if dev else r) + r * (3 * cu + LD(4.5) * cu * cu - LD(1.5) * (ux * ux + uy * uy)))
    done = done.astype(bool)
    near = np.abs(m[:, 0] / rho0 - 1) < 4e-3
    assert done[near & (np.abs(m[:, 1:]).max(1) < 0.19)].all()   # a low-Mach flow stays in fixed point
    assert np.max(np.abs(out.T - want)[:, done]) < UPDATE_TOL * 1.04 * rho0


def test_equilibrium_deviations_of_slow_nodes(host):
    """Velocities down to the smallest: a float that is not the rounded one is left to the FP64 instructions."""
    rng = np.random.default_rng(6)
    n = 4000
    u = 10.0 ** rng.uniform(-30, -1, (n, 2)) * rng.choice([-1, 1], (n, 2))
    u[:500, 1] = 0.0
    rho = 1 + np.where(rng.uniform(size=n) < 0.5, 0.0, 10.0 ** rng.uniform(-16, -2, n))
    m = np.ascontiguousarray(np.column_stack([rho, u]))
    out, done = np.zeros((n, 9), np.float32), np.zeros(n, np.int32)
    host.fx_host_equilibrium_f32(ctypes.c_double(1.0), ctypes.c_long(n), _ptr(m), _ptr(out), _ptr(done))
    r, ux, uy = m.T.astype(LD)
    cu = C[0][:, None] * ux + C[1][:, None] * uy
    w = np.array([LD(4) / 9] + [LD(1) / 9] * 4 + [LD(1) / 36] * 4)[:, None]
    want = w * ((r - 1) + r * (3 * cu + LD(4.5) * cu * cu - LD(1.5) * (ux * ux + uy * uy)))
    done = done.astype(bool)
    assert done[np.abs(u).max(1) > 1e-3].mean() > 0.98   # a flow at speed stays in fixed point
    assert np.array_equal(out.T[:, done], want.astype(np.float32)[:, done])


@pytest.mark.parametrize("rho0", [1.0, 0.7, 0.51])
@pytest.mark.parametrize("spread", [0, 3, 9, 30])
def test_fields_of_deviations_of_any_size(host, rho0, spread):
    """rho and u of FP32 / FP16 storage: a deviation has its 24 bits whatever its size, so u has the precision of a double
    (2^-53 for the rounding, 2^-56 for the quotient), or the node is left to the FP64 instructions."""
    rng = np.random.default_rng(8)
    n = 20000
    size = 10.0 ** rng.uniform(-30, -1.3, n)
    d = (size[:, None] * 10.0 ** -rng.uniform(0, spread, (n, 9)) * rng.uniform(-1, 1, (n, 9))).astype(np.float32)
    d[rng.uniform(size=(n, 9)) < 0.05] = 0
    d[::50] = 0                                     # at rest
    d[1::50, 3], d[1::50, 1] = d[1::50, 1], d[1::50, 1] * np.float32(1 + 2.0 ** -20)   # the sums cancel
    d[1::50, 5:] = 0
    d = np.ascontiguousarray(d)
    out, done = np.zeros((n, 3)), np.zeros(n, np.int32)
    host.fx_host_moments_dev(ctypes.c_double(rho0), ctypes.c_long(n), _ptr(d), _ptr(out), _ptr(done))
    done = done.astype(bool)
    f = d.T.astype(LD)
    jx, jy = f[1] - f[3] + (f[5] - f[6]) + (f[8] - f[7]), f[2] - f[4] + (f[5] + f[6]) - (f[7] + f[8])
    rho = LD(rho0) + f.sum(0)
    for got, want in zip(out.T, (rho, jx / rho, jy / rho)):
        assert np.all(np.abs(got - want)[done] <= 1.3e-16 * np.abs(want)[done])
    inside = (size > 1e-25) & (rho > 0.5)           # the density's range is [2^(E-1), 1.5 2^E)
    if spread < 9:                                  # nearly all within 2^34 of the node's largest
        assert done[inside].mean() > 0.999
    rest = out[::50][done[::50]]
    assert np.all(rest == [rho0, 0.0, 0.0])


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 0.2, 1e-42])
def test_fields_of_deviations_out_of_range_are_left_to_fp64(host, value):
    d = np.full((9, 9), 1e-3, np.float32)
    d[np.arange(9), np.arange(9)] = value
    out, done = np.zeros((9, 3)), np.ones(9, np.int32)
    host.fx_host_moments_dev(ctypes.c_double(1.0), ctypes.c_long(9), _ptr(d), _ptr(out), _ptr(done))
    assert not done.any()


@pytest.mark.parametrize("g", [(1e-6, 3e-7), (1e-9, -2e-9), (1e-12, 1e-12), (1e-12, 7e-13), (-1e-14, 1e-16), (1e-20, 0.06),
                               (0.0624, 1e-19), (0.0, -1e-17), (0.01, 0.0)])
def test_momentum_gained_from_a_uniform_acceleration(host, g):
    """rho g per node and step without a bias: the mean over n nodes of the update's rounding, which is at most 1e-17 rho a
    node (the doubles that are stored: two of 2^-57, four of 2^-59; units of 2^-60 in the force).  An acceleration that
    the grid does not hold is left to the FP64 instructions, but for a component within 2^-50 of the other's rounding."""
    n = 300000
    f, _ = _nodes(n, 1.0, 10)
    mean = np.zeros(2)
    s = _rates()
    done = host.fx_host_gain(_ptr(s), ctypes.c_double(g[0]), ctypes.c_double(g[1]), ctypes.c_long(n), _ptr(f), _ptr(mean))
    assert done == (max(map(abs, g)) > 2.0 ** -40 and (min(map(abs, g)) > 2.0 ** -40 or min(map(abs, g)) <= 2.0 ** -50 * max(map(abs, g))))
    if done:
        assert np.max(np.abs(mean)) < 5 * 1e-17 / np.sqrt(n) + 2.0 ** -50 * max(map(abs, g))
