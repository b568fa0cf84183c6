// The FP64 path's MRT update in 64-bit fixed point on the integer pipes.
//
// What bounds it: GB300 issues two FP64 lanes per clock and SM, so the 111
// FP64 instructions of the update kept that pipe busy for 55 clocks per node
// and nothing else mattered (4.1 k MLUPS on 2048 x 1024, 9 % of the HBM
// rate).  The integer pipes are 32 to 64 times as wide, and a node's
// populations share one scale (they are fractions of rho ~ rho0), so the
// update runs on integers: additions are exact, a product is three 32-bit
// wide multiplies, and the collision is written as f + M^-1 (dm), which
// needs six products with the relaxation rates, five for the velocity and
// the quadratic terms, and one reciprocal.
//
// Numbers.  A population f is the integer x = f 2^(59 - E), 2^E >= rho0 >
// 2^(E-1): the grid is 2^-59 of that scale, at or below the spacing of the
// doubles it is read from for f >= 2^(E-7) (an ordinary diagonal population
// is rho0 / 36), so the read is exact there.  Every product is rounded to
// the nearest grid point (plus at most one more unit), the results are
// rounded to doubles to nearest even.  The collision's increments conserve
// mass, and without forcing momentum, exactly.  Its error against exact
// arithmetic is a third of that of the FP64 instructions it replaces (RMS
// over the populations of an update at rho0 = 1, in 113-bit arithmetic:
// 0.7e-17 against 2.2e-17, most of it the final rounding to double).
//
// Measured (GB300, us per step, best block shape): 2048 x 1024 513 -> 63.5
// (32.9 k MLUPS, 4.7 TB/s), 256 x 128 28 -> 13.5 (there the launch boundary
// and the body's sums remain); 2048 x 1024 under a uniform
// acceleration 110.
//
// Range.  A node takes this path if every population is in
// [2^(E-32), 2^E), rho in [2^(E-1), 1.5 2^E), |j| < 0.35 2^E and (body
// nodes) the slip |u_s - v| < 1/4, and if every result is at least
// 2^(E-27); sums and products then stay below 2^63.  Any other node (a
// negative population, a density far from rho0, NaN, infinities) takes the
// FP64 instructions, which accept everything.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define VPLBM_FX __host__ __device__ __forceinline__
#else
#define VPLBM_FX inline
#endif

namespace vplbm {
namespace {

// A factor r as r = hi 2^-32 + lo 2^-64 with signed digits, which hold
// -1/2 <= r < 1/2 - 2^-33.
struct FxFactor {
    int hi, lo;
};

// The factor of a double in (0, 1/2) known at compile time.
constexpr FxFactor fx_const(double r)
{
    const long long v = (long long)(r * 0x1p64);   // exact: 53 bits
    const int lo = (int)(uint32_t)(uint64_t)v;
    return {(int)((v - (long long)lo) >> 32), lo};
}
constexpr FxFactor FX_W0 = fx_const(4.0 / 9.0), FX_W1 = fx_const(1.0 / 9.0), FX_W2 = fx_const(1.0 / 36.0);

// Host-folded constants of the fixed-point update (uniform over a run).
struct FixedConsts {
    int ok;                     // the run's rho0, g and factors are in range
    int e;                      // E
    double unit;                // 2^(E - 59)
    unsigned hi_min, hi_max;    // high words of the doubles in [2^(E-32), 2^E)
    FxFactor r1, r2, r4, r6, r7, r8;   // s1/36, s2/12, s4/12, s6/12, s7/4, s8/4
    // forcing: (1 - s/2) / 6 for e and eps, / 12 for q, / 2 and / 4 for the
    // stress, 1/6, and pen_k / 8 (pen_k = 1 / (eta + 1/2) tends to 2)
    FxFactor h1, h2, h4, h6, h7, h8, sixth, k8;
    long long gvx, gvy;         // g 2^60, for the velocity j / rho + g / 2
    // g / 48 for the force rho g / 6 that a population takes, to 2^-96 (from g
    // 2^60 it would be off by up to 4e-19, every step with the same sign)
    FxFactor gx, gy;
    int gx3, gy3;               // its third digits (2^-96)
    int forced;                 // g is not zero
    long long rho0;             // in units of 2^(E - 59)
};

// ok is cleared where the digits do not hold r.
inline FxFactor fx_factor(double r, int &ok)
{
    FxFactor f = {0, 0};
    if (!(fabs(r) <= 0.5 - 0x1p-32)) {
        ok = 0;
        return f;
    }
    const long long v = llrint(ldexp(r, 64));
    f.lo = (int)(uint32_t)(uint64_t)v;
    f.hi = (int)((v - (long long)f.lo) >> 32);
    return f;
}

// g / 48 and its third digit.  other: the other component.  A force of a few
// units or less is not rounded without a bias (a uniform density rounds it the
// same way everywhere): below 2^-40 the run takes the FP64 instructions, but
// for a component that is only the other's rounding (a direction at right
// angles computed by cos).
inline FxFactor fx_accel(double g, double other, int &third, int &ok)
{
    if (g != 0.0 && fabs(g) < 0x1p-40 && !(fabs(g) <= 0x1p-50 * fabs(other))) ok = 0;
    const double r = g / 48.0, rest = ldexp(r, 64) - rint(ldexp(r, 64));
    third = (int)fmin(rint(ldexp(rest, 32)), 2147483647.0);
    return fx_factor(r, ok);
}

inline void fold_fixed(FixedConsts &k, const double *s, double rho0, double gx, double gy, double pen_k)
{
    memset(&k, 0, sizeof k);
    int e = 0;
    const double m = frexp(rho0, &e);   // rho0 = m 2^e, m in [1/2, 1)
    if (m == 0.5) e -= 1;               // rho0 in (2^(E-1), 2^E]
    if (!(rho0 > 0.0) || e < -400 || e > 400 || !(fabs(gx) < 0.0625) || !(fabs(gy) < 0.0625)) return;
    k.e = e;
    k.unit = ldexp(1.0, e - 59);
    k.hi_min = (unsigned)(991 + e) << 20;
    k.hi_max = (unsigned)(1023 + e) << 20;
    // a rate s_7 or s_8 within 2^-30 of 2, or an s_7 below 2^-30, makes a
    // factor that does not fit; such a run takes the FP64 instructions
    int ok = 1;
    k.r1 = fx_factor(s[1] / 36.0, ok); k.r2 = fx_factor(s[2] / 12.0, ok); k.r4 = fx_factor(s[4] / 12.0, ok);
    k.r6 = fx_factor(s[6] / 12.0, ok); k.r7 = fx_factor(s[7] / 4.0, ok); k.r8 = fx_factor(s[8] / 4.0, ok);
    k.h1 = fx_factor((1.0 - 0.5 * s[1]) / 6.0, ok); k.h2 = fx_factor((1.0 - 0.5 * s[2]) / 6.0, ok);
    k.h4 = fx_factor((1.0 - 0.5 * s[4]) / 12.0, ok); k.h6 = fx_factor((1.0 - 0.5 * s[6]) / 12.0, ok);
    k.h7 = fx_factor((1.0 - 0.5 * s[7]) / 2.0, ok); k.h8 = fx_factor((1.0 - 0.5 * s[8]) / 4.0, ok);
    k.sixth = fx_factor(1.0 / 6.0, ok);
    k.k8 = fx_factor(0.125 * pen_k, ok);
    k.gvx = llrint(ldexp(gx, 60));
    k.gvy = llrint(ldexp(gy, 60));
    k.gx = fx_accel(gx, gy, k.gx3, ok);
    k.gy = fx_accel(gy, gx, k.gy3, ok);
    k.forced = gx != 0.0 || gy != 0.0;
    k.rho0 = llrint(ldexp(rho0, 59 - e));
    k.ok = ok;
}

VPLBM_FX int fx_clz(uint32_t x)
{
#if defined(__CUDA_ARCH__)
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}

VPLBM_FX int fx_clz64(uint64_t x)
{
    const uint32_t hi = (uint32_t)(x >> 32);
    return hi ? fx_clz(hi) : 32 + fx_clz((uint32_t)x);
}

VPLBM_FX uint64_t fx_bits(double d)
{
#if defined(__CUDA_ARCH__)
    return (uint64_t)__double_as_longlong(d);
#else
    uint64_t b;
    memcpy(&b, &d, 8);
    return b;
#endif
}

VPLBM_FX double fx_double(uint64_t b)
{
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)b);
#else
    double d;
    memcpy(&d, &b, 8);
    return d;
#endif
}

VPLBM_FX uint32_t fx_float_bits(float f)
{
#if defined(__CUDA_ARCH__)
    return __float_as_uint(f);
#else
    uint32_t b;
    memcpy(&b, &f, 4);
    return b;
#endif
}

// 2^k, -126 <= k <= 127.
VPLBM_FX float fx_pow2f(int k)
{
    const uint32_t b = (uint32_t)(127 + k) << 23;
#if defined(__CUDA_ARCH__)
    return __uint_as_float(b);
#else
    float f;
    memcpy(&f, &b, 4);
    return f;
#endif
}

VPLBM_FX FxFactor fx_split(long long r)
{
    FxFactor f;
    f.lo = (int)(uint32_t)(uint64_t)r;
    f.hi = (int)(r >> 32) + (int)((uint32_t)f.lo >> 31);
    return f;
}

// x r to the nearest integer but for the product of the two low digits
// (below half a unit); |x| < 2^63.
VPLBM_FX long long fx_mul(long long x, FxFactor r)
{
    const FxFactor a = fx_split(x);
    const long long m = (long long)a.lo * r.hi + 0x80000000LL + (long long)a.hi * r.lo;
    return (long long)a.hi * r.hi + (m >> 32);
}

// The same with a third digit (2^-96) of r.
VPLBM_FX long long fx_mul3(long long x, FxFactor r, int third)
{
    const FxFactor a = fx_split(x);
    const long long m = (long long)a.lo * r.hi + 0x80000000LL + (long long)a.hi * r.lo + (((long long)a.hi * third) >> 32);
    return (long long)a.hi * r.hi + (m >> 32);
}

// The double with bits b, in [2^(E-32), 2^E), on the grid (truncated).
VPLBM_FX long long fx_from(uint64_t b, int e)
{
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
    const uint32_t s = (uint32_t)(1022 + e) - (hi >> 20);   // 0 .. 31 in range
    const uint32_t mh = (((hi << 6) | (lo >> 26)) & 0x3ffffffu) | 0x4000000u, ml = lo << 6;
#if defined(__CUDA_ARCH__)
    const uint32_t rl = __funnelshift_r(ml, mh, s), rh = mh >> (s & 31);
#else
    const uint64_t m = ((((uint64_t)mh) << 32) | ml) >> (s & 31);
    const uint32_t rl = (uint32_t)m, rh = (uint32_t)(m >> 32);
#endif
    return (long long)(((uint64_t)rh << 32) | rl);
}

// The grid point x in [2^32, 2^61) as a double, to nearest even.
VPLBM_FX double fx_to(long long x, int e)
{
    const uint32_t hi = (uint32_t)((uint64_t)x >> 32), lo = (uint32_t)(uint64_t)x;
    const uint32_t n = (uint32_t)fx_clz(hi) - 1;   // leading bit to bit 62
#if defined(__CUDA_ARCH__)
    const uint32_t yh = __funnelshift_l(lo, hi, n), yl = lo << (n & 31);
#else
    const uint64_t yy = ((((uint64_t)hi) << 32) | lo) << n;
    const uint32_t yh = (uint32_t)(yy >> 32), yl = (uint32_t)yy;
#endif
    uint64_t y = ((uint64_t)yh << 32) | yl;
    y += 0x1ffu + ((yl >> 10) & 1u);
    y >>= 10;
    return fx_double(y + ((uint64_t)((uint32_t)(1025 + e - (int)n) << 20) << 32));
}

// 2^120 / rho for rho in [2^58, 2^60), relative error below 2^-60: a 32-bit
// estimate from the FP32 reciprocal, then 1 / (1 - d) = 1 + d + d^2 with the
// exact residual d.
VPLBM_FX long long fx_recip(long long rho)
{
    const uint32_t rh = (uint32_t)((uint64_t)rho >> 32), rl = (uint32_t)(uint64_t)rho;
    const float rf = (float)(uint32_t)((uint64_t)rho >> 28);   // rho 2^-28
#if defined(__CUDA_ARCH__)
    float inv;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(inv) : "f"(rf));
#else
    const float inv = 1.0f / rf;
#endif
    const uint32_t r0 = (uint32_t)(inv * 1152921504606846976.0f);   // 2^60 / (rho 2^-28) = 2^88 / rho
    // d = (2^88 - rho r0) / 2^16, the residual in units of 2^-72: |d| < 2^52
    const uint64_t pl = (uint64_t)rl * r0;
    const uint64_t ph = (uint64_t)rh * r0 + (pl >> 32);
    long long d = -(long long)((ph << 16) | ((uint32_t)pl >> 16));
    const long long dh = (int)(d >> 32);
    d += (dh * dh) >> 8;
    const long long lo = (long long)((uint64_t)r0 * (uint32_t)(uint64_t)d >> 32);
    return (long long)((uint64_t)r0 << 32) + (((long long)(int)(d >> 32) * (long long)r0 + lo) >> 8);
}

// The part of the update that a penalized node (or a lattice under a uniform
// acceleration) does differently, a function of its own on the device: few
// nodes take it, and inlined it costs the others registers.  In: the moments
// (v: velocity times 2^61) and the solid velocity us; out: the increments
// along the rows of M and G / 6, and a 2^60 of the penalization.  False if
// the slip is out of range.
struct FxForced {
    long long rho, jx, jy, vx, vy, usx, usy, f0, sa, sd, qx, qy, pxx, pxy;   // in
    long long de, dep, dqx, dqy, dp, dr, gx6, gy6, ax, ay;                   // out
};

// G: the lattice may be under a uniform acceleration.
template <bool G>
VPLBM_FX bool fx_forced_here(const FixedConsts &k, bool chi, FxForced &w)
{
    const long long gx = G ? k.gvx : 0, gy = G ? k.gvy : 0;
    const long long wx = w.vx + gx, wy = w.vy + gy;   // v = j / rho + g / 2
    long long ax = 0, ay = 0;                               // a 2^60
    if (chi) {
        const long long lx = w.usx - wx, ly = w.usy - wy;
        constexpr long long Q = 1LL << 59;
        if ((uint64_t)(lx + Q) >= (uint64_t)(2 * Q) || (uint64_t)(ly + Q) >= (uint64_t)(2 * Q)) return false;
        ax = fx_mul(4 * lx, k.k8);   // |4 l| < 2^61
        ay = fx_mul(4 * ly, k.k8);
    }
    const FxFactor ux = fx_split(wx + ax), uy = fx_split(wy + ay);   // u = v + a / 2
    const long long r8 = (long long)((uint64_t)w.rho << 3);
    const long long Gx = fx_mul(r8, fx_split(2 * (ax + gx))), Gy = fx_mul(r8, fx_split(2 * (ay + gy)));
    if (!G || !k.forced) {
        w.gx6 = fx_mul(Gx, k.sixth);
        w.gy6 = fx_mul(Gy, k.sixth);
    } else {
        // rho g / 6 in one rounding: that of a sixth of Gx, a whole number,
        // favours the sign of g (it is halfway one time in six)
        w.gx6 = fx_mul3(r8, k.gx, k.gx3);
        w.gy6 = fx_mul3(r8, k.gy, k.gy3);
        if (chi) {
            w.gx6 += fx_mul(fx_mul(r8, fx_split(2 * ax)), k.sixth);
            w.gy6 += fx_mul(fx_mul(r8, fx_split(2 * ay)), k.sixth);
        }
    }
    const long long mx = w.jx + (Gx >> 1), my = w.jy + (Gy >> 1);    // rho u = j + G / 2
    const long long mx8 = (long long)((uint64_t)mx << 3), my8 = (long long)((uint64_t)my << 3);
    const long long A = fx_mul(mx8, ux), B = fx_mul(my8, uy), C = fx_mul(mx8, uy);
    const long long Gx8 = (long long)((uint64_t)Gx << 3), Gy8 = (long long)((uint64_t)Gy << 3);
    const long long xx = fx_mul(Gx8, ux), yy = fx_mul(Gy8, uy), xy = fx_mul(Gy8, ux) + fx_mul(Gx8, uy);
    const long long K = A + B;
    w.de = fx_mul(2 * w.f0 - w.sa - 4 * w.sd + 3 * K, k.r1) + fx_mul(xx + yy, k.h1);
    w.dep = fx_mul(w.sa - w.f0 - K, k.r2) - fx_mul(xx + yy, k.h2);
    w.dqx = fx_mul(w.qx - (Gx >> 1), k.r4) - fx_mul(Gx, k.h4);
    w.dqy = fx_mul(w.qy - (Gy >> 1), k.r6) - fx_mul(Gy, k.h6);
    w.dp = fx_mul(A - B - w.pxx, k.r7) + fx_mul(xx - yy, k.h7);
    w.dr = fx_mul(C - w.pxy, k.r8) + fx_mul(xy, k.h8);
    w.ax = ax;
    w.ay = ay;
    return true;
}

#if defined(__CUDACC__)
__device__ __noinline__
#else
inline
#endif
bool fx_forced(const FixedConsts &k, bool chi, FxForced &w) { return fx_forced_here<true>(k, chi, w); }

// One node: pulled populations f (bits of doubles) -> post-collision
// populations out.  chi: the node is in a body of solid velocity us (times
// 2^61).  Returns false (out untouched) if the node is out of range; rho and
// a 2^60 (the penalization's acceleration) are kept for the body's sums.
// HERE: a caller of solid nodes only, without a uniform acceleration, has the
// penalized part inlined.
template <bool HERE = false>
#if defined(__CUDACC__)
__device__ __forceinline__
#else
inline
#endif
bool fx_update(const FixedConsts &k, const uint64_t fb[9], bool chi, long long usx, long long usy,
                        double out[9], long long &rho_o, long long &ax_o, long long &ay_o)
{
    uint32_t top = 0, low = 0xffffffffu;
    long long f[9];
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int a = 0; a < 9; ++a) {
        const uint32_t hi = (uint32_t)(fb[a] >> 32);
        top = hi > top ? hi : top;
        low = hi < low ? hi : low;
        f[a] = fx_from(fb[a], k.e);
    }
    bool ok = top < k.hi_max && low >= k.hi_min;
    const long long d13 = f[1] - f[3], d24 = f[2] - f[4], b13 = f[1] + f[3], b24 = f[2] + f[4];
    const long long d56 = f[5] - f[6], d87 = f[8] - f[7], a56 = f[5] + f[6], a78 = f[7] + f[8];
    const long long sx = d56 + d87, ty = a56 - a78, sa = b13 + b24, sd = a56 + a78;
    const long long rho = f[0] + sa + sd;
    const long long jx = d13 + sx, jy = d24 + ty;
    constexpr long long J = 201769274521386496LL;   // 0.35 2^59
    ok = ok && (uint64_t)(rho - (1LL << 58)) < (uint64_t)(1LL << 59) && (uint64_t)(jx + J) < (uint64_t)(2 * J) &&
         (uint64_t)(jy + J) < (uint64_t)(2 * J);
    if (!ok) return false;
    const FxFactor inv = fx_split(fx_recip(rho));
    const long long vx = fx_mul((long long)((uint64_t)jx << 5), inv), vy = fx_mul((long long)((uint64_t)jy << 5), inv);   // u 2^61
    long long de, dep, dqx = d13 - 2 * sx, dqy = d24 - 2 * ty, dp, dr;
    long long gx6 = 0, gy6 = 0;
    if (chi || k.forced) {
        FxForced w;
        w.rho = rho; w.jx = jx; w.jy = jy; w.vx = vx; w.vy = vy; w.usx = usx; w.usy = usy;
        w.f0 = f[0]; w.sa = sa; w.sd = sd; w.qx = dqx; w.qy = dqy; w.pxx = b13 - b24; w.pxy = d56 - d87;
        if (!(HERE ? fx_forced_here<false>(k, chi, w) : fx_forced(k, chi, w))) return false;
        de = w.de; dep = w.dep; dqx = w.dqx; dqy = w.dqy; dp = w.dp; dr = w.dr;
        gx6 = w.gx6; gy6 = w.gy6;
        ax_o = w.ax;
        ay_o = w.ay;
    } else {
        const FxFactor ux = fx_split(vx), uy = fx_split(vy);
        const long long jx8 = (long long)((uint64_t)jx << 3), jy8 = (long long)((uint64_t)jy << 3);
        const long long A = fx_mul(jx8, ux), B = fx_mul(jy8, uy), C = fx_mul(jx8, uy);   // rho ux^2, uy^2, ux uy
        const long long K = A + B;
        de = fx_mul(2 * f[0] - sa - 4 * sd + 3 * K, k.r1);
        dep = fx_mul(sa - f[0] - K, k.r2);
        dqx = fx_mul(dqx, k.r4);
        dqy = fx_mul(dqy, k.r6);
        dp = fx_mul(A - B - (b13 - b24), k.r7);
        dr = fx_mul(C - (d56 - d87), k.r8);
    }
    // M^-1 dm: the rows of Eq. (15) over their squared norms
    const long long ax1 = -de - 2 * dep, dg = 2 * de + dep;
    const long long x1 = gx6 - 2 * dqx, y1 = gy6 - 2 * dqy, x2 = gx6 + dqx, y2 = gy6 + dqy;
    const long long p1 = ax1 + dp, p2 = ax1 - dp, q1 = dg + dr, q2 = dg - dr;
    const long long s2 = x2 + y2, m2 = x2 - y2;
    f[0] += 4 * (dep - de);
    f[1] += p1 + x1;
    f[3] += p1 - x1;
    f[2] += p2 + y1;
    f[4] += p2 - y1;
    f[5] += q1 + s2;
    f[7] += q1 - s2;
    f[8] += q2 + m2;
    f[6] += q2 - m2;
    int lo = (int)(f[0] >> 32);
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int a = 1; a < 9; ++a) {
        const int h = (int)(f[a] >> 32);
        lo = h < lo ? h : lo;
    }
    if (lo < 1) return false;
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int a = 0; a < 9; ++a) out[a] = fx_to(f[a], k.e);
    rho_o = rho;
    return true;
}

// ---- fields and equilibria ------------------------------------------------

// x 2^k as a double, to nearest even, for any x.
VPLBM_FX double fx_signed_to(long long x, int k)
{
    if (x == 0) return 0.0;
    const uint64_t sign = (uint64_t)x & 0x8000000000000000ull, m = x < 0 ? 0 - (uint64_t)x : (uint64_t)x;
    const int n = fx_clz64(m);
    const uint64_t y = m << n;   // leading bit at 63
    const uint64_t q = y >> 11, half = (y >> 10) & 1, rest = (y & 0x3ff) | (q & 1);
    return fx_double(sign | ((q + (half & (rest != 0))) + ((uint64_t)(1023 + 63 - 1 + k - n) << 52)));
}

// x 2^k as a float, to nearest, for |x| < 2^62 and a result in the normal
// range.  near_tie is set where x is within 512 units of halfway between two
// floats (FP64 arithmetic, whose error is below that, could round the other
// way there), and where x is too small for the float's digits or zero (what
// was rounded to zero need not be).
VPLBM_FX float fx_signed_to_float(long long x, int k, bool &near_tie)
{
    if (x == 0) {
        near_tie = true;
        return 0.f;
    }
    const uint64_t m = x < 0 ? 0 - (uint64_t)x : (uint64_t)x;
    const int n = fx_clz64(m);
    const uint64_t y = m << n;
    const long long off = (long long)(y & 0xffffffffffull) - (1LL << 39);   // from halfway
    near_tie = near_tie || n >= 30 || (off < 0 ? -off : off) <= (512LL << n);
    const uint32_t t = (uint32_t)(y >> 32) | ((uint32_t)y != 0);   // the leading 32 bits, the rest sticky
    const float f = (float)t * fx_pow2f(k + 32 - n);
    return x < 0 ? -f : f;
}

// A double of magnitude below 1/4 times 2^61, to nearest even.
VPLBM_FX long long fx_from_signed(uint64_t b)
{
    const uint64_t m = ((b & 0xfffffffffffffull) | (1ull << 52)) << 10;
    const uint32_t s = 1024u - (uint32_t)((b >> 52) & 0x7ff);   // 3 or more
    if (s > 63) return 0;
    const uint64_t q = m >> s, half = (m >> (s - 1)) & 1, rest = (m << (65 - s)) | (q & 1);
    const uint64_t x = q + (half & (rest != 0));
    return (long long)b < 0 ? -(long long)x : (long long)x;
}

// rho and u of nine pulled populations away from the body, without a uniform
// acceleration: FP64 storage.  False if the node is out of range.
VPLBM_FX bool fx_moments(const FixedConsts &k, const uint64_t fb[9], double &rho_o, double &ux_o, double &uy_o)
{
    uint32_t top = 0, low = 0xffffffffu;
    long long f[9];
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int a = 0; a < 9; ++a) {
        const uint32_t hi = (uint32_t)(fb[a] >> 32);
        top = hi > top ? hi : top;
        low = hi < low ? hi : low;
        f[a] = fx_from(fb[a], k.e);
    }
    if (top >= k.hi_max || low < k.hi_min) return false;
    const long long sx = f[5] - f[6] - f[7] + f[8], sy = f[5] + f[6] - f[7] - f[8];
    const long long rho = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8];
    const long long jx = f[1] - f[3] + sx, jy = f[2] - f[4] + sy;
    constexpr long long J = 201769274521386496LL;   // 0.35 2^59
    if ((uint64_t)(rho - (1LL << 58)) >= (uint64_t)(1LL << 59) || (uint64_t)(jx + J) >= (uint64_t)(2 * J) ||
        (uint64_t)(jy + J) >= (uint64_t)(2 * J))
        return false;
    const FxFactor inv = fx_split(fx_recip(rho));
    rho_o = fx_to(rho, k.e);
    ux_o = fx_signed_to(fx_mul((long long)((uint64_t)jx << 5), inv), -61);
    uy_o = fx_signed_to(fx_mul((long long)((uint64_t)jy << 5), inv), -61);
    return true;
}

// The same for FP32 / FP16 storage (deviations, as floats).  A deviation has
// its 24 bits relative to itself, so the sums are on a grid of their own, set
// by the node's largest one: d 2^(56 - T), 2^T > |d|, on which a float down to
// 2^-31 of the largest is exact (a node with a smaller one that is not zero,
// or with a largest one below 2^-95, is left to the FP64 code).  The sums are
// then exact, and u has the precision of a double for any size of the
// deviations; on the grid of rho0 a deviation of 1e-14 would keep 15 bits.
VPLBM_FX bool fx_moments_dev(const FixedConsts &k, const float d[9], double &rho_o, double &ux_o, double &uy_o)
{
    uint32_t top = 0, low = 0xffffffffu;   // largest; smallest but zero, minus one
    long long f[9];
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int a = 0; a < 9; ++a) {
        const uint32_t m = fx_float_bits(d[a]) & 0x7fffffffu;
        top = m > top ? m : top;
        low = m - 1u < low ? m - 1u : low;
    }
    const int et = (int)(top >> 23), el = (int)((low + 1u) >> 23);
    if (k.e < -30 || k.e > 60 || top >= (uint32_t)(124 + k.e) << 23 || (top != 0 && (et < 32 || et - el > 31))) return false;
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int a = 0; a < 9; ++a) {
        // a zero has no leading bit; its shift does not matter
        const uint32_t b = fx_float_bits(d[a]), m = b & 0x7fffffffu, s = (uint32_t)et - (m >> 23);
        const uint32_t hi = (m & 0x7fffffu) | (m < 0x800000u ? m : 0x800000u);
#if defined(__CUDA_ARCH__)
        const uint64_t x = ((uint64_t)(hi >> (s & 31)) << 32) | __funnelshift_r(0u, hi, s);
#else
        const uint64_t x = ((uint64_t)hi << 32) >> (s & 31);
#endif
        const long long sign = (int)b >> 31;
        f[a] = ((long long)x ^ sign) - sign;
    }
    const long long sx = f[5] - f[6] - f[7] + f[8], sy = f[5] + f[6] - f[7] - f[8];
    const long long rs = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8];   // below 9 2^56
    const long long jx = f[1] - f[3] + sx, jy = f[2] - f[4] + sy;                        // below 6 2^56
    const int T = et - 126, n = k.e - 3 - T;   // to the grid of rho: 2^(E - 59)
    const long long rho = k.rho0 + (n > 62 ? 0 : n > 0 ? (rs + (1LL << (n - 1))) >> n : rs);
    if ((uint64_t)(rho - (1LL << 58)) >= (uint64_t)(1LL << 59)) return false;
    const FxFactor inv = fx_split(fx_recip(rho));   // 2^120 / rho
    auto quotient = [&](long long j) {              // its leading bit to bit 61 first
        if (j == 0) return 0.0;
        const uint64_t m = j < 0 ? 0 - (uint64_t)j : (uint64_t)j;
        const int up = fx_clz64(m) - 2;
        const long long q = fx_mul((long long)(m << up), inv);
        return fx_signed_to(j < 0 ? -q : q, T - k.e - 53 - up);
    };
    rho_o = fx_to(rho, k.e);
    ux_o = quotient(jx);
    uy_o = quotient(jy);
    return true;
}

// Equilibrium (Eq. 11) of (rho, u): val[a] in units of 2^(E - 62) for the
// deviation f_a - w_a rho0 (dev), of 2^(E - 59) for the full f_a.  False if
// out of range (|u| >= 1/4, rho outside [rho0 / 2, 1.5 2^E); dev: a density
// further than 2^(E - 4) from rho0, a deviation of w_a 2^(E + 1) or more,
// which its finer unit does not hold: |u| above 0.2 along a diagonal).
VPLBM_FX bool fx_equilibrium(const FixedConsts &k, uint64_t rho_b, uint64_t ux_b, uint64_t uy_b, bool dev, long long val[9])
{
    const uint32_t rh = (uint32_t)(rho_b >> 32), xh = (uint32_t)(ux_b >> 32) & 0x7fffffffu, yh = (uint32_t)(uy_b >> 32) & 0x7fffffffu;
    // rho in [2^(E-1), 2^(E+1)): twice the range of a population, so on the
    // grid as twice the value of its half
    if (dev && (k.e < -30 || k.e > 60)) return false;
    if (rh < (unsigned)(1022 + k.e) << 20 || rh >= (unsigned)(1024 + k.e) << 20 || xh >= 0x3fd00000u || yh >= 0x3fd00000u) return false;
    const long long rho = 2 * fx_from(rho_b - (1ull << 52), k.e);
    if (rho >= (3LL << 58)) return false;
    const long long ux = fx_from_signed(ux_b), uy = fx_from_signed(uy_b);   // 2^61
    const FxFactor fx = fx_split(ux), fy = fx_split(uy);
    const long long xx = fx_mul(ux, fx), yy = fx_mul(uy, fy), xy = fx_mul(ux, fy);   // 2^58
    const long long drho = rho - k.rho0;
    if (dev && (uint64_t)(drho + (1LL << 55)) >= (uint64_t)(1LL << 56)) return false;
    const long long r8 = (long long)((uint64_t)rho << 3);
    const long long u15 = 6 * (xx + yy);   // 3/2 u^2 2^60
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
    for (int a = 0; a < 9; ++a) {
        const int cx = a == 1 || a == 5 || a == 8 ? 1 : (a == 3 || a == 6 || a == 7 ? -1 : 0);
        const int cy = a == 2 || a == 5 || a == 6 ? 1 : (a == 4 || a == 7 || a == 8 ? -1 : 0);
        const long long cu = cx * ux + cy * uy, cu2 = (cx ? xx : 0) + (cy ? yy : 0) + 2 * cx * cy * xy;
        const long long poly = ((3 * cu) >> 1) + 18 * cu2 - u15;   // 3 c.u + 9/2 (c.u)^2 - 3/2 u^2, 2^60
        const long long rp = fx_mul(r8, fx_split(2 * poly));        // rho poly, 2^(E - 59)
        const FxFactor w = a == 0 ? FX_W0 : a <= 4 ? FX_W1 : FX_W2;
        if (dev) {
            const long long d = drho + rp;
            if ((uint64_t)(d + (1LL << 60)) >= (uint64_t)(1LL << 61)) return false;
            val[a] = fx_mul(8 * d, w);
        } else {
            val[a] = fx_mul(rho + rp, w);
        }
    }
    return true;
}

}  // namespace
}  // namespace vplbm
