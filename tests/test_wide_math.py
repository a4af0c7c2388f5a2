"""csrc/wide_math.cuh (FP64 results on the FP32 and integer pipes), compiled for the host, against the
FP64 formulas it stands for: every accepted result is theirs bit for bit, and few are refused.

The hardware's inverse square root estimate is stood in for by the rounded one moved by up to
+-2^-22.3 (its documented error is 2^-22.4).  Refusals: w_rsqrt53 leaves 33 of 65536 values to FP64
and those whose mantissa lies within 2^-20 of a power of 4; w_kick the results within 2^-41 of a
rounding boundary of FP32 (spaced 2^-24 to 2^-23 apart), three times per call: 2^-15 of them, and
2^-18 more for u_0's estimate; the bounds below are four times that.
"""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_14256_gb300", "csrc")
SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
static float g_skew = 0;
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
template <class T, class S> static inline T bits(S s) { T t; std::memcpy(&t, &s, sizeof(t)); return t; }
static inline uint32_t __float_as_uint(float f) { return bits<uint32_t>(f); }
static inline float __uint_as_float(uint32_t u) { return bits<float>(u); }
static inline int __double2hiint(double d) { return (int)(bits<uint64_t>(d) >> 32); }
static inline int __double2loint(double d) { return (int)bits<uint64_t>(d); }
static inline double __hiloint2double(int h, int l) { return bits<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, uint32_t s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
static inline uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) { return s ? (lo >> s) | (hi << (32 - s)) : lo; }
static inline float __int2float_rn(int i) { return (float)i; }
static inline float __uint2float_rn(uint32_t i) { return (float)i; }
static inline int __float2int_rn(float f) { return (int)std::nearbyint(f); }
static inline float w_rsqrt(float f) { return (float)(1.0 / std::sqrt((double)f) * (1.0 + g_skew)); }
static inline float w_rcp(float f) { return (float)(1.0 / f * (1.0 + g_skew)); }
#include "wide_math.cuh"
#include "wide_poly.cuh"
using namespace fdf;
// round to float, ties away from zero
static float d2f(double d)
{
    const uint64_t u = bits<uint64_t>(d);
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u, mag = hi & 0x7FFFFFFFu;
    const uint32_t f = (((mag - 0x38000000u) << 3) | (lo >> 29)) + ((lo >> 28) & 1u);
    return bits<float>((hi & 0x80000000u) | (mag < 0x38100000u ? 0u : f));
}
static double rsqrt64(double u, float y)
{
    const double yd = y, yh = 0.5f * y, eh = std::fma(-(u * yd), yh, 0.5);
    const float f = d2f(eh);
    return std::fma(yd, eh + (double)(1.5f * f * f), yd);
}
static void skew(int i) { g_skew = (float)((i * 7 % 13 - 6) / 6.0 * 1.9e-7); }
// counts: [0] refused, [1] accepted with other bits than FP64's
extern "C" void check_rsqrt(int n, const double* v, long* counts)
{
    for (int i = 0; i < n; ++i) {
        skew(i);
        const float y = w_rsqrt(d2f(v[i]));
        double r;
        int64_t R;
        int k;
        if (!w_rsqrt53(v[i], y, r, R, k)) ++counts[0];
        else if (r != rsqrt64(v[i], y) || w_square53(R, k) != r * r) ++counts[1];
    }
}
extern "C" void check_add(int n, const double* q, const float* d, long* counts)
{
    for (int i = 0; i < n; ++i) {
        double r;
        const double x = std::fabs(d[i]) < 1.1754943508222875e-38f ? 0.0 : (double)d[i];
        if (!w_add(q[i], d[i], r)) ++counts[0];
        else if (bits<uint64_t>(r) != bits<uint64_t>(q[i] + x)) ++counts[1];
    }
}
extern "C" void check_mul(int n, const long* R, const int* k, const double* g, long* counts)
{
    for (int i = 0; i < n; ++i) {
        double x;
        const double r = std::ldexp((double)R[i], -53 - k[i]);
        if (!w_mul53(R[i], k[i], g[i], x)) ++counts[0];
        else if (bits<uint64_t>(x) != bits<uint64_t>(r * g[i])) ++counts[1];
    }
}
extern "C" void check_sqrt(int n, const double* v, long* counts)
{
    for (int i = 0; i < n; ++i) {
        skew(i);
        double r;
        if (!w_sqrt53(v[i], w_rsqrt(d2f(v[i])), r)) ++counts[0];
        else if (r != std::sqrt(v[i])) ++counts[1];
        const float f = w_d2f(v[i]);
        if (v[i] > 1.2e-38 && v[i] < 3.4e38 && f != (float)v[i]) ++counts[1];
    }
}
// estimates off by up to `off` last places
extern "C" void check_div(int n, const double* a, const double* b, int off, long* counts)
{
    for (int i = 0; i < n; ++i) {
        const double q = a[i] / b[i];
        double r;
        const double est = bits<double>(bits<uint64_t>(q) + (uint64_t)(int64_t)(i % (2 * off + 1) - off));
        if (!w_div53(a[i], b[i], est, r)) ++counts[0];
        else if (r != q) ++counts[1];
    }
}
extern "C" void check_square(int n, const long* R, long* counts)
{
    for (int i = 0; i < n; ++i)
        if (w_square53(R[i], 0) != ((double)R[i] * 0x1p-53) * ((double)R[i] * 0x1p-53)) ++counts[1];
}
// a kick over nodes W, e (mu = m^2 a_c^2) at momenta q[n][3]; series: c_0 (FP64) and c_1.. (FP32)
extern "C" int check_kick(int series, int m, const double* W, const double* e, double mu, double unit, const double* cpsi,
                          const double* cphi, int n, const float* q, long* counts)
{
    KickPoly psi, phi;
    std::memset(&psi, 0, sizeof(psi));
    std::memset(&phi, 0, sizeof(phi));
    if (series) {
        for (int k = 0; k <= KickLen<true>::kDeg; ++k) {
            kick_coef(psi, k, cpsi[k] / unit);
            kick_coef(phi, k, cphi[k] * unit);
        }
    } else if (!kick_node_poly(W, e, m, 0.5, 1.0 / unit, psi) || !kick_node_poly(W, e, m, -0.5, unit, phi)) {
        return 0;
    }
    const float u2 = (float)(unit * unit), muh = (float)(mu * unit * unit), mul = (float)(mu * unit * unit - (double)muh);
    for (int i = 0; i < n; ++i) {
        skew(i);
        const double a = q[3 * i], b = q[3 * i + 1], c = q[3 * i + 2], s0 = std::fma(a, a, std::fma(b, b, c * c));
        const float s0h = d2f(s0), s0l = d2f((s0 - (double)s0h) * (double)u2);
        float kp, kf;
        const bool ok = series ? w_kick<true>(s0h * u2, s0l, muh, mul, psi, phi, kp, kf)
                               : w_kick<false>(s0h * u2, s0l, muh, mul, psi, phi, kp, kf);
        double dp = 0, df = 0;
        if (series) {
            const double u0 = s0 + mu;
            const float y = w_rsqrt(d2f(u0));
            const double yd = y, yh = 0.5f * y, r0 = std::fma(yd, std::fma(-(u0 * yd), yh, 0.5), yd);
            const float r = d2f(r0), t = d2f(mu) * r * r;
            float tp = 0, tf = 0;
            for (int k = KickLen<true>::kDeg; k >= 1; --k) {
                tp = std::fma(tp, t, (float)cpsi[k]);
                tf = std::fma(tf, t, (float)cphi[k]);
            }
            df = r0 * std::fma((double)tf, (double)t, cphi[0]);
            dp = (u0 * r0) * std::fma((double)tp, (double)t, cpsi[0]);
        } else {
            for (int j = 0; j < m; ++j) {
                const double e2 = s0 + mu * (1.0 + e[j]), ie = rsqrt64(e2, w_rsqrt(d2f(e2)));
                dp = std::fma(W[j], e2 * ie, dp);
                df = std::fma(W[j], ie, df);
            }
        }
        if (!ok) ++counts[0];
        else if (kp != d2f(dp) || kf != d2f(df)) ++counts[1];
    }
    return 1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("wide")
    (d / "w.cpp").write_text(SHIM)
    cmd = ["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-Wno-unknown-pragmas", "-I", CSRC, "-shared", "-fPIC",
           "-o", str(d / "w.so"), str(d / "w.cpp")]
    subprocess.run(cmd, check=True)
    return C.CDLL(str(d / "w.so"))


def _ptr(a):
    return a.ctypes.data_as(C.c_void_p)


@pytest.mark.parametrize("lo,hi", [(1.0, 4.0), (1.0, 1.0 + 2e-6), (4.0 - 4e-6, 4.0), (1e-9, 1e13), (1e-30, 1e30)])
def test_rsqrt_bits(lib, lo, hi):
    rng = np.random.default_rng(3)
    n = 1000000
    v = np.exp(rng.uniform(math.log(lo), math.log(hi), n)) if hi > 8 else rng.uniform(lo, hi, n)
    counts = np.zeros(2, np.int64)
    lib.check_rsqrt(n, _ptr(v), _ptr(counts))
    assert counts[1] == 0
    if hi - lo > 1e-3:
        assert counts[0] <= 4 * 33 / 65536 * n


@pytest.mark.parametrize("lo,hi", [(1.0, 4.0), (1.0, 1.0 + 2e-6), (4.0 - 4e-6, 4.0), (1e-30, 1e30)])
def test_sqrt_bits(lib, lo, hi):
    rng = np.random.default_rng(13)
    n = 1000000
    v = np.exp(rng.uniform(math.log(lo), math.log(hi), n)) if hi > 8 else rng.uniform(lo, hi, n)
    v[::3] = (v[::3] * 2.0 ** 20).round() * 2.0 ** -20          # short, and squares among them
    v[1::3] = np.sqrt(v[1::3]).astype(np.float32).astype(np.float64) ** 2
    v = np.concatenate([v, [0.0, -1.0, 5e-324, np.inf, np.nan, 1e300, 1e-300]])
    counts = np.zeros(2, np.int64)
    lib.check_sqrt(len(v), _ptr(v), _ptr(counts))
    assert counts[1] == 0
    if hi - lo > 1e-3:
        # refused: zeros, estimates outside [1/2, 1), mantissas within 2^-20 of a power of 4
        v = np.ascontiguousarray(v[v > 0])
        counts[:] = 0
        lib.check_sqrt(len(v), _ptr(v), _ptr(counts))
        assert counts[0] <= 2e-3 * n


@pytest.mark.parametrize("scale", [1.0, 1e-4, 1e30])
def test_div_bits(lib, scale):
    rng = np.random.default_rng(17)
    n = 1000000
    a = scale * rng.normal(size=n)
    b = rng.uniform(1e-3, 2.0, n)
    a[::5] = (b[::5] * rng.integers(1, 100, len(b[::5])))         # exact and nearly exact quotients
    a[-3:] = 0.0, np.inf, np.nan
    counts = np.zeros(2, np.int64)
    lib.check_div(n, _ptr(a), _ptr(b), 3, _ptr(counts))
    assert counts[1] == 0
    assert counts[0] <= 2e-3 * n + len(a[::5]) / 10               # powers of two among the exact ones


def test_square_bits(lib):
    rng = np.random.default_rng(7)
    R = rng.integers(2 ** 52, 2 ** 53, 1000000)
    root2 = int(2 ** 52 * math.sqrt(2.0))
    # short significands, whose squares round at ties or not at all, and both ends of each binade
    R = np.concatenate([R, (R >> 27) << 27, (R >> 26) << 26, (R >> 25) << 25, 2 ** 52 + np.arange(999),
                        2 ** 53 - 1 - np.arange(999), root2 + np.arange(-999, 999)])
    counts = np.zeros(2, np.int64)
    lib.check_square(len(R), _ptr(R), _ptr(counts))
    assert counts[1] == 0


def test_mul_bits(lib):
    rng = np.random.default_rng(19)
    n = 1000000
    R = rng.integers(2 ** 52, 2 ** 53, n)
    R[::5] = (R[::5] >> 30) << 30                    # short significands: ties and exact products
    k = rng.integers(-60, 60, n).astype(np.int32)
    g = rng.normal(size=n) * np.exp2(rng.integers(-40, 40, n))
    g[::7] = np.float32(g[::7])
    g[::11] = np.exp2(rng.integers(-40, 40, len(g[::11])))
    counts = np.zeros(2, np.int64)
    lib.check_mul(n, _ptr(R), _ptr(k), _ptr(g), _ptr(counts))
    assert counts[1] == 0 and counts[0] == 0
    g = np.tile(np.array([0.0, -0.0, np.inf, np.nan, 5e-324, 1e-300, 1e300, -1e308]), 100)
    R, k = R[:len(g)].copy(), rng.integers(-60, 60, len(g)).astype(np.int32)
    lib.check_mul(len(g), _ptr(R), _ptr(k), _ptr(g), _ptr(counts))
    assert counts[1] == 0


@pytest.mark.parametrize("scale", [1e-4, 1.0, 1e25])
def test_add_bits(lib, scale):
    rng = np.random.default_rng(11)
    n = 1000000
    q = scale * rng.normal(size=n)
    # from |d| = 2|q| down past q's last place; zeros, and ties (odd multiples of half a last place)
    d = (q * rng.choice([-1.0, 1.0], n) * np.exp2(-rng.uniform(-1.0, 60.0, n))).astype(np.float32)
    d[::97] = 0.0
    tie = np.arange(0, n, 13)
    d[tie] = (np.spacing(np.abs(q[tie])) * (rng.integers(0, 1 << 20, len(tie)) + 0.5)).astype(np.float32)
    q[1::101] = scale * np.exp2(rng.integers(-3, 3, len(q[1::101])))          # powers of two: the binade's edge
    counts = np.zeros(2, np.int64)
    lib.check_add(n, _ptr(q), _ptr(d), _ptr(counts))
    assert counts[1] == 0
    # refused: sums that leave the binade, likely only where |d| > 2^-7 |q|
    small = np.abs(d) < np.exp2(-7.0) * np.abs(q)
    small[1::101] = False
    qs, ds = np.ascontiguousarray(q[small]), np.ascontiguousarray(d[small])
    counts[:] = 0
    lib.check_add(len(qs), _ptr(qs), _ptr(ds), _ptr(counts))
    assert counts[0] <= 2.0 ** -7 * len(qs)
    special = np.array([0.0, -0.0, 5e-324, 1e-310, np.inf, -np.inf, np.nan, 1.0, -1.0])
    q = np.repeat(special, 6)
    d = np.tile(np.array([0.0, -0.0, 1e-39, np.inf, -np.inf, 1e-30], np.float32), len(special))
    counts[:] = 0
    lib.check_add(len(q), _ptr(q), _ptr(d), _ptr(counts))
    assert counts[1] == 0


@pytest.mark.parametrize("T", [1.7e-4, 1e-12])
@pytest.mark.parametrize("series,dlna,ngl", [(1, 0.0575, 4), (1, -0.0863, 4), (1, 0.115, 4), (0, 0.0863, 4), (0, -0.12, 4),
                                             (0, 0.1726, 5), (0, 0.19, 5), (0, 0.3, 2), (0, 0.0575, 8)])
def test_kick_bits(lib, T, series, dlna, ngl):
    rng = np.random.default_rng(5)
    n = 60000
    q = T * rng.gamma(3.2, 1.0, n) * np.where(rng.random(n) < 0.05, 1e-3, 1.0)
    d = rng.normal(size=(n, 3))
    q = (q[:, None] * d / np.linalg.norm(d, axis=1)[:, None]).astype(np.float32)
    x, w = np.polynomial.legendre.leggauss(ngl)
    unit = 2.0 ** min(50, max(-50, round(-math.log2(T))))
    # a H goes like a power of a between -1 (radiation) and -1/2 (matter): the weights' slope
    for slope, mac in ((1.0, 0.0), (1.0, 1e-3 * T), (0.5, T), (0.8, 30.0 * T), (0.5, 3e3 * T)):
        lna = 0.5 * dlna * x
        W = 700.0 * w * 0.5 * dlna * np.exp(slope * lna)
        e = np.exp(2.0 * lna) - 1.0
        # a fit as the host makes it: c_0 in FP64, the others FP32
        t = 0.5 * (1.0 + np.cos(np.pi * (np.arange(6) + 0.5) / 6))
        cs = []
        for power in (0.5, -0.5):
            g = (W[:, None] * (1.0 + e[:, None] * t) ** power).sum(0)
            c = np.polynomial.polynomial.polyfit(t, g, 5)
            cs.append(np.concatenate([c[:1], c[1:].astype(np.float32).astype(np.float64)]))
        counts = np.zeros(2, np.int64)
        ok = lib.check_kick(series, ngl, _ptr(W), _ptr(e), C.c_double(mac * mac), C.c_double(unit), _ptr(cs[0]),
                            _ptr(cs[1]), n, _ptr(q), _ptr(counts))
        assert ok
        assert counts[1] == 0, (slope, mac)
        assert counts[0] <= 4 * (2.0 ** -15 + 2.0 ** -18) * n, (slope, mac)


def test_kick_node_poly_refuses_coarse_steps(lib):
    x, w = np.polynomial.legendre.leggauss(5)
    e = np.exp(0.2 * x) - 1.0
    q = np.ones((1, 3), np.float32)
    assert not lib.check_kick(0, 5, _ptr(w), _ptr(e), C.c_double(1.0), C.c_double(1.0), None, None, 1, _ptr(q),
                              _ptr(np.zeros(2, np.int64)))
