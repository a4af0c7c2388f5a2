"""The integer conversions of csrc/wide_math.cuh and the weight of csrc/device_math.cuh, compiled for
the host, at values outside FP32's normal range: they are those of plain casts, so that NaN,
infinities and overflows of a state reach the weights and the density as what they are.  Reads at
such positions stay in the grid.
"""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2207_14256_gb300", "csrc")
SHIM = r"""
#include <cuda_runtime.h>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __noinline__ __attribute__((noinline))
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __ddiv_rn(double a, double b) { return a / b; }
static inline double __dsqrt_rn(double a) { return std::sqrt(a); }
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
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static inline float rsqrtf(float f) { return (float)(1.0 / std::sqrt((double)f)); }
#include "device_math.cuh"
using namespace fdf;
// results that are neither the cast's bits nor both NaN
extern "C" long check_narrow(long n, const double* d)
{
    long bad = 0;
    for (long i = 0; i < n; ++i) {
        const float f = w_d2f(d[i]), g = (float)d[i];
        bad += bits<uint32_t>(f) != bits<uint32_t>(g) && !(f != f && g != g);
    }
    return bad;
}
extern "C" long check_widen(long n, const float* f)
{
    long bad = 0;
    for (long i = 0; i < n; ++i) {
        const double d = w_f2d(f[i]), g = (double)f[i];
        bad += bits<uint64_t>(d) != bits<uint64_t>(g) && !(d != d && g != g);
    }
    return bad;
}
extern "C" void weights(long n, const double* q, const double* p, double T, float* w)
{
    for (long i = 0; i < n; ++i) w[i] = dfweight_split(norm3_rn(q + 3 * i), p[i], T, 1.0 / T);
}
extern "C" void tsc(double u, int N, int* idx, double* w) { tsc_f64(u, N, idx, w); }
extern "C" double kicked(double q, float d) { return add_slow(q, d); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("nonfinite")
    (d / "w.cpp").write_text(SHIM)
    cmd = ["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-Wno-unknown-pragmas", "-I", CSRC, "-I",
           os.path.join(ROOT, "include"), "-I", "/usr/local/cuda/include", "-shared", "-fPIC", "-o", str(d / "w.so"),
           str(d / "w.cpp")]
    subprocess.run(cmd, check=True)
    L = C.CDLL(str(d / "w.so"))
    L.check_narrow.restype = L.check_widen.restype = C.c_long
    L.kicked.restype, L.kicked.argtypes = C.c_double, [C.c_double, C.c_float]
    L.tsc.argtypes = [C.c_double, C.c_int, C.c_void_p, C.c_void_p]
    return L


def _ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def test_narrowing_is_the_cast(lib):
    rng = np.random.default_rng(3)
    edge = np.array([3.4028234663852886e38, 3.4028235677973362e38, 3.4028235677973366e38, 1e39, 1e300, np.inf, np.nan,
                     1.1754943508222875e-38, 1.1754942807573643e-38, 1.4e-45, 7.006492321624085e-46, 7.1e-46, 1e-46,
                     2.1019476964872256e-45, 5e-324, 1e-310, 0.0, 1.0])
    d = np.concatenate([edge, -edge, np.exp2(rng.uniform(-160, -120, 200000)), np.exp2(rng.uniform(120, 140, 20000)),
                        rng.integers(0, 1 << 25, 200000) * 2.0 ** -150,        # ties of the subnormal range
                        rng.integers(0, 1 << 63, 500000, dtype=np.int64).view(np.float64)])
    d = np.concatenate([d, -d])
    assert lib.check_narrow(len(d), _ptr(d)) == 0


def test_widening_is_the_cast(lib):
    rng = np.random.default_rng(4)
    f = np.concatenate([rng.integers(0, 1 << 32, 1000000, dtype=np.uint64).astype(np.uint32),
                        np.array([0, 1, 0x7FFFFF, 0x800000, 0x7F7FFFFF, 0x7F800000, 0x7FC00000, 0x7F800001], np.uint32),
                        np.arange(0, 0x800000, 97, dtype=np.uint32)])
    f = np.concatenate([f, f ^ np.uint32(0x80000000)]).view(np.float32)
    assert lib.check_widen(len(f), _ptr(f)) == 0


def test_weight_of_a_non_finite_momentum(lib):
    T = 1.7e-4
    q = np.array([[np.nan, 0, 0], [0, -np.nan, T], [np.inf, 0, 0], [T, T, T], [T, T, T]])
    p = np.array([T, 2 * T, T, np.nan, np.sqrt(3.0) * T])
    w = np.zeros(5, np.float32)
    lib.weights(5, _ptr(q), _ptr(p), C.c_double(T), _ptr(w))
    assert np.isnan(w[[0, 1, 3]]).all()
    # |q| -> infinity: w = -expm1(-inf) / (1 + exp(-inf)) = 1
    assert w[2] == 1.0 and abs(w[4]) < 1e-6


def test_kick_of_a_non_finite_gradient(lib):
    assert np.isnan(lib.kicked(1e-4, np.nan))
    assert lib.kicked(1e-4, np.inf) == np.inf and lib.kicked(1e-4, -np.inf) == -np.inf
    assert lib.kicked(1e-4, 1e-6) == 1e-4 + float(np.float32(1e-6))


@pytest.mark.parametrize("N", [8, 512])
def test_order_2_reads_stay_in_the_grid(lib, N):
    idx, w = np.zeros(3, np.int32), np.zeros(3)
    for u in (np.nan, -np.nan, np.inf, -np.inf, 1e30, -1e30, 3e9, -3e9, 2.0 ** 31, 1.0 * N, N - 0.5, N + 0.5, 2.5 * N, -0.75,
              -1.0 * N, 0.0, 0.49, 3.5, 4.25):
        lib.tsc(u, N, _ptr(idx), _ptr(w))
        assert ((idx >= 0) & (idx < N)).all(), u
        if 0 <= u <= N:
            c = math.floor(u + 0.5)
            assert list(idx) == [(c + o) % N for o in (-1, 0, 1)]
            assert np.allclose(w, [0.5 * (0.5 - (u - c)) ** 2, 0.75 - (u - c) ** 2, 0.5 * (0.5 + (u - c)) ** 2], 1e-15)
        elif not np.isfinite(u):
            assert np.isnan(w).all()
