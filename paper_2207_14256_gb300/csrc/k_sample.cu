// k_sample.cu -- pre-initial particle sampling (Sec. 2.1 of Elbers 2022):
// positions uniform in the periodic box, |q| from the Fermi-Dirac distribution
// fbar(q) = 1/(1 + e^{q/T}) by inversion of its tabulated CDF, and an
// isotropic direction by rejection from the cube.
//
// Every particle is addressed by its global index g (species-major) so the
// draw does not depend on the launch shape.  Philox4x32-10 keyed by the seed
// with counter (g_lo, g_hi, stream, attempt):
//   stream 0: X_c = word c (c = 0, 1, 2); x_c = L X_c / 2^32
//   stream 1: u from words 0,1 (53 bits) -> t = F^{-1}(u) -> |q| = T t
//   streams 2, 3 (attempt a): v = 2 u - 1 from (2: words 0,1), (2: words 2,3),
//     (3: words 0,1); accept 1e-300 < |v|^2 <= 1; n = v / |v|.
// Only correctly rounded IEEE operations are used (explicit _rn intrinsics, so
// no FMA contraction), which makes the result exact and reproducible.
#include "device_math.cuh"

namespace fdf {

// The 53-bit integer m = (w0 >> 5) 2^26 + (w1 >> 6) of two words, exact in 64 bits.
__device__ __forceinline__ uint64_t m53(uint32_t w0, uint32_t w1)
{
    return ((uint64_t)(w0 >> 5) << 26) | (uint64_t)(w1 >> 6);
}

// 1 + (m mod 2^52) 2^-52, a bit pattern (no FP64 conversion, which costs an FP64 slot)
__device__ __forceinline__ double one_plus(uint64_t m)
{
    return __longlong_as_double((long long)((m & 0xFFFFFFFFFFFFFull) | 0x3FF0000000000000ull));
}

// u = m 2^-53, exact
__device__ __forceinline__ double u53(uint32_t w0, uint32_t w1)
{
    const uint64_t m = m53(w0, w1);
    const double x = (m >> 52) ? one_plus(m) : __dsub_rn(one_plus(m), 1.0);    // m 2^-52
    return __dmul_rn(x, 0.5);
}

// v = 2u - 1 = (m - 2^52) 2^-52, exact
__device__ __forceinline__ double v53(uint32_t w0, uint32_t w1)
{
    const uint64_t m = m53(w0, w1);
    return __dsub_rn(one_plus(m), (m >> 52) ? 1.0 : 2.0);
}

__device__ __forceinline__ double fd_inverse(const double* __restrict__ t, const double* __restrict__ F, int n,
                                             double u)
{
    if (u >= F[n - 1]) return t[n - 1];
    // F and u are non-negative, so their IEEE bit patterns order like their values:
    // the bisection compares 64-bit integers instead of FP64 values
    const long long ub = __double_as_longlong(u);
    const long long* Fb = reinterpret_cast<const long long*>(F);
    int lo = 0, hi = n - 1;  // F[lo] <= u < F[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (Fb[mid] <= ub) lo = mid;
        else hi = mid;
    }
    const double du = __dsub_rn(u, F[lo]);
    const double dt = __dsub_rn(t[lo + 1], t[lo]);
    const double dF = __dsub_rn(F[lo + 1], F[lo]);
    return __dadd_rn(t[lo], __ddiv_rn(__dmul_rn(du, dt), dF));
}

// Attempt `att` of the direction of particle (g0, g1): the words of v from streams 2 and 3;
// accepted when 1e-300 < |v|^2 <= 1 in FP64.  FP32 settles that (the first word of each
// component, |v|^2 to 3.5e-7) unless |v|^2 is within 1e-6 of 1 or of 0.
__device__ __forceinline__ bool direction_attempt(uint32_t g0, uint32_t g1, uint32_t att, uint32_t key0, uint32_t key1,
                                                  uint32_t w[6])
{
    const uint4 a = philox4x32_10(make_uint4(g0, g1, 2u, att), key0, key1);
    const uint4 b = philox4x32_10(make_uint4(g0, g1, 3u, att), key0, key1);
    w[0] = a.x;
    w[1] = a.y;
    w[2] = a.z;
    w[3] = a.w;
    w[4] = b.x;
    w[5] = b.y;
    // (w0 - 2^31) 2^-31 is v to 2^-26 (m's top 27 bits are w0's; the next come from the second
    // word), and FP32 rounds it and the sum: |v|^2 to 3.5e-7
    const float f0 = (float)(int)(a.x - 0x80000000u), f1 = (float)(int)(a.z - 0x80000000u);
    const float f2 = (float)(int)(b.x - 0x80000000u);
    const float r2 = (f0 * f0 + f1 * f1 + f2 * f2) * 2.168404344971009e-19f;   // 2^-62
    if (fabsf(r2 - 1.f) > 1e-6f && r2 > 1e-6f) return r2 < 1.f;
    const double v0 = v53(w[0], w[1]), v1 = v53(w[2], w[3]), v2 = v53(w[4], w[5]);
    const double s = __dadd_rn(__dadd_rn(__dmul_rn(v0, v0), __dmul_rn(v1, v1)), __dmul_rn(v2, v2));
    return (s > 1e-300) && (s <= 1.0);
}

constexpr uint32_t kMaxAttempts = 64;

// The directions of a warp's particles, the whole warp working on every round.  A
// particle's direction is its lowest accepted attempt (at most kMaxAttempts), as a
// loop over its attempts would find; but instead of each lane looping until the
// warp's unluckiest lane accepts, every round spreads the attempts of the particles
// still pending over all 32 lanes: with np pending, lane l tries attempt
// next + l / np of the (l mod np)-th pending particle.  Lanes without a particle
// (live = false) only help.  Returns whether this lane's particle got a direction.
__device__ bool warp_direction(bool live, uint32_t g0, uint32_t g1, uint32_t key0, uint32_t key1, uint32_t v[6])
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned pending = __ballot_sync(full, live);
    uint32_t next = 0;      // the owner's next untried attempt
    bool ok = false;
    while (pending) {
        const int np = __popc(pending);
        const int k = lane % np, rep = lane / np;
        unsigned m = pending;                              // the k-th pending lane
        for (int j = 0; j < k; ++j) m &= m - 1u;
        const int owner = __ffs(m) - 1;
        const uint32_t og0 = __shfl_sync(full, g0, owner), og1 = __shfl_sync(full, g1, owner);
        const uint32_t att = __shfl_sync(full, next, owner) + (uint32_t)rep;
        uint32_t a[6] = {0u, 0u, 0u, 0u, 0u, 0u};
        const bool acc = att < kMaxAttempts && direction_attempt(og0, og1, att, key0, key1, a);
        const unsigned accepted = __ballot_sync(full, acc);
        // an owner's lanes are its rank r + j np, j = 0, 1, ...: the lowest accepted one wins
        const bool mine = (pending >> lane) & 1u;
        const int r = mine ? __popc(pending & ((1u << lane) - 1u)) : 0;
        unsigned lanes = 0u;
        if (mine)
            for (int l = r; l < 32; l += np) lanes |= 1u << l;
        const int win = mine ? __ffs(accepted & lanes) - 1 : -1;
        const int src = win >= 0 ? win : lane;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const uint32_t w = __shfl_sync(full, a[j], src);
            if (win >= 0) v[j] = w;
        }
        bool done = false;
        if (mine) {
            if (win >= 0) {
                ok = true;
                done = true;
            } else {
                next += (uint32_t)__popc(lanes);
                done = next >= kMaxAttempts;
            }
        }
        pending &= ~__ballot_sync(full, done);
    }
    return ok;
}

// a / b, correctly rounded (__ddiv_rn's bits), with inv within a few last places of 1/b
__device__ __forceinline__ double div_rn(double a, double b, double inv)
{
    double r;
    if (!w_div53(a, b, a * inv, r)) r = div_slow(a, b);
    return r;
}

// Bound: the FP64 pipe.  The roots and quotients have their correctly rounded bits from the
// integer pipe, and attempts are settled in FP32: 36 FP64 instructions per particle
// against 105 (3 x 200^3 particles: 4.63 -> 1.71 ms).  The FP64 fallbacks are calls
// (sqrt_slow and its kin): inlined, they ran for every particle (3.54 ms).
__global__ void __launch_bounds__(256) k_sample(int64_t N, uint32_t key0, uint32_t key1, double T_ev,
                                                const double* __restrict__ cdf_t, const double* __restrict__ cdf_F,
                                                int ncdf, uint32_t* __restrict__ X, double* __restrict__ qs,
                                                double* __restrict__ pmag, uint32_t* __restrict__ id, int* flag)
{
    // warp-uniform trip count: every lane takes part in the warp's direction rounds
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x; i0 < N; i0 += stride) {
        const int64_t i = i0 + threadIdx.x;
        const bool live = i < N;
        const uint32_t g0 = (uint32_t)i, g1 = (uint32_t)((uint64_t)i >> 32);
        uint32_t v[6] = {0u, 0u, 0u, 0u, 0u, 0u};
        const bool ok = warp_direction(live, g0, g1, key0, key1, v);
        if (!live) continue;
        uint4 w = philox4x32_10(make_uint4(g0, g1, 0u, 0u), key0, key1);
        X[i] = w.x;
        X[N + i] = w.y;
        X[2 * N + i] = w.z;
        w = philox4x32_10(make_uint4(g0, g1, 1u, 0u), key0, key1);
        const double qmag = __dmul_rn(T_ev, fd_inverse(cdf_t, cdf_F, ncdf, u53(w.x, w.y)));
        double v0 = v53(v[0], v[1]), v1 = v53(v[2], v[3]), v2 = v53(v[4], v[5]);
        double r2 = __dadd_rn(__dadd_rn(__dmul_rn(v0, v0), __dmul_rn(v1, v1)), __dmul_rn(v2, v2));
        if (!ok) {
            atomicOr(flag, 1);
            r2 = 1.0;
            v0 = 1.0;
            v1 = v2 = 0.0;
        }
        // v / sqrt(r2): the quotients' estimates from 1/sqrt(r2)
        const float y = rsqrtf(d2f_bits(r2));
        double s, inv;
        if (!w_sqrt53(r2, y, s)) s = sqrt_slow(r2);
        if (!w_rsqrt53(r2, y, inv)) inv = div_slow(1.0, s);
        const double n[3] = {div_rn(v0, s, inv), div_rn(v1, s, inv), div_rn(v2, s, inv)};
        const double q[3] = {__dmul_rn(qmag, n[0]), __dmul_rn(qmag, n[1]), __dmul_rn(qmag, n[2])};
        qs[i] = q[0];
        qs[N + i] = q[1];
        qs[2 * N + i] = q[2];
        pmag[i] = norm3_rn(q);
        id[i] = (uint32_t)i;
    }
}

cudaError_t launch_sample(cudaStream_t s, int64_t n, uint32_t key0, uint32_t key1, double T_ev, const double* cdf_t,
                          const double* cdf_F, int ncdf, uint32_t* X, double* qs, double* pmag, uint32_t* id,
                          int* flag)
{
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 64) blocks = 152 * 64;
    k_sample<<<(unsigned)blocks, 256, 0, s>>>(n, key0, key1, T_ev, cdf_t, cdf_F, ncdf, X, qs, pmag, id, flag);
    return cudaGetLastError();
}

}  // namespace fdf
