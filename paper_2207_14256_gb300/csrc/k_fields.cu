// k_fields.cu -- potential-gradient grids at one scale factor (Sec. 2.1 of
// Elbers 2022: the potentials follow from the transfer functions by Fourier
// transform, and the grids are shared by all particles of a step).
//
// Eight real fields are built, packed in pairs into four complex transforms
// (a real field has a Hermitian spectrum, so F_a + i F_b transforms to
// f_a + i f_b):
//   P0 = d_x psi + i d_y psi     P1 = d_z psi + i d_x phi
//   P2 = d_y phi + i d_z phi     P3 = phi_dot + i psi
// (P3 = phi_dot + i (phi + psi) for the steps of the exact equations of motion, and
// phi_dot + i 0 for the steps of the separable forms, whose passes read no slot 7)
// with d_j f = sum_n i k_j T_f(k, a) R_n e^{i k.x}, phi_dot = a H dT_phi/dln a R.
// R_n is a Hermitian Gaussian field drawn from Philox4x32-10 addressed by the
// signed mode (so the realisation does not depend on the launch), with
// <|R_n|^2> = P_R(k)/V, P_R = 2 pi^2 A_s k^-3 (k/k_pivot)^(n_s-1).
//
// Three passes over the 4 x N^3 complex work arrays, each an inverse DFT of
// length N = N1 N2 along one axis (16 x 16 at N = 256): a line's N2 threads
// each hold N1 values in registers, transform them, twiddle, exchange through
// a padded transpose in shared memory and transform the other factor:
//   z: form the spectrum from the stored unit Gaussian field and the per-step
//      amplitude table, and transform along z;
//   y: transform along y;
//   x: transform along x and write the interleaved gather grid G[cell][8] as
//      whole 32-byte records.
// That is the FP32 form, bound by memory.  The FP64 passes, bound by the FP64 pipe, hold half
// spectra instead (the columns jx < N/2 of a real field's Hermitian spectrum) and take each
// axis' gradients at that axis' pass, so that fewer columns are transformed along z and y:
//   z: psi, d_z psi, phi, d_z phi and phi_dot (five half arrays: 2.5 N^3 of 4 N^3);
//   y: those, d_y psi and d_y phi (seven: 3.5 N^3);
//   x: the pairs P0..P3 formed line by line from the half spectra, d_x there.
#include <cuda_bf16.h>

#include <utility>

#include "device_math.cuh"

namespace fdf {

namespace {

// ---- in-register DFTs ----------------------------------------------------------
// e^{2 pi i j / 32}, j = 0..31 (exact zeros and ones on the axes).
#define C0 0.9807852804032304491262
#define C1 0.9238795325112867561282
#define C2 0.8314696123025452370788
#define C3 0.7071067811865475244008
#define C4 0.5555702330196022247428
#define C5 0.3826834323650897717285
#define C6 0.1950903220161282678483
__constant__ double2 kTw32d[32] = {
    {1, 0}, {C0, C6}, {C1, C5}, {C2, C4}, {C3, C3}, {C4, C2}, {C5, C1}, {C6, C0},
    {0, 1}, {-C6, C0}, {-C5, C1}, {-C4, C2}, {-C3, C3}, {-C2, C4}, {-C1, C5}, {-C0, C6},
    {-1, 0}, {-C0, -C6}, {-C1, -C5}, {-C2, -C4}, {-C3, -C3}, {-C4, -C2}, {-C5, -C1}, {-C6, -C0},
    {0, -1}, {C6, -C0}, {C5, -C1}, {C4, -C2}, {C3, -C3}, {C2, -C4}, {C1, -C5}, {C0, -C6}};
__constant__ float2 kTw32f[32] = {
    {1, 0}, {(float)C0, (float)C6}, {(float)C1, (float)C5}, {(float)C2, (float)C4}, {(float)C3, (float)C3},
    {(float)C4, (float)C2}, {(float)C5, (float)C1}, {(float)C6, (float)C0}, {0, 1}, {(float)-C6, (float)C0},
    {(float)-C5, (float)C1}, {(float)-C4, (float)C2}, {(float)-C3, (float)C3}, {(float)-C2, (float)C4},
    {(float)-C1, (float)C5}, {(float)-C0, (float)C6}, {-1, 0}, {(float)-C0, (float)-C6}, {(float)-C1, (float)-C5},
    {(float)-C2, (float)-C4}, {(float)-C3, (float)-C3}, {(float)-C4, (float)-C2}, {(float)-C5, (float)-C1},
    {(float)-C6, (float)-C0}, {0, -1}, {(float)C6, (float)-C0}, {(float)C5, (float)-C1}, {(float)C4, (float)-C2},
    {(float)C3, (float)-C3}, {(float)C2, (float)-C4}, {(float)C1, (float)-C5}, {(float)C0, (float)-C6}};
#undef C0
#undef C1
#undef C2
#undef C3
#undef C4
#undef C5
#undef C6

template <typename V> __device__ __forceinline__ V tw32(int j);
template <> __device__ __forceinline__ float2 tw32<float2>(int j) { return kTw32f[j]; }
template <> __device__ __forceinline__ double2 tw32<double2>(int j) { return kTw32d[j]; }

// Compile-time loops: f(Idx<I>) for I = 0..N-1, so that every register-array index
// below is a constant expression.
template <int I> struct Idx {
    __host__ __device__ constexpr operator int() const { return I; }
};
template <typename F, int... Is>
__device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, Is...>)
{
    (f(Idx<Is>{}), ...);
}
template <int N, typename F>
__device__ __forceinline__ void sfor(F&& f)
{
    sfor_impl(f, std::make_integer_sequence<int, N>{});
}

__host__ __device__ constexpr int bitrev(int i, int R)
{
    int j = 0;
    for (int b = 1; b < R; b <<= 1, i >>= 1) j = (j << 1) | (i & 1);
    return j;
}
__host__ __device__ constexpr int ilog2c(int R) { return R <= 1 ? 0 : 1 + ilog2c(R / 2); }

// One butterfly, (u, t) -> (u + w t, u - w t), w = e^{2 pi i k / len}.  In FP64, whose pipe the
// FP64 transforms are bound by, a general w takes six fused multiply-adds (u + w t, then
// 2 u - (u + w t)) instead of a product and two sums, eight; in FP32, bound by memory, the
// product form.  With the twiddles between the levels taken the same way (line_part), the
// packed FP64 passes of 128^3 took 405, 290 and 302 us (z, y, x) against 460, 344 and 358.
template <int k, int len, typename V>
__device__ __forceinline__ void butterfly(V& a, V& b)
{
    const V u = a;
    V t = b;
    if constexpr (k != 0 && 4 * k != len && sizeof(V) == 16) {
        const V w = tw32<V>(k * (32 / len));
        a = mk<V>(fma(-w.y, t.y, fma(w.x, t.x, u.x)), fma(w.y, t.x, fma(w.x, t.y, u.y)));
        b = mk<V>(fma(2.0, u.x, -a.x), fma(2.0, u.y, -a.y));
    } else {
        if constexpr (k != 0) {
            if constexpr (4 * k == len) t = cmuli(t);
            else t = cmul(t, tw32<V>(k * (32 / len)));
        }
        a = cadd(u, t);
        b = csub(u, t);
    }
}

// The stages of dft_reg from butterflies of length 2 << S0 on, on bit-reversed values.
template <int R, int S0, typename V>
__device__ __forceinline__ void dft_stages(V* v)
{
    sfor<ilog2c(R) - S0>([&](auto S) {
        constexpr int len = 2 << (S + S0);
        sfor<R / len>([&](auto B) {
            constexpr int i = B * len;
            sfor<len / 2>([&](auto K) {
                constexpr int k = K;
                butterfly<k, len>(v[i + k], v[i + k + len / 2]);
            });
        });
    });
}

template <int R, typename V>
__device__ __forceinline__ void bit_reverse(V* v)
{
    sfor<R>([&](auto I) {
        constexpr int i = I, j = bitrev(I, R);
        if constexpr (i < j) {
            const V t = v[i];
            v[i] = v[j];
            v[j] = t;
        }
    });
}

// In-place inverse DFT of R <= 32 values in registers, X_k = sum_n v_n e^{+2 pi i n k / R}:
// iterative radix-2 Cooley-Tukey on a bit-reversed copy.
template <int R, typename V>
__device__ __forceinline__ void dft_reg(V* v)
{
    bit_reverse<R>(v);
    dft_stages<R, 0>(v);
}

// ---- the line transform: N = N1 N2, two levels ----------------------------------
// X[k1 + N1 k2] = sum_n2 w_N2^(n2 k2) [ w_N^(n2 k1) sum_n1 x[N2 n1 + n2] w_N1^(n1 k1) ],
// w_M = e^{2 pi i / M}.  Thread n2 holds x[N2 n1 + n2] (n1 = 0..N1-1), transforms them
// and applies w_N^(n2 k1); one padded shared-memory transpose; thread t then does
// the N2-point transforms of k1 = t, t + N2, ... (G = N1 / N2 of them).
template <int N> struct Split;
template <> struct Split<8> { static constexpr int N1 = 4, N2 = 2; };
template <> struct Split<16> { static constexpr int N1 = 4, N2 = 4; };
template <> struct Split<32> { static constexpr int N1 = 8, N2 = 4; };
template <> struct Split<64> { static constexpr int N1 = 8, N2 = 8; };
template <> struct Split<128> { static constexpr int N1 = 16, N2 = 8; };
template <> struct Split<256> { static constexpr int N1 = 16, N2 = 16; };
template <> struct Split<512> { static constexpr int N1 = 32, N2 = 16; };

template <int N> struct Shape {
    static constexpr int N1 = Split<N>::N1, N2 = Split<N>::N2, G = N1 / N2;
    static constexpr int T = N2;                               // threads per line
    static constexpr int TS0 = N2 * (N1 + 1);                  // transpose buffer per line (elements)
    // y and z passes: TX lines (consecutive x) per block, lane = xo + TX t.
    static constexpr int TX0 = 128 / T > 16 ? 128 / T : 16;
    static constexpr int TX = TX0 < N ? TX0 : N;
    static constexpr int THREADS = TX * T;
    // Line stride of the y and z passes' transpose buffers, in elements of E bytes.  One
    // shared-memory wavefront serves 128 bytes: P = 128 / E consecutive lanes over P bank
    // groups.  Lane xo + TXl t touches element n2 (N1 + 1) + k of the line at xo * stride
    // (n2 = t, N1 + 1 odd).  With stride = P / TXl (mod P) for TXl < P (a wavefront spans
    // P / TXl values of t), else 1 (mod P), the P lanes fall in P distinct bank groups.
    template <int E, int TXl>
    __host__ __device__ static constexpr int line_stride()
    {
        constexpr int P = 128 / E;
        constexpr int S = TXl < P ? P / TXl : 1;
        return TS0 + ((S - TS0 % P) % P + P) % P;
    }
    // x pass: XL lines of each of the four grids per block, lane = t + T (line): 64 threads up to
    // N = 64 (N = 32: 256 blocks for 64, an FP64 build 38.6 -> 34.8 us), then 256; transpose
    // stride TSX = T (mod 16), result rows of XPS elements.
    static constexpr int XL = (N <= 64 ? 64 : 256) / (4 * T);
    static constexpr int THREADS_X = 4 * XL * T;
    static constexpr int SX = T % 16;
    static constexpr int TSX = TS0 + ((SX - TS0 % 16) + 16) % 16;
    static constexpr int XPS = N;
    template <typename V> static constexpr size_t x_smem()
    {
        return (size_t)(N2 * (N1 + 1) + 4 * XL * (TSX > XPS ? TSX : XPS)) * sizeof(V);
    }
    static constexpr int TWS = N2 * (N1 + 1);                  // per-thread twiddle rows, padded
    // z pass: 128 threads (its per-thread amplitudes live in shared memory) that form all four
    // packed grids in turn.  Up to N = 64 that would be N^2 T / 128 <= 256 blocks of a long
    // chain for 152 SMs: there a block is 8 columns of one grid (N = 32 in FP64: 512 blocks of
    // 32 threads for 32 of 128, 28 -> 13 us a pass when FP64 took this path).
    static constexpr bool kSplitGrids = N <= 64;
    static constexpr int TZ0 = kSplitGrids ? 8 : 128 / T;
    static constexpr int TZ = TZ0 < N ? TZ0 : N;
    static constexpr int THREADS_Z = TZ * T;
    // the half-spectrum passes' tiles, of rows of N / 2
    static constexpr int HX = TX0 < N / 2 ? TX0 : N / 2;
    static constexpr int HZ = TZ0 < N / 2 ? TZ0 : N / 2;
};

// The half-spectrum work array: arrays of N^2 (N/2) values [z][y][x].  The z pass writes the
// first five, the y pass transforms 1, 3 and 4 in place and 0 and 2 twice, into the last four.
enum Half { kHPsi0, kHDzPsi, kHPhi0, kHDzPhi, kHDot, kHPsi, kHDyPsi, kHPhi, kHDyPhi };
constexpr int kHalfZ = 5, kHalfY = 7;

// Twiddles of the first level, w_N^(n2 k1) at [n2 (N1 + 1) + k1]: a thread reads its
// own row, and lanes with different n2 fall in different banks.
template <typename V, int N>
__device__ __forceinline__ void load_line_twiddles(V* s_tw2, const V* __restrict__ tw)
{
    constexpr int N1 = Shape<N>::N1, N2 = Shape<N>::N2;
    for (int i = threadIdx.x; i < N1 * N2; i += blockDim.x) {
        const int n2 = i / N1, k1 = i - n2 * N1;
        s_tw2[n2 * (N1 + 1) + k1] = tw[(n2 * k1) & (N - 1)];
    }
}

template <typename V, int N>
__device__ __forceinline__ void line_first(V* v, int n2, const V* __restrict__ s_tw, V* tr)
{
    constexpr int N1 = Shape<N>::N1;
    dft_reg<N1>(v);
    if constexpr (sizeof(V) == 16) {
        // the twiddles go into the second level's first butterflies (line_part)
        sfor<N1>([&](auto K1) { tr[n2 * (N1 + 1) + K1] = v[K1]; });
    } else {
        const V* row = s_tw + n2 * (N1 + 1);
        sfor<N1>([&](auto K1) { tr[n2 * (N1 + 1) + K1] = cmul(v[K1], row[K1]); });
    }
}

// The second level of one k1: u[k2] = X[k1 + N1 k2].
template <typename V, int N>
__device__ __forceinline__ void line_part(int k1, const V* tr, const V* __restrict__ s_tw, V* u)
{
    constexpr int N1 = Shape<N>::N1, N2 = Shape<N>::N2;
    sfor<N2>([&](auto N2i) { u[N2i] = tr[N2i * (N1 + 1) + k1]; });
    if constexpr (sizeof(V) == 16) {
        // a w_a +- b w_b: ten fused multiply-adds (six for n2 = 0, where w_a = 1) instead of two
        // products and two sums, twelve
        sfor<N2 / 2>([&](auto J) {
            constexpr int j = J, h = J + N2 / 2;
            const V wb = s_tw[h * (N1 + 1) + k1], b = u[h];
            V a = u[j];
            if constexpr (j != 0) a = cmul(a, s_tw[j * (N1 + 1) + k1]);
            u[j] = mk<V>(fma(-wb.y, b.y, fma(wb.x, b.x, a.x)), fma(wb.y, b.x, fma(wb.x, b.y, a.y)));
            u[h] = mk<V>(fma(2.0, a.x, -u[j].x), fma(2.0, a.y, -u[j].y));
        });
        bit_reverse<N2>(u);
        dft_stages<N2, 1>(u);
    } else {
        dft_reg<N2>(u);
    }
}

// Second level for k1 = t + g N2; out(k2, value) receives X[k1 + N1 k2].
template <typename V, int N, typename Out>
__device__ __forceinline__ void line_second(int t, const V* tr, const V* __restrict__ s_tw, Out&& out)
{
    constexpr int N1 = Shape<N>::N1, N2 = Shape<N>::N2, G = Shape<N>::G;
    sfor<G>([&](auto Gi) {
        const int k1 = t + Gi * N2;
        V u[N2];
        line_part<V, N>(k1, tr, s_tw, u);
        sfor<N2>([&](auto K2) { out(k1 + N1 * K2, u[K2]); });
    });
}

// ---- precision-dependent scalar math -------------------------------------
__device__ __forceinline__ float f_log(float x) { return logf(x); }
__device__ __forceinline__ double f_log(double x) { return log(x); }
__device__ __forceinline__ float f_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double f_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ void f_sincospi(float x, float* s, float* c) { sincospif(x, s, c); }
__device__ __forceinline__ void f_sincospi(double x, double* s, double* c) { sincospi(x, s, c); }

// |n| < 2^20 in FP64, in integer operations: the conversion would take a slot of the FP64 pipe.
__device__ __forceinline__ double small_int(int n)
{
    const uint32_t f = __float_as_uint((float)n);
    return __hiloint2double((int)(n == 0 ? 0u : (f & 0x80000000u) | (((f & 0x7FFFFFFFu) >> 3) + 0x38000000u)), 0);
}

__device__ __forceinline__ int sidx(int j, int N) { return j < (N >> 1) ? j : j - N; }

// The unit Gaussian of mode (jx, jy, jz), R/sqrt(P_R/V): zero for the mean and the
// Nyquist planes, conj of the mirror mode for non-canonical n.  Drawn once per run
// by k_noise.
template <typename V>
__device__ __forceinline__ V mode_unit(const FieldArgs& a, int jx, int jy, int jz)
{
    using T = typename Real<V>::T;
    const int N = a.N;
    const int nx = sidx(jx, N), ny = sidx(jy, N), nz = sidx(jz, N);
    const int h = -(N >> 1);
    if (nx == h || ny == h || nz == h || (nx == 0 && ny == 0 && nz == 0)) return mk<V>(T(0), T(0));
    const bool canon = nz > 0 || (nz == 0 && (ny > 0 || (ny == 0 && nx > 0)));
    const int mx = canon ? nx : -nx, my = canon ? ny : -ny, mz = canon ? nz : -nz;
    const uint64_t pack = (uint64_t)(uint32_t)(mx + (1 << 20)) | ((uint64_t)(uint32_t)(my + (1 << 20)) << 21) |
                          ((uint64_t)(uint32_t)(mz + (1 << 20)) << 42);
    const uint4 w = philox4x32_10(make_uint4((uint32_t)pack, (uint32_t)(pack >> 32), 16u, 0u), a.key0, a.key1);
    const T u1 = (T)((w.x >> 8) + 1u) * (T)5.9604644775390625e-08;  // (0, 1]
    const T u2 = (T)(w.y >> 8) * (T)5.9604644775390625e-08;         // [0, 1)
    T s, c;
    f_sincospi((T)2 * u2, &s, &c);
    T re, im;
    if (a.fixed_amp) {
        re = c;
        im = s;
    } else {
        const T r = f_sqrt((T)-2 * f_log(u1)) * (T)0.70710678118654752440;
        re = r * c;
        im = r * s;
    }
    if (!canon) im = -im;
    return mk<V>(re, im);
}

// The N^3 mode array, drawn by `blocks` blocks of which this is number `block`.
template <typename V>
__device__ __forceinline__ void noise_part(const FieldArgs& a, V* __restrict__ R, unsigned block, unsigned blocks)
{
    const int N = a.N;
    const size_t N3 = (size_t)N * N * N;
    for (size_t c = block * (size_t)blockDim.x + threadIdx.x; c < N3; c += (size_t)blocks * blockDim.x) {
        const int jx = (int)(c % N), jy = (int)((c / N) % N), jz = (int)(c / ((size_t)N * N));
        R[c] = mode_unit<V>(a, jx, jy, jz);
    }
}

template <typename V>
__global__ void __launch_bounds__(256) k_noise(FieldArgs a, V* __restrict__ R)
{
    noise_part<V>(a, R, blockIdx.x, gridDim.x);
}

// Packed spectrum p of a mode with unit Gaussian R and amplitudes (Apsi, Aphi, Adot):
//   P0 = i kx Apsi R + i (i ky Apsi R)      (d_x psi + i d_y psi)
//   P1 = i kz Apsi R + i (i kx Aphi R)      (d_z psi + i d_x phi)
//   P2 = i ky Aphi R + i (i kz Aphi R)      (d_y phi + i d_z phi)
//   P3 = Adot R + i Apsi R                  (phi_dot + i psi)
template <typename V>
__device__ __forceinline__ V packed(int p, V R, typename Real<V>::T Apsi, typename Real<V>::T Aphi,
                                    typename Real<V>::T Adot, typename Real<V>::T kx, typename Real<V>::T ky,
                                    typename Real<V>::T kz)
{
    const V iR = cmuli(R);
    switch (p) {
        case 0: return mk<V>(Apsi * (kx * iR.x - ky * R.x), Apsi * (kx * iR.y - ky * R.y));
        case 1: return mk<V>(kz * Apsi * iR.x - kx * Aphi * R.x, kz * Apsi * iR.y - kx * Aphi * R.y);
        case 2: return mk<V>(Aphi * (ky * iR.x - kz * R.x), Aphi * (ky * iR.y - kz * R.y));
        default: return mk<V>(Adot * R.x + Apsi * iR.x, Adot * R.y + Apsi * iR.y);
    }
}

// In FP64, for every m = |n|^2 in [0, M): k = k_f sqrt(m), the amplitude sqrt(P_R(k)/V) =
// sqrt(2 pi^2 A_s / V) k^-3/2 (k/k_pivot)^((n_s-1)/2) and k's place in the transfer tables'
// uniform ln k grid (clamped): what no step changes.  Once per run: its chain of a root, a
// logarithm, an exponential and a division takes 10 us however small the grid is.
__device__ __forceinline__ ModeKey mode_key(const FieldArgs& a, int m)
{
    ModeKey key{0.0, 0.0, 0, 0};
    if (m > 0) {
        const double k = a.kf * sqrt((double)m);
        const double lnk = log(k);
        key.amp = a.amp0 / (k * sqrt(k)) * exp(a.half_nsm1 * (lnk - a.lnkp));
        const double pos = (lnk - a.lnk0) * a.inv_dlnk;
        if (pos <= 0.0) {
            key.ik = 0;
            key.fk = 0.0;
        } else if (pos >= a.nk - 1) {
            key.ik = a.nk - 2;
            key.fk = 1.0;
        } else {
            key.ik = (int)pos;
            key.fk = pos - key.ik;
        }
    }
    return key;
}

__global__ void __launch_bounds__(256) k_mode_keys(FieldArgs a, int M, ModeKey* __restrict__ keys)
{
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x) keys[m] = mode_key(a, m);
}

// A mode's four table values from rows ia and ia + 1 of the FP64 tables [3][na][nk].
template <typename T>
__device__ __forceinline__ void mode_values(const ModeKey& key, int ia, double fa, double aH, int na, int nk,
                                            const double* __restrict__ tabs, T* __restrict__ out)
{
    double v[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        const double* r0 = tabs + ((size_t)t * na + ia) * nk;
        const double* r1 = r0 + nk;
        const double v0 = (1.0 - key.fk) * r0[key.ik] + key.fk * r0[key.ik + 1];
        const double v1 = (1.0 - key.fk) * r1[key.ik] + key.fk * r1[key.ik + 1];
        v[t] = key.amp * ((1.0 - fa) * v0 + fa * v1);
    }
    v[2] *= aH;
    out[0] = (T)v[0];
    out[1] = (T)v[1];
    out[2] = (T)v[2];
    out[3] = T(0);
}

// Per scale factor and m: the amplitude times T_psi, T_phi and a H dT_phi/dln a, read
// bilinearly in (ln k, ln a) from the FP64 tables [3][na][nk].  One launch makes the tables
// of every step of a pass (blockIdx.y).
template <typename T>
__global__ void __launch_bounds__(256) k_mode_tables(const __grid_constant__ ModeSteps st, int M, int nk, int na,
                                                     const ModeKey* __restrict__ keys, const double* __restrict__ tabs,
                                                     T* __restrict__ A)
{
    const int b = blockIdx.y;
    T* out = A + (size_t)b * 4 * M;
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M; m += gridDim.x * blockDim.x)
        mode_values<T>(keys[m], st.ia[b], st.fa[b], st.aH[b], na, nk, tabs, out + 4 * (size_t)m);
}

// Both parts of a build that keeps nothing, in one launch: the first blocks make the
// amplitude table of one scale factor, the others draw the mode array.
template <typename V>
__global__ void __launch_bounds__(256) k_modes_once(FieldArgs a, int M, const double* __restrict__ tabs,
                                                    typename Real<V>::T* __restrict__ A, V* __restrict__ R)
{
    const unsigned nm = (unsigned)((M + 255) / 256);
    if (blockIdx.x >= nm) {
        noise_part<V>(a, R, blockIdx.x - nm, gridDim.x - nm);
        return;
    }
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < M) mode_values(mode_key(a, m), a.ia, a.fa, a.aH, a.na, a.nk, tabs, A + 4 * (size_t)m);
}

// One entry of the FP32 amplitude table (4 values per |n|^2) in one load.
__device__ __forceinline__ void amp_entry(const float* A, int m, float& ap, float& af, float& ad)
{
    const float4 v = __ldg(reinterpret_cast<const float4*>(A) + m);
    ap = v.x;
    af = v.y;
    ad = v.z;
}

// ---- pass z: spectrum + inverse DFT along z ---------------------------------
// Block (x-tile, jy): TX columns along z.  Each thread reads the unit Gaussians of
// its N1 modes once, with their amplitudes A[|n|^2] at this scale factor, then forms,
// transforms and writes each of the four packed grids in turn.  Its shared-memory traffic (two
// transposes per grid, the amplitudes) needs warps to hide it: with the amplitudes of half the
// modes in shared memory (44 -> 32 KB a block) and 96 registers, five blocks per SM instead of
// four; N = 256: a build 493 -> 478 us (FP32), 458 -> 443 us (BF16); six blocks of 80 registers:
// 487 and 452; N = 128: 67.0, 66.7 and 66.2 us.
template <typename V, int N>
__global__ void __launch_bounds__(Shape<N>::THREADS_Z, N >= 512 ? 4 : 5) k_fields_z(FieldArgs a,
                                                                  const typename Real<V>::T* __restrict__ A,
                                                                  const V* __restrict__ R, const V* __restrict__ tw,
                                                                  V* __restrict__ W)
{
    using T = typename Real<V>::T;
    using S = Shape<N>;
    constexpr int TX = S::TZ, N1 = S::N1, N2 = S::N2, NT = S::THREADS_Z;
    constexpr int TSZ = S::template line_stride<sizeof(V), S::TZ>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* s_tw = reinterpret_cast<V*>(smem_raw);
    V* tr = s_tw + S::TWS;                                  // TX * TSZ
    T* As = reinterpret_cast<T*>(tr + TX * TSZ);            // [3][N1 / 2][NT]: each thread's own column
    load_line_twiddles<V, N>(s_tw, tw);
    const int xo = threadIdx.x % TX, t = threadIdx.x / TX;
    const int x0 = blockIdx.x * TX, jy = blockIdx.y;
    const int nx = sidx(x0 + xo, N), ny = sidx(jy, N), h = -(N >> 1);
    const T kf = (T)a.kf;
    const T kx = kf * (T)nx, ky = kf * (T)ny;
    const size_t NN = (size_t)N * N;
    V Rv[N1];
    sfor<N1>([&](auto I) { Rv[I] = R[(size_t)(N2 * I + t) * NN + (size_t)jy * N + x0 + xo]; });
    // The amplitudes depend on |n|^2 only, so the modes nz and -nz of a column share
    // them: each thread looks up the first half of its modes, nz >= 0.  Mode z = N2 I + t
    // mirrors to z' = N - z: for t > 0 that is thread N2 - t, index N1 - 1 - I; for t = 0 it
    // is thread 0, index N1 - I (I = N1 / 2: the Nyquist mode, zero).
    constexpr int NH = N1 / 2;
    sfor<NH>([&](auto I) {
        const int nz = N2 * I + t;
        T ap = T(0), af = T(0), ad = T(0);
        if (nx != h && ny != h) amp_entry(A, nx * nx + ny * ny + nz * nz, ap, af, ad);
        As[(0 * NH + I) * NT + threadIdx.x] = ap;
        As[(1 * NH + I) * NT + threadIdx.x] = af;
        As[(2 * NH + I) * NT + threadIdx.x] = ad;
    });
    const int mirror = t == 0 ? (int)threadIdx.x + NT : xo + TX * (N2 - t);
    auto amp = [&](int slot, auto I) {
        const T* Aq = As + slot * NH * NT;
        if constexpr (I < NH) return Aq[I * NT + threadIdx.x];
        else return I == NH && t == 0 ? T(0) : Aq[(N1 - 1 - I) * NT + mirror];
    };
    __syncthreads();
    const size_t N3 = NN * N;
    // this block's packed grids: all of them, or one of gridDim.z
    const int p0 = gridDim.z == 1 ? 0 : blockIdx.z, p1 = gridDim.z == 1 ? a.grids : p0 + 1;
#pragma unroll 1
    for (int p = p0; p < p1; ++p) {
        // one branch per packed grid, so that each reads only the amplitudes it uses
        // (psi; psi and phi; phi; phi_dot and psi) from shared memory
        V v[N1];
        // Q = 4 is grid 3 with slot 7 = phi + psi (the exact drift's factor), Q = 5 grid 3
        // with slot 7 = 0 (phi_dot transformed alone)
        auto form = [&](auto Q) {
            constexpr int P = Q < 4 ? (int)Q : 3;
            sfor<N1>([&](auto I) {
                const T kz = kf * (T)sidx(N2 * I + t, N);
                const T apsi = (P == 2 || Q == 5) ? T(0) : amp(0, I);
                const T aphi = (P == 1 || P == 2 || Q == 4) ? amp(1, I) : T(0);
                const T adot = (P == 3) ? amp(2, I) : T(0);
                v[I] = packed<V>(P, Rv[I], Q == 4 ? apsi + aphi : apsi, aphi, adot, kx, ky, kz);
            });
        };
        switch (p) {
            case 0: form(Idx<0>{}); break;
            case 1: form(Idx<1>{}); break;
            case 2: form(Idx<2>{}); break;
            case 4: form(Idx<3>{}); break;
            default:
                if (a.slot7 == kSlot7Sum) form(Idx<4>{});
                else if (a.slot7 == kSlot7Zero) form(Idx<5>{});
                else form(Idx<3>{});
                break;
        }
        line_first<V, N>(v, t, s_tw, tr + xo * TSZ);
        __syncthreads();
        V* dst = W + p * N3 + (size_t)jy * N + x0 + xo;
        line_second<V, N>(t, tr + xo * TSZ, s_tw, [&](int z, V val) { dst[(size_t)z * NN] = val; });
        __syncthreads();
    }
}

// ---- pass y: inverse DFT along y --------------------------------------------
// Block (x-tile, jz, packed grid p): TX lines along y, read and written in place in rows
// of TX consecutive x.
template <typename V, int N>
__global__ void __launch_bounds__(Shape<N>::THREADS) k_fields_y(const V* __restrict__ tw, V* W)
{
    using S = Shape<N>;
    constexpr int TX = S::TX, N1 = S::N1, N2 = S::N2;
    constexpr int TS = S::template line_stride<sizeof(V), S::TX>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* s_tw = reinterpret_cast<V*>(smem_raw);
    V* tr = s_tw + S::TWS;
    load_line_twiddles<V, N>(s_tw, tw);
    const int xo = threadIdx.x % TX, t = threadIdx.x / TX;
    const int x0 = blockIdx.x * TX, jz = blockIdx.y, p = blockIdx.z;
    const size_t N3 = (size_t)N * N * N;
    V* dst = W + p * N3 + (size_t)jz * N * N + x0 + xo;
    V v[N1];
    sfor<N1>([&](auto N1i) { v[N1i] = dst[(size_t)(N2 * N1i + t) * N]; });
    __syncthreads();
    line_first<V, N>(v, t, s_tw, tr + xo * TS);
    __syncthreads();
    line_second<V, N>(t, tr + xo * TS, s_tw, [&](int y, V val) { dst[(size_t)y * N] = val; });
}

// ---- the half-spectrum passes z and y (FP64) ----------------------------------
// All three FP64 passes are bound by the FP64 pipe (84-85 % busy), so the transforms that half
// spectra save are time: 128^3, a build 997 -> 857 us (z 405 -> 238, y 290 -> 280, x 302 -> 340,
// which now forms its lines and d_x); a run of 100 steps 158 -> 145 ms, and 5.16 -> 4.2 ms at 32^3.
// Block (array f and x tile, jy): HZ columns along z of one of the five arrays, the real
// fields' spectra A R or i k_z A R.  The array index runs fastest, so that the five blocks
// that read the same unit Gaussians run together.
template <int N>
__global__ void __launch_bounds__(Shape<N>::HZ * Shape<N>::T, Shape<N>::N1 == 32 ? 2 : 4)
    k_half_z(FieldArgs a, const double* __restrict__ A, const double2* __restrict__ R, const double2* __restrict__ tw,
             double2* __restrict__ W)
{
    using S = Shape<N>;
    constexpr int TX = S::HZ, N1 = S::N1, N2 = S::N2, NT = TX * S::T;
    constexpr int TSZ = S::template line_stride<16, TX>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* s_tw = reinterpret_cast<double2*>(smem_raw);
    double2* tr = s_tw + S::TWS;                            // TX * TSZ
    double* As = reinterpret_cast<double*>(tr + TX * TSZ);  // [N1][NT]: each thread's own column
    load_line_twiddles<double2, N>(s_tw, tw);
    const int xo = threadIdx.x % TX, t = threadIdx.x / TX;
    const int f = blockIdx.x % kHalfZ, x0 = blockIdx.x / kHalfZ * TX, jy = blockIdx.y;
    const int nx = x0 + xo, ny = sidx(jy, N), h = -(N >> 1);
    const bool dz = f == kHDzPsi || f == kHDzPhi;
    const size_t NN = (size_t)N * N;
    double2 v[N1];
    sfor<N1>([&](auto I) { v[I] = R[(size_t)(N2 * I + t) * NN + (size_t)jy * N + nx]; });
    // The amplitudes, each looked up once for the modes nz and -nz (as in k_fields_z); a z
    // gradient's factor k_z A changes sign between them.
    {
        const double* row = A + (f <= kHDzPsi ? 0 : f <= kHDzPhi ? 1 : 2);
        const int tp = t == 0 ? 0 : N2 - t;
        const int partner = xo + TX * tp;
        sfor<N1 / 2 + 1>([&](auto I) {
            if (I < N1 / 2 || t == 0) {
                const int nz = sidx(N2 * I + t, N);
                const int Ip = t == 0 ? (N1 - I) % N1 : N1 - 1 - I;
                double ap = 0.0;
                if (ny != h && nz != h) ap = __ldg(row + 4 * (size_t)(nx * nx + ny * ny + nz * nz));
                if (dz) ap *= a.kf * small_int(nz);
                As[I * NT + threadIdx.x] = ap;
                As[Ip * NT + partner] = dz ? -ap : ap;
            }
        });
    }
    __syncthreads();
    sfor<N1>([&](auto I) {
        const double ap = As[I * NT + threadIdx.x];
        const double re = ap * v[I].x, im = ap * v[I].y;
        v[I] = dz ? make_double2(-im, re) : make_double2(re, im);
    });
    line_first<double2, N>(v, t, s_tw, tr + xo * TSZ);
    __syncthreads();
    double2* dst = W + f * (NN * (N / 2)) + (size_t)jy * (N / 2) + nx;
    line_second<double2, N>(t, tr + xo * TSZ, s_tw, [&](int z, double2 val) { dst[(size_t)z * (NN / 2)] = val; });
}

// Block (transform q and x tile, jz): HX lines along y of one of the seven transforms, the y
// gradients multiplied by i k_y as they are read.
template <int N>
__global__ void __launch_bounds__(Shape<N>::HX * Shape<N>::T) k_half_y(double kf, const double2* __restrict__ tw,
                                                                        double2* W)
{
    using S = Shape<N>;
    constexpr int TX = S::HX, N1 = S::N1, N2 = S::N2;
    constexpr int TS = S::template line_stride<16, TX>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* s_tw = reinterpret_cast<double2*>(smem_raw);
    double2* tr = s_tw + S::TWS;
    load_line_twiddles<double2, N>(s_tw, tw);
    const int xo = threadIdx.x % TX, t = threadIdx.x / TX;
    const int q = blockIdx.x % kHalfY, x0 = blockIdx.x / kHalfY * TX, jz = blockIdx.y;
    // psi, d_y psi, phi, d_y phi (out of place: their sources are read twice), then in place
    const int src = q < 2 ? kHPsi0 : q < 4 ? kHPhi0 : q == 4 ? kHDzPsi : q == 5 ? kHDzPhi : kHDot;
    const int to = q < 4 ? kHPsi + q : src;
    const size_t NH = (size_t)N * (N / 2), N3H = NH * N;
    const size_t at = (size_t)jz * NH + x0 + xo;
    double2 v[N1];
    sfor<N1>([&](auto I) { v[I] = W[src * N3H + at + (size_t)(N2 * I + t) * (N / 2)]; });
    if (q == 1 || q == 3)
        sfor<N1>([&](auto I) {
            const double ky = kf * small_int(sidx(N2 * I + t, N));
            v[I] = make_double2(-ky * v[I].y, ky * v[I].x);
        });
    __syncthreads();
    line_first<double2, N>(v, t, s_tw, tr + xo * TS);
    __syncthreads();
    double2* dst = W + to * N3H + at;
    line_second<double2, N>(t, tr + xo * TS, s_tw, [&](int y, double2 val) { dst[(size_t)y * (N / 2)] = val; });
}

// The x spectrum of packed grid p (4: grid 3 as kSlot7Psi has it) along one line, thread t's
// values, from the half spectra: F(N - k) = conj F(k), F(N/2) = 0.
//   P0 = i (k_x psi + d_y psi)    P1 = d_z psi - k_x phi    P2 = d_y phi + i d_z phi
//   P3 = phi_dot + i psi, phi_dot + i (phi + psi) or phi_dot
template <int N>
__device__ __forceinline__ void half_line(double2* v, int p, int t, double kf, int slot7, size_t line,
                                          const double2* __restrict__ W)
{
    constexpr int N1 = Shape<N>::N1, N2 = Shape<N>::N2;
    const size_t N3H = (size_t)N * N * (N / 2);
    const double2* a = W + line * (N / 2) + N3H * (p == 0 ? kHDyPsi : p == 1 ? kHDzPsi : p == 2 ? kHDyPhi : kHDot);
    const double2* b = W + line * (N / 2) + N3H * (p == 1 ? kHPhi : p == 2 ? kHDzPhi : kHPsi);
    auto each = [&](auto&& f) {
        sfor<N1>([&](auto I) {
            const int k = N2 * I + t;
            if constexpr (I < N1 / 2) {
                v[I] = f(k, [&](const double2* s) { return s[k]; });
            } else {
                if (I == N1 / 2 && t == 0) v[I] = make_double2(0.0, 0.0);
                else
                    v[I] = f(k - N, [&](const double2* s) {
                        const double2 u = s[N - k];
                        return make_double2(u.x, -u.y);
                    });
            }
        });
    };
    if (p < 2) {
        const double kp = p == 0 ? kf : -kf;
        each([&](int n, auto&& get) {
            const double2 u = get(a), w = get(b);
            const double k = kp * small_int(n), x = fma(k, w.x, u.x), y = fma(k, w.y, u.y);
            return p == 0 ? make_double2(-y, x) : make_double2(x, y);
        });
    } else if (p == 3 && slot7 == kSlot7Zero) {
        each([&](int, auto&& get) { return get(a); });
    } else if (p == 3 && slot7 == kSlot7Sum) {
        const double2* c = W + line * (N / 2) + N3H * kHPhi;
        each([&](int, auto&& get) {
            const double2 u = get(a), w = get(b), z = get(c);
            return make_double2(u.x - (w.y + z.y), u.y + (w.x + z.x));
        });
    } else {
        each([&](int, auto&& get) {
            const double2 u = get(a), w = get(b);
            return make_double2(u.x - w.y, u.y + w.x);
        });
    }
}

// Thread t's values of a line of packed grid p: read (FP32) or formed (FP64).
template <typename V, int N>
__device__ __forceinline__ void x_line(V* v, int p, int t, double kf, int slot7, size_t line, const V* __restrict__ W)
{
    if constexpr (sizeof(V) == 16) {
        half_line<N>(v, p, t, kf, slot7, line, W);
    } else {
        const V* src = W + p * ((size_t)N * N * N) + line * N;
        sfor<Shape<N>::N1>([&](auto I) { v[I] = src[Shape<N>::N2 * I + t]; });
    }
}

// ---- pass x: inverse DFT along x, interleave into G[cell][8] ----------------
template <typename Gt, typename V> struct GRec;
template <> struct GRec<float, float2> {
    // one 32-byte store per record (the record is 32-byte aligned)
    __device__ static void put(float* G, size_t cell, float2 a, float2 b, float2 c, float2 d)
    {
        float* g = G + 8 * cell;
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(g), "f"(a.x), "f"(a.y),
                     "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y), "f"(d.x), "f"(d.y)
                     : "memory");
    }
};
template <> struct GRec<double, double2> {
    // two 32-byte stores per record
    __device__ static void put(double* G, size_t cell, double2 a, double2 b, double2 c, double2 d)
    {
        double* g = G + 8 * cell;
        asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(g), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y)
                     : "memory");
        asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(g + 4), "d"(c.x), "d"(c.y), "d"(d.x), "d"(d.y)
                     : "memory");
    }
};
template <> struct GRec<__nv_bfloat16, float2> {
    __device__ static void put(__nv_bfloat16* G, size_t cell, float2 a, float2 b, float2 c, float2 d)
    {
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(b.x, b.y);
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(c.x, c.y), h3 = __floats2bfloat162_rn(d.x, d.y);
        uint4 u;
        u.x = *reinterpret_cast<const uint32_t*>(&h0);
        u.y = *reinterpret_cast<const uint32_t*>(&h1);
        u.z = *reinterpret_cast<const uint32_t*>(&h2);
        u.w = *reinterpret_cast<const uint32_t*>(&h3);
        reinterpret_cast<uint4*>(G)[cell] = u;
    }
};

// Block: XL consecutive x-lines (line index = jz * N + jy) of all four packed grids, one
// line of one grid per T threads.  The transforms end in shared memory ([line][grid][x],
// over the transpose buffers), from where each cell's four values leave as one whole
// record.  Every grid's threads work at once: with one set of threads that transformed
// the grids in turn and parked three of them, 69 KB of shared memory held 128 threads.
// Bound by DRAM at N = 256 (48 (BF16) or 64 (FP32) bytes per cell): BF16 records 164 ->
// 120 us; N = 128 in FP32 28.9 -> 23.8 us, N = 32 in FP64 22.9 -> 12.5 us.
template <typename V, typename Gt, int N>
__global__ void __launch_bounds__(Shape<N>::THREADS_X) k_fields_x(double kf, int slot7, const V* __restrict__ tw,
                                                                  const V* __restrict__ W, Gt* __restrict__ G)
{
    using S = Shape<N>;
    constexpr int XL = S::XL, N1 = S::N1, N2 = S::N2, T = S::T, PS = S::XPS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* s_tw = reinterpret_cast<V*>(smem_raw);
    V* tr = s_tw + S::TWS;          // 4 XL TSX transpose elements, then 4 XL PS results
    const int t = threadIdx.x % T, lp = threadIdx.x / T;
    const int lo = lp % XL, p = lp / XL;
    const size_t line0 = (size_t)blockIdx.x * XL;
    V v[N1];
    x_line<V, N>(v, p, t, kf, slot7, line0 + lo, W);
    load_line_twiddles<V, N>(s_tw, tw);
    __syncthreads();
    line_first<V, N>(v, t, s_tw, tr + lp * S::TSX);
    __syncthreads();
    V r[N1];
    sfor<S::G>([&](auto Gi) {
        V u[N2];
        line_part<V, N>(t + Gi * N2, tr + lp * S::TSX, s_tw, u);
        sfor<N2>([&](auto K2) { r[Gi * N2 + K2] = u[K2]; });
    });
    __syncthreads();
    V* park = tr + (lo * 4 + p) * PS;
    sfor<S::G>([&](auto Gi) { sfor<N2>([&](auto K2) { park[t + Gi * N2 + N1 * K2] = r[Gi * N2 + K2]; }); });
    __syncthreads();
#pragma unroll
    for (int c = threadIdx.x; c < XL * N; c += S::THREADS_X) {
        const int l = c / N, x = c % N;
        const V* q = tr + l * 4 * PS + x;
        GRec<Gt, V>::put(G, (line0 + l) * N + x, q[0], q[PS], q[2 * PS], q[3 * PS]);
    }
}

// The x pass of a build for inspection: five packed grids (the fifth is phi_dot + i psi), the
// values as a gather grid of type Gt would hold them, straight into out[8][N^3] (slots 0-5
// from grids 0-2, phi_dot from grid 3, psi from grid 4).
template <typename V, typename Gt, int N>
__global__ void __launch_bounds__(Shape<N>::THREADS) k_fields_x_planar(double kf, const V* __restrict__ tw,
                                                                       const V* __restrict__ W,
                                                                       double* __restrict__ out)
{
    using S = Shape<N>;
    constexpr int N1 = S::N1, T = S::T, LPB = S::THREADS / T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* s_tw = reinterpret_cast<V*>(smem_raw);
    V* tr = s_tw + S::TWS;
    const int t = threadIdx.x % T, lo = threadIdx.x / T, p = blockIdx.y;
    const size_t N3 = (size_t)N * N * N;
    const size_t line = (size_t)blockIdx.x * LPB + lo;
    V v[N1];
    x_line<V, N>(v, p, t, kf, kSlot7Zero, line, W);
    load_line_twiddles<V, N>(s_tw, tw);
    __syncthreads();
    line_first<V, N>(v, t, s_tw, tr + lo * S::TSX);
    __syncthreads();
    line_second<V, N>(t, tr + lo * S::TSX, s_tw, [&](int x, V val) {
        double re = val.x, im = val.y;
        if constexpr (sizeof(Gt) == 2) {
            re = (double)__bfloat162float(__float2bfloat16_rn(val.x));
            im = (double)__bfloat162float(__float2bfloat16_rn(val.y));
        }
        if (p < 4) out[(size_t)(2 * p) * N3 + line * N + x] = re;
        if (p != 3) out[(size_t)(p == 4 ? 7 : 2 * p + 1) * N3 + line * N + x] = im;
    });
}

// ---- [8][N^3] FP64 into a gather grid (test hook) ---------------------------
template <typename Gt>
__global__ void k_fields_from_f64(size_t N3, const double* __restrict__ in, Gt* __restrict__ G)
{
    for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < N3; c += (size_t)gridDim.x * blockDim.x)
        for (int s = 0; s < 8; ++s) {
            if constexpr (sizeof(Gt) == 2) G[c * 8 + s] = __float2bfloat16_rn((float)in[s * N3 + c]);
            else G[c * 8 + s] = (Gt)in[s * N3 + c];
        }
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename V, int N>
cudaError_t run_z(cudaStream_t s, const FieldArgs& a, const void* A, const void* R, const void* tw, void* W)
{
    using S = Shape<N>;
    using T = typename Real<V>::T;
    constexpr int TSZ = S::template line_stride<sizeof(V), S::TZ>();
    const size_t sm = (size_t)(S::TWS + S::TZ * TSZ) * sizeof(V) + (size_t)3 * (S::N1 / 2) * S::THREADS_Z * sizeof(T);
    cudaError_t e = set_smem(k_fields_z<V, N>, sm);
    if (e != cudaSuccess) return e;
    k_fields_z<V, N><<<dim3(N / S::TZ, N, S::kSplitGrids ? a.grids : 1), S::THREADS_Z, sm, s>>>(
        a, (const T*)A, (const V*)R, (const V*)tw, (V*)W);
    return cudaGetLastError();
}

template <int N>
cudaError_t run_half_z(cudaStream_t s, const FieldArgs& a, const void* A, const void* R, const void* tw, void* W)
{
    using S = Shape<N>;
    constexpr int NT = S::HZ * S::T;
    const size_t sm = (size_t)(S::TWS + S::HZ * S::template line_stride<16, S::HZ>()) * 16 + (size_t)S::N1 * NT * 8;
    cudaError_t e = set_smem(k_half_z<N>, sm);
    if (e != cudaSuccess) return e;
    k_half_z<N><<<dim3(kHalfZ * (N / 2 / S::HZ), N), NT, sm, s>>>(a, (const double*)A, (const double2*)R,
                                                                   (const double2*)tw, (double2*)W);
    return cudaGetLastError();
}

template <int N>
cudaError_t run_half_y(cudaStream_t s, double kf, const void* tw, void* W)
{
    using S = Shape<N>;
    const size_t sm = (size_t)(S::TWS + S::HX * S::template line_stride<16, S::HX>()) * 16;
    cudaError_t e = set_smem(k_half_y<N>, sm);
    if (e != cudaSuccess) return e;
    k_half_y<N><<<dim3(kHalfY * (N / 2 / S::HX), N), S::HX * S::T, sm, s>>>(kf, (const double2*)tw, (double2*)W);
    return cudaGetLastError();
}

template <typename V, int N>
cudaError_t run_y(cudaStream_t s, int grids, const void* tw, void* W)
{
    using S = Shape<N>;
    constexpr int TS = S::template line_stride<sizeof(V), S::TX>();
    const size_t sm = (size_t)(S::TWS + S::TX * TS) * sizeof(V);
    cudaError_t e = set_smem(k_fields_y<V, N>, sm);
    if (e != cudaSuccess) return e;
    k_fields_y<V, N><<<dim3(N / S::TX, N, grids), S::THREADS, sm, s>>>((const V*)tw, (V*)W);
    return cudaGetLastError();
}

template <typename V, typename Gt, int N>
cudaError_t run_x(cudaStream_t s, const FieldArgs& a, const void* tw, const void* W, void* G)
{
    using S = Shape<N>;
    const size_t sm = S::template x_smem<V>();
    cudaError_t e = set_smem(k_fields_x<V, Gt, N>, sm);
    if (e != cudaSuccess) return e;
    k_fields_x<V, Gt, N><<<(unsigned)((size_t)N * N / S::XL), S::THREADS_X, sm, s>>>(a.kf, a.slot7, (const V*)tw,
                                                                                      (const V*)W, (Gt*)G);
    return cudaGetLastError();
}

template <typename V, typename Gt, int N>
cudaError_t run_x_planar(cudaStream_t s, const FieldArgs& a, const void* tw, const void* W, double* out)
{
    using S = Shape<N>;
    constexpr int LPB = S::THREADS / S::T;
    const size_t sm = (size_t)(S::TWS + LPB * S::TSX) * sizeof(V);
    cudaError_t e = set_smem(k_fields_x_planar<V, Gt, N>, sm);
    if (e != cudaSuccess) return e;
    k_fields_x_planar<V, Gt, N><<<dim3((unsigned)((size_t)N * N / LPB), 5), S::THREADS, sm, s>>>(
        a.kf, (const V*)tw, (const V*)W, out);
    return cudaGetLastError();
}

#define FDF_DISPATCH_N(N, CALL)                     \
    switch (N) {                                    \
        case 8: return CALL(8);                     \
        case 16: return CALL(16);                   \
        case 32: return CALL(32);                   \
        case 64: return CALL(64);                   \
        case 128: return CALL(128);                 \
        case 256: return CALL(256);                 \
        case 512: return CALL(512);                 \
        default: return cudaErrorInvalidValue;      \
    }

}  // namespace

// ---- super-steps: G = (1 - w) A + w B, element by element -------------------
__global__ void __launch_bounds__(256) k_interp_f32(size_t n4, const float4* __restrict__ A,
                                                    const float4* __restrict__ B, float w, float4* __restrict__ G)
{
    const float u = 1.f - w;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
        const float4 a = __ldcs(A + i), b = __ldcs(B + i);
        G[i] = make_float4(u * a.x + w * b.x, u * a.y + w * b.y, u * a.z + w * b.z, u * a.w + w * b.w);
    }
}

__global__ void __launch_bounds__(256) k_interp_f64(size_t n2, const double2* __restrict__ A,
                                                    const double2* __restrict__ B, double w,
                                                    double2* __restrict__ G)
{
    const double u = 1.0 - w;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n2; i += (size_t)gridDim.x * blockDim.x) {
        const double2 a = A[i], b = B[i];
        G[i] = make_double2(u * a.x + w * b.x, u * a.y + w * b.y);
    }
}

// BF16 cells (8 values, 16 bytes): interpolated in FP32, rounded to nearest
__global__ void __launch_bounds__(256) k_interp_bf16(size_t n, const uint4* __restrict__ A,
                                                     const uint4* __restrict__ B, float w, uint4* __restrict__ G)
{
    const float u = 1.f - w;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const uint4 a = A[i], b = B[i];
        const uint32_t ai[4] = {a.x, a.y, a.z, a.w}, bi[4] = {b.x, b.y, b.z, b.w};
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float lo = u * __uint_as_float(ai[k] << 16) + w * __uint_as_float(bi[k] << 16);
            const float hi = u * __uint_as_float(ai[k] & 0xFFFF0000u) + w * __uint_as_float(bi[k] & 0xFFFF0000u);
            const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
            o[k] = *reinterpret_cast<const uint32_t*>(&h);
        }
        G[i] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

int mode_table_size(int N) { return 3 * (N / 2 - 1) * (N / 2 - 1) + 1; }

cudaError_t launch_interp_grid(cudaStream_t s, int precision, int N, const void* A, const void* B, double w,
                               void* G)
{
    const size_t N3 = (size_t)N * N * N;
    const size_t items = precision == FDF_PREC_F64 ? 4 * N3 : (precision == FDF_PREC_F32 ? 2 * N3 : N3);
    size_t blocks = (items + 255) / 256;
    if (blocks > 152 * 32) blocks = 152 * 32;
    if (precision == FDF_PREC_F64)
        k_interp_f64<<<(unsigned)blocks, 256, 0, s>>>(items, (const double2*)A, (const double2*)B, w, (double2*)G);
    else if (precision == FDF_PREC_F32)
        k_interp_f32<<<(unsigned)blocks, 256, 0, s>>>(items, (const float4*)A, (const float4*)B, (float)w,
                                                       (float4*)G);
    else
        k_interp_bf16<<<(unsigned)blocks, 256, 0, s>>>(items, (const uint4*)A, (const uint4*)B, (float)w, (uint4*)G);
    return cudaGetLastError();
}

cudaError_t launch_mode_keys(cudaStream_t s, const FieldArgs& a, ModeKey* keys)
{
    const int M = mode_table_size(a.N);
    k_mode_keys<<<(unsigned)((M + 255) / 256), 256, 0, s>>>(a, M, keys);
    return cudaGetLastError();
}

cudaError_t launch_mode_tables(cudaStream_t s, int precision, const FieldArgs& a, const ModeSteps& st, const ModeKey* keys,
                               const double* tabs64, void* A)
{
    if (st.count < 1 || st.count > kMaxSub) return cudaErrorInvalidValue;
    const int M = mode_table_size(a.N);
    const dim3 g((unsigned)((M + 255) / 256), (unsigned)st.count);
    if (precision == FDF_PREC_F64) k_mode_tables<double><<<g, 256, 0, s>>>(st, M, a.nk, a.na, keys, tabs64, (double*)A);
    else k_mode_tables<float><<<g, 256, 0, s>>>(st, M, a.nk, a.na, keys, tabs64, (float*)A);
    return cudaGetLastError();
}

cudaError_t launch_modes_once(cudaStream_t s, int precision, const FieldArgs& a, const double* tabs64, void* A, void* R)
{
    const int M = mode_table_size(a.N);
    const size_t N3 = (size_t)a.N * a.N * a.N;
    const unsigned nb = (unsigned)((M + 255) / 256 + ((N3 + 255) / 256 < 152 * 32 ? (N3 + 255) / 256 : 152 * 32));
    if (precision == FDF_PREC_F64) k_modes_once<double2><<<nb, 256, 0, s>>>(a, M, tabs64, (double*)A, (double2*)R);
    else k_modes_once<float2><<<nb, 256, 0, s>>>(a, M, tabs64, (float*)A, (float2*)R);
    return cudaGetLastError();
}

cudaError_t launch_noise(cudaStream_t s, int precision, const FieldArgs& a, void* R)
{
    const size_t N3 = (size_t)a.N * a.N * a.N;
    const unsigned blocks = (unsigned)((N3 + 255) / 256 < 152 * 32 ? (N3 + 255) / 256 : 152 * 32);
    if (precision == FDF_PREC_F64) k_noise<double2><<<blocks, 256, 0, s>>>(a, (double2*)R);
    else k_noise<float2><<<blocks, 256, 0, s>>>(a, (float2*)R);
    return cudaGetLastError();
}

cudaError_t launch_fields_z(cudaStream_t s, int precision, const FieldArgs& a, const void* A, const void* R,
                            const void* tw, void* W)
{
#define Z64(n) run_half_z<n>(s, a, A, R, tw, W)
#define Z32(n) run_z<float2, n>(s, a, A, R, tw, W)
    if (precision == FDF_PREC_F64) FDF_DISPATCH_N(a.N, Z64)
    FDF_DISPATCH_N(a.N, Z32)
#undef Z64
#undef Z32
}

cudaError_t launch_fields_y(cudaStream_t s, int precision, const FieldArgs& a, const void* tw, void* W)
{
#define Y64(n) run_half_y<n>(s, a.kf, tw, W)
#define Y32(n) run_y<float2, n>(s, a.grids, tw, W)
    if (precision == FDF_PREC_F64) FDF_DISPATCH_N(a.N, Y64)
    FDF_DISPATCH_N(a.N, Y32)
#undef Y64
#undef Y32
}

cudaError_t launch_fields_x(cudaStream_t s, int precision, const FieldArgs& a, const void* tw, const void* W, void* G)
{
#define X64(n) run_x<double2, double, n>(s, a, tw, W, G)
#define X32(n) run_x<float2, float, n>(s, a, tw, W, G)
#define X16(n) run_x<float2, __nv_bfloat16, n>(s, a, tw, W, G)
    if (precision == FDF_PREC_F64) FDF_DISPATCH_N(a.N, X64)
    if (precision == FDF_PREC_F32) FDF_DISPATCH_N(a.N, X32)
    FDF_DISPATCH_N(a.N, X16)
#undef X64
#undef X32
#undef X16
}

cudaError_t launch_fields_x_planar(cudaStream_t s, int precision, const FieldArgs& a, const void* tw, const void* W,
                                   double* out)
{
#define P64(n) run_x_planar<double2, double, n>(s, a, tw, W, out)
#define P32(n) run_x_planar<float2, float, n>(s, a, tw, W, out)
#define P16(n) run_x_planar<float2, __nv_bfloat16, n>(s, a, tw, W, out)
    if (precision == FDF_PREC_F64) FDF_DISPATCH_N(a.N, P64)
    if (precision == FDF_PREC_F32) FDF_DISPATCH_N(a.N, P32)
    FDF_DISPATCH_N(a.N, P16)
#undef P64
#undef P32
#undef P16
}

cudaError_t launch_fields_from_f64(cudaStream_t s, int precision, int N, const double* in, void* G)
{
    const size_t N3 = (size_t)N * N * N;
    const unsigned blocks = (unsigned)((N3 + 255) / 256 < 152 * 32 ? (N3 + 255) / 256 : 152 * 32);
    if (precision == FDF_PREC_F64) k_fields_from_f64<double><<<blocks, 256, 0, s>>>(N3, in, (double*)G);
    else if (precision == FDF_PREC_F32) k_fields_from_f64<float><<<blocks, 256, 0, s>>>(N3, in, (float*)G);
    else k_fields_from_f64<__nv_bfloat16><<<blocks, 256, 0, s>>>(N3, in, (__nv_bfloat16*)G);
    return cudaGetLastError();
}

}  // namespace fdf
