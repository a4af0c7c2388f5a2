// Checks on the device that the library's entry points cannot make: the sources of the library's
// host side with functions beside them that see a context's grids and the passes it launches.
// Compiled and linked with the library's other objects by device_checks.py.
#include "device_math.cuh"

namespace fdf {

// A pass as it is launched, or (fdf_check_kick_fp64) with its kick's integrals in FP64;
// g_fast counts the passes that came with them on the FP32 pipe, by KickFast.
static int g_kick_fp64 = 0, g_fast[3] = {};
static cudaError_t checked_push(cudaStream_t s, int precision, const ParticleState& st, const PushArgs& a)
{
    if (form_of(precision) != kWide) return launch_push(s, precision, st, a);
    ++g_fast[a.kick_fast];
    if (!g_kick_fp64) return launch_push(s, precision, st, a);
    PushArgs b = a;
    b.kick_fast = kKickFp64;
    return launch_push(s, precision, st, b);
}

}  // namespace fdf

#define launch_push checked_push
#include "fdf_api.cu"
#undef launch_push

extern "C" FDF_API void fdf_check_kick_fp64(int32_t on, int32_t* fast)
{
    g_kick_fp64 = on;
    std::copy(g_fast, g_fast + 3, fast);
    std::fill(g_fast, g_fast + 3, 0);
}

// The gather grid of step k, as it lies in memory, into out (device, `bytes` long).
extern "C" FDF_API int fdf_check_grid(fdf_ctx* c, int32_t k, void* out, size_t bytes)
{
    const size_t N3 = (size_t)c->p.n_grid * c->p.n_grid * c->p.n_grid;
    if (bytes != N3 * grid_bytes_per_cell(c->p.precision)) return fail(FDF_EINVAL, "wrong size");
    FDF_CUDA(cudaStreamSynchronize(c->sf), "fdf_check_grid");
    FDF_CUDA(cudaStreamSynchronize(c->stream), "fdf_check_grid");
    const int b = find_grid(c, k);
    if (b < 0) return fail(FDF_ESTATE, "no grid of that step is held");
    FDF_CUDA(cudaMemcpy(out, c->G[b], bytes, cudaMemcpyDeviceToDevice), "fdf_check_grid");
    return FDF_OK;
}

// ---- the pass's integer and FP32 forms against their FP64 formulas, on the device ------------
namespace fdf {
namespace {

// q, u: n values; d: n increments.  counts[2 f]: refused, counts[2 f + 1]: accepted with other
// bits, of f = 0 w_rsqrt53, 1 w_square53, 2 w_mul53, 3 w_add, 4 w_sqrt53, 5 w_div53.
__global__ void k_check_bits(int64_t n, const double* __restrict__ u, const double* __restrict__ q,
                             const float* __restrict__ d, unsigned long long* __restrict__ counts)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        auto count = [&](int f, bool ok, double got, double want) {
            if (!ok) atomicAdd(counts + 2 * f, 1ull);
            else if (__double_as_longlong(got) != __double_as_longlong(want)) atomicAdd(counts + 2 * f + 1, 1ull);
        };
        const double v = u[i], y = q[i];
        const float yf = rsqrtf(d2f_bits(v));
        double r, x;
        int64_t R;
        int k;
        const bool ok = w_rsqrt53(v, yf, r, R, k);
        const double want = rsqrt_fp64(v);
        count(0, ok, r, want);
        if (ok) {
            count(1, true, w_square53(R, k), __dmul_rn(want, want));
            const bool okm = w_mul53(R, k, y, x);
            count(2, okm, x, __dmul_rn(want, y));
        }
        const bool oka = w_add(y, d[i], x);
        count(3, oka, x, __dadd_rn(y, f2d_bits(d[i])));
        double s;
        const bool oks = w_sqrt53(v, yf, s);
        count(4, oks, s, __dsqrt_rn(v));
        // the sampler's quotient: its estimate is a product with the reciprocal of the root
        const double root = __dsqrt_rn(v);
        const bool okd = w_div53(y, root, y * want, x);
        count(5, okd, x, __ddiv_rn(y, root));
    }
}

}  // namespace
}  // namespace fdf

extern "C" FDF_API int fdf_check_bits(int64_t n, const double* u, const double* q, const float* d, int64_t* counts)
{
    k_check_bits<<<152 * 4, 256>>>(n, u, q, d, (unsigned long long*)counts);
    FDF_CUDA(cudaGetLastError(), "fdf_check_bits");
    FDF_CUDA(cudaDeviceSynchronize(), "fdf_check_bits");
    return FDF_OK;
}
