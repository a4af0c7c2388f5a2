// fields_noalloc.cu -- fdf_build_fields_noalloc: the field build of
// fdf_build_fields without a context and without any device allocation.
//
// Some callers cannot allocate device memory: a simulation code that embeds
// this library and whose own allocator owns the whole device budget, or a
// serving loop that forbids cudaMalloc/cudaFree after start-up because those
// calls synchronise the device and fragment its memory.  This entry point
// serves them.  Its work arrays live in one file-scope device array of
// FDF_NOALLOC_SCRATCH_BYTES that every GPU loading the library holds until the
// process exits; the caller passes the inputs (host tables) and the output
// (device memory).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "device_math.cuh"

namespace fdf {
namespace {

// The shared scratch.  Host code must not pass g_scratch itself to a kernel:
// in host code the name is a host-side stand-in, not a device address.  Its
// device address comes from cudaGetSymbolAddress, once per device.
static __device__ __align__(256) unsigned char g_scratch[FDF_NOALLOC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
void* g_scratch_addr[kMaxDevices] = {};
std::mutex g_scratch_mu;

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// Device address of g_scratch on the current device; looked up on the first
// call made with that device current.
int scratch_address(unsigned char** out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_error(FDF_ECUDA, (std::string("cudaGetDevice: ") + cudaGetErrorString(e)).c_str());
    if (dev < 0 || dev >= kMaxDevices) return set_error(FDF_ENOSYS, "device index beyond 63");
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess || !p)
            return set_error(FDF_ECUDA, (std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e)).c_str());
        g_scratch_addr[dev] = p;
    }
    *out = (unsigned char*)g_scratch_addr[dev];
    return FDF_OK;
}

}  // namespace
}  // namespace fdf

using namespace fdf;

extern "C" int fdf_build_fields_noalloc(const fdf_params* p, const fdf_tables* t, double lna, double* out,
                                        void* stream)
{
    int rc = validate_params(p);
    if (rc) return rc;
    if (!t || !t->lnk || !t->lna || !t->T_psi || !t->T_phi || !t->dTphi_dlna || !out || !std::isfinite(lna))
        return set_error(FDF_EINVAL, "bad arguments");
    if (t->nk < 2 || t->na < 2 || t->nk > 1024 || t->na > 256)
        return set_error(FDF_EINVAL, "table sizes out of range (nk 2..1024, na 2..256)");
    double lnk0, dlnk, lnat0, dlnat;
    if (!uniform_grid(t->lnk, t->nk, &lnk0, &dlnk) || !uniform_grid(t->lna, t->na, &lnat0, &dlnat))
        return set_error(FDF_EINVAL, "lnk and lna must be uniform ascending grids");
    const int gp = grid_prec(p->precision);
    const bool f64 = gp == FDF_PREC_F64;
    const size_t N = (size_t)p->n_grid, N3 = N * N * N;
    const size_t csz = f64 ? 16 : 8, rsz = f64 ? 8 : 4;
    // scratch layout: W (five packed grids) | FP64 table rows and twiddles | amplitude table | noise
    const size_t M = (size_t)mode_table_size(p->n_grid), nk = (size_t)t->nk;
    const size_t oT64 = align256(5 * N3 * csz), oTw = oT64 + 6 * nk * 8;
    const size_t oA = align256(oTw + N * csz), oR = oA + align256(4 * M * rsz);
    // the limit counts two work arrays of four grids and the tables in full
    const size_t need = 2 * align256(4 * N3 * csz) + align256(3 * (size_t)t->na * nk * 8) + align256(4 * M * rsz) +
                        align256(N * csz) + align256(N3 * csz);
    if (need > FDF_NOALLOC_SCRATCH_BYTES) {
        char msg[200];
        snprintf(msg, sizeof msg,
                 "fdf_build_fields_noalloc: n_grid %d at this precision needs %zu bytes of scratch; the static "
                 "scratch holds %zu (FDF_NOALLOC_SCRATCH_BYTES)",
                 p->n_grid, need, (size_t)FDF_NOALLOC_SCRATCH_BYTES);
        return set_error(FDF_EINVAL, msg);
    }
    unsigned char* s = nullptr;
    rc = scratch_address(&s);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    // what the build reads of the host's tables, in one copy: the two rows around ln a of each
    // of the three tables, and the twiddles fdf_create uploads.  The copy is from pageable
    // host memory, so the stream is synchronised before the vector goes.
    FieldArgs a = make_field_args(*p, t->nk, t->na, lnk0, dlnk, lnat0, dlnat, lna);
    std::vector<double> up(6 * nk + 2 * N), twd(2 * N);
    const double* tables[3] = {t->T_psi, t->T_phi, t->dTphi_dlna};
    for (int k = 0; k < 3; ++k) std::memcpy(up.data() + 2 * k * nk, tables[k] + (size_t)a.ia * nk, 2 * nk * 8);
    twiddle_table((int)N, twd.data());
    if (f64) std::copy(twd.begin(), twd.end(), up.begin() + 6 * nk);
    else {
        const std::vector<float> twf(twd.begin(), twd.end());
        std::memcpy(up.data() + 6 * nk, twf.data(), twf.size() * 4);
    }
    cudaError_t e = cudaMemcpyAsync(s + oT64, up.data(), 6 * nk * 8 + N * csz, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return set_error(FDF_ECUDA, (std::string("table upload: ") + cudaGetErrorString(e)).c_str());
    a.ia = 0;
    a.na = 2;
    a.slot7 = kSlot7Zero;
    a.grids = 5;
    // as fdf_build_fields: slots 0-6 with phi_dot transformed alone, slot 7 (psi) from the
    // fifth packed grid
    e = launch_modes_once(st, gp, a, (const double*)(s + oT64), s + oA, s + oR);
    if (e == cudaSuccess) e = launch_fields_z(st, gp, a, s + oA, s + oR, s + oTw, s);
    if (e == cudaSuccess) e = launch_fields_y(st, gp, a, s + oTw, s);
    if (e == cudaSuccess) e = launch_fields_x_planar(st, gp, a, s + oTw, s, out);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess)
        return set_error(FDF_ECUDA, (std::string("fdf_build_fields_noalloc: ") + cudaGetErrorString(e)).c_str());
    return FDF_OK;
}
