// Checks on the device that the library's entry points cannot make: the sources of the library's
// host side with functions beside them that see a context's grids.  Compiled and linked with
// the library's other objects by test_gpu_gather_grid.py.
#include "fdf_api.cu"

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
