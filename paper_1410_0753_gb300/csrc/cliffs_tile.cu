// The tile kernels (tile_kernels.cuh) with reflecting outer edges, and the launchers of all of
// them. The OPEN instantiations and those of the alternating order are in translation units
// of their own, so that they compile in parallel.
#include <algorithm>

#include "tile_kernels.cuh"

namespace cliffs {

// index: spherical +1, friction +2, eq. (solver1) +4; k_step_tile: y first +8
#define CLIFFS_V2T(K, ...) (const void*)K<false, false, __VA_ARGS__>, (const void*)K<true, false, __VA_ARGS__>, \
                           (const void*)K<false, true, __VA_ARGS__>, (const void*)K<true, true, __VA_ARGS__>
const void* tile_kernel_open(int v);       // cliffs_tile_open.cu
const void* batch_tile_kernel_open(int v);
const void* batch_tile_kernel_alt(int v);       // cliffs_tile_alt.cu; open edges +8

static const void* tile_kernel(const StepArgs& a) {
    static const void* const t[16] = {CLIFFS_V2T(k_step_tile, false, false, false), CLIFFS_V2T(k_step_tile, false, true, false),
                                      CLIFFS_V2T(k_step_tile, true, false, false), CLIFFS_V2T(k_step_tile, true, true, false)};
    const int v = (a.sph ? 1 : 0) + (a.K.fric ? 2 : 0) + (a.K.inv_dt2 > 0.f ? 4 : 0) + (a.yfirst ? 8 : 0);
    return a.open_edges ? tile_kernel_open(v) : t[v];
}
static const void* batch_tile_kernel(const StepArgs& a, bool alt) {
    static const void* const t[8] = {CLIFFS_V2T(k_batch_tile, false, false, false), CLIFFS_V2T(k_batch_tile, true, false, false)};
    const int v = (a.sph ? 1 : 0) + (a.K.fric ? 2 : 0) + (a.K.inv_dt2 > 0.f ? 4 : 0);
    if (alt) return batch_tile_kernel_alt(v + (a.open_edges ? 8 : 0));
    return a.open_edges ? batch_tile_kernel_open(v) : t[v];
}

static int tile_smem(int tile_rows) { return tile_rows * (TROW_FLOATS * 4 + 1) + 15; }
// two blocks on an SM share 227 KB (1 KB of it reserved per block)
int tile_max_rows() { return (113 * 1024 - 1024 - 16) / (TROW_FLOATS * 4 + 1); }
int tile_warps_per_block() { return TILE_WARPS; }

static cudaError_t optin(const void* k) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem(tile_max_rows()));
}

int tile_blocks_per_sm(int tile_rows) {
    const void* k = (const void*)k_batch_tile<true, true, false, false, false>;
    int nb = 0;
    if (optin(k) != cudaSuccess) return 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, TILE_WARPS * 32, tile_smem(tile_rows));
    return std::max(1, nb);
}

cudaError_t launch_step_tile(const StepArgs& a, int batch, cudaStream_t s) {
    const void* k = tile_kernel(a);
    const cudaError_t e = optin(k);
    if (e != cudaSuccess) return e;
    StepArgs aa = a;
    void* args[] = {&aa};
    return cudaLaunchKernel(k, dim3(a.nitems, batch), dim3(TILE_WARPS * 32), args, tile_smem(a.tile_rows), s);
}

cudaError_t launch_batch_tile(const StepArgs& a, const BatchArgs& b, int blocks, cudaStream_t s) {
    const void* k = batch_tile_kernel(a, b.alternate != 0);
    const cudaError_t e = optin(k);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(TILE_WARPS * 32);
    cfg.dynamicSmemBytes = tile_smem(a.tile_rows);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;         // all blocks resident: the grid barrier
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    StepArgs aa = a;
    BatchArgs bb = b;
    void* args[] = {&aa, &bb};
    return cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace cliffs
