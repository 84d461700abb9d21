// The tile kernels for grids with open (radiating) outer edges.
#include "tile_kernels.cuh"

namespace cliffs {

#define CLIFFS_V2TO(K, ...) (const void*)K<false, false, __VA_ARGS__>, (const void*)K<true, false, __VA_ARGS__>, \
                            (const void*)K<false, true, __VA_ARGS__>, (const void*)K<true, true, __VA_ARGS__>

const void* tile_kernel_open(int v) {
    static const void* const t[16] = {CLIFFS_V2TO(k_step_tile, false, false, true), CLIFFS_V2TO(k_step_tile, false, true, true),
                                      CLIFFS_V2TO(k_step_tile, true, false, true), CLIFFS_V2TO(k_step_tile, true, true, true)};
    return t[v];
}
const void* batch_tile_kernel_open(int v) {
    static const void* const t[8] = {CLIFFS_V2TO(k_batch_tile, false, true, false), CLIFFS_V2TO(k_batch_tile, true, true, false)};
    return t[v];
}

}  // namespace cliffs
