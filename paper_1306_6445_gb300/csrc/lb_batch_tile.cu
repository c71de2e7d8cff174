// The direct step kernel of batches with float storage (lb_tile.cuh).
#include "lb_tile.cuh"

namespace lbm {

cudaError_t batch_tile_f32(int eos, const BatchGroup &group, int n, int max_tiles, const void *maps,
                           const void *lats, int phase, int *errs, cudaStream_t st) {
    return batch_tile_dispatch<float>(eos, group, n, max_tiles, maps, lats, phase, errs, st);
}

}  // namespace lbm
