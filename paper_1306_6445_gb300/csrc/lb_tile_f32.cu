// The direct step kernel with float storage (lb_tile.cuh).
#include "lb_tile.cuh"

namespace lbm {

cudaError_t tile_f32(const Consts &c, const Geom &g, int order, const void *gin, void *gout,
                      int *err, cudaStream_t st) {
    return tile_dispatch<float>(c, g, order, gin, gout, err, st);
}

}  // namespace lbm
