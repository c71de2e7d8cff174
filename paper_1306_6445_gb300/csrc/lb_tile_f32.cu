// The direct step kernel with float storage (lb_tile.cuh).
#include "lb_tile.cuh"

namespace lbm {

cudaError_t tile_f32(const Consts &c, const Geom &g, int variant, int order,
                     const StepBuffers &b, int *err, cudaStream_t st) {
    return tile_dispatch<float>(c, g, variant, order, b, err, st);
}

}  // namespace lbm
