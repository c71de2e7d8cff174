// The direct step kernel with BF16 storage (lb_tile.cuh).
#include "lb_tile.cuh"

namespace lbm {

cudaError_t tile_bf16(const Consts &c, const Geom &g, int variant, int order,
                     const StepBuffers &b, int *err, cudaStream_t st) {
    return tile_dispatch<__nv_bfloat16>(c, g, variant, order, b, err, st);
}

}  // namespace lbm
