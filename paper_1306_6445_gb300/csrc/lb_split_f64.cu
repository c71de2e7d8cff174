// The FP64 step in two passes (psi, collision; lb_tile.cuh).
#include "lb_tile.cuh"

namespace lbm {

cudaError_t split_f64(const Consts &c, const Geom &g, const StepBuffers &b, int *err, cudaStream_t st) {
    switch (c.eos_kind) {
        case LB_EOS_CS: return split_bc<double, LB_EOS_CS>(c, g, b, err, st);
        case LB_EOS_EXP: return split_bc<double, LB_EOS_EXP>(c, g, b, err, st);
        default: return split_bc<double, LB_EOS_PIECEWISE>(c, g, b, err, st);
    }
}

}  // namespace lbm
