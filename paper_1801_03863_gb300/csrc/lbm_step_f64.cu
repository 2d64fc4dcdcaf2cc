// lbm_step_f64.cu -- fused step kernels with double storage and double arithmetic.
#include "lbm_aux.h"
#include "lbm_step.cuh"

namespace lbm {

const void* step_kernel_f64(int lattice, int collision, int V) {
    if (lattice == 1) {
        if (V == 1) return (const void*)&step_tube_kernel<double, double, 1>;
        if (V == 2) return (const void*)&step_tube_kernel<double, double, 2>;
        if (V == 4) return (const void*)&step_tube_kernel<double, double, 4>;
        return nullptr;
    }
    if (V == 1) return pick_step_flat_kernel(collision);
    if (V == 2) return pick_step_kernel<double, double, 2>(collision);
    return nullptr;
}

}  // namespace lbm
