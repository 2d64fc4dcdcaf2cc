// lbm_step_f32.cu -- fused step kernels with float storage and float arithmetic.
#include "lbm_aux.h"
#include "lbm_step.cuh"
#include "lbm_step_block.cuh"
#include "lbm_step_smem.cuh"

namespace lbm {

const void* step_kernel_f32(int lattice, int collision, int V) {
    if (lattice == 1) {
        if (V == 2) return (const void*)&step_tube_kernel<float, float, 2>;
        if (V == 4) return (const void*)&step_tube_kernel<float, float, 4>;
        if (V == 8) return (const void*)&step_tube_kernel<float, float, 8>;
        return nullptr;
    }
    if (V == 2) return pick_step_kernel<float, float, 2>(collision);
    if (V == 4) return pick_step_kernel<float, float, 4>(collision);
    return nullptr;
}

const void* step_kernel_single_tube_f32() { return pick_step_single_tube_kernel<float, 4>(); }

const void* step_kernel_block_f32(int collision, int rows) {
    return pick_step_block_kernel<float>(collision, rows);
}

const void* step_kernel_smem_f32(int collision, int variant, bool draws, size_t* smem_bytes) {
    if (variant == 2) return pick_step_kernel_smem<float, 2>(collision, draws, smem_bytes);
    if (variant == 3) return pick_step_kernel_smem<float, 3>(collision, draws, smem_bytes);
    return variant == 1 ? pick_step_kernel_smem<float, 1>(collision, draws, smem_bytes)
                        : pick_step_kernel_smem<float, 0>(collision, draws, smem_bytes);
}

}  // namespace lbm
