// The unit loop's kernels for batch tiles of 8 (a file of their own: they compile for a while).
#include "csb_rnn_unit_kernel.cuh"

namespace csb {

const void* ru_kernel_b8(int cell, int val_dtype) {
    return val_dtype == CSB_F16 ? pick_unit_kernel<__half, 8>(cell) : pick_unit_kernel<float, 8>(cell);
}

}  // namespace csb
