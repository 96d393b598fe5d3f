// The resident time loop's kernels for batch tiles of 8 (a file of their own: they compile for a while).
#include "csb_rnn1_kernel.cuh"

namespace csb {

const void* r1_kernel_b8(int cell, int val_dtype) {
    return val_dtype == CSB_F16 ? pick_kernel<__half, 8>(cell) : nullptr;   // fp32 values: tiles of 4
}

}  // namespace csb
