// What the resident time loop's kernel is launched with.
#pragma once

#include <cuda_runtime.h>

#include "csb_rnn1.hpp"
#include "csb_rnn_unit.hpp"

namespace csb {

struct R1Common {
    const uint8_t* images;
    const float* x; const float* h0; const float* c0;
    float* y; float* hT; float* cT;
    const float* bias[kMaxLayers];
    int in_size[kMaxLayers];
    uint32_t* epoch;                           // per CTA: step numbers used so far
    uint32_t* progress;                        // per layer: blocks of kR1Block input steps read, summed over its CTAs, never cleared
    int layer_ctas[kMaxLayers];
    uint32_t* status;
    unsigned long long limit_ns;
    uint32_t never;                            // test hook: wait for step numbers that never come
    int T, B, H, S, L;
#ifdef CSB_PHASE_CLOCKS
    long long* clocks;                         // [CTA][8] cycles of thread 0 summed over the steps
#endif
};
struct R1Args : R1Common {
    const R1Cta* ctas;
    const uint32_t* wmap[2][kMaxLayers];       // first element | elements << 24 of every exchange word
    int words[2][kMaxLayers];
    uint4* ex[2][kMaxLayers];                  // [kR1Ring][words]
    uint32_t vu[2], vr, vm, part[2], z[2], cs, bias0, bias1, misc;   // shared-memory offsets behind the image
};
struct RuArgs : R1Common {
    const RuCta* ctas;
    uint2* ex[2][kMaxLayers];                  // [kR1Ring][elements]: the state; what the first of two products gives
    uint32_t vu[2], vr[2], vm, misc;           // shared-memory offsets behind the image
};

// The kernels by cell (R1Cell) and value type, per batch tile.
const void* r1_kernel_b1(int cell, int val_dtype);
const void* r1_kernel_b4(int cell, int val_dtype);
const void* r1_kernel_b8(int cell, int val_dtype);
const void* ru_kernel_b1(int cell, int val_dtype);
const void* ru_kernel_b4(int cell, int val_dtype);
const void* ru_kernel_b8(int cell, int val_dtype);

}  // namespace csb
