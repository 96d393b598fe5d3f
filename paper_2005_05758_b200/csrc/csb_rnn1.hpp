// Batch-1 time loop: what its planner (csb_rnn1_plan.cpp) and its kernel (csb_rnn1.cu) share.
//
// A CTA owns a contiguous range of hidden units of one layer with all rows that produce them, and
// keeps their compressed weights in shared memory for the whole sequence.  The weights are laid out
// for threads, not for blocks: every thread works for ONE row, so its sum stays in a register from
// the first block-column to the last, and a row has as many threads as its weights ask for.  A
// thread's work is a list of slots: four weights of a block's kernel-matrix row (the last slot of a
// row of a block is padded with zeros) and the place of their four gathered inputs.  Slots go
// through the warp in pairs, [pair][lane], 16 bytes of fp16 weights and two 16-bit places per lane.
// The first pairs of the recurrent part (the one on the critical path) are held in registers.
#pragma once

#include "csb_internal.hpp"

namespace csb {

enum R1Cell { kR1Lstm = 0, kR1Gru = 1, kR1Lstmp = 2, kR1Ligru = 3, kR1GruRb = 4 };
enum { kR1Threads = 512, kR1Warps = kR1Threads / 32,
       kR1WarpUnits = 6,                       // hidden units whose gates one warp applies: four lanes each, two words of three units
       kR1MaxUnits = kR1Warps * kR1WarpUnits,
       kR1Words = 2,                           // exchange words a thread polls at most
       kR1Ring = 32, kR1Block = 8 };           // steps a published vector stays; steps between two looks at the readers' progress

// One product of a CTA: its rows' weights over an input part and a recurrent part (either may be empty).
struct R1Op {
    uint32_t rows_off;                         // u32 per row: first thread | threads << 16
    uint32_t warp_off;                         // uint4 per warp: weights (16-byte units), places (bytes), pairs in, pairs rec
    uint32_t gather_off[2];                    // u16 per gathered input: index into the staged vector (its length = a zero)
    uint16_t quads[2];                         // gathered inputs / 4, input and recurrent part
    uint16_t n_rows, units;                    // rows = gates * units, gate-major
    uint32_t unit0;                            // first unit
    uint32_t word0;                            // first exchange word of the units this product publishes
    uint32_t reg_off;                          // [warp][pair][lane] weights of the register pairs (behind what is copied to shared memory)
    uint32_t reg_places;                       // [warp][pair][lane] u32
    uint32_t pad[2];
};
static_assert(sizeof(R1Op) == 48, "three 16-byte words");
struct R1Header { R1Op op[2]; };               // start of a CTA's image; offsets are from the image's start
struct R1Cta { uint32_t off16, bytes, smem_bytes; int32_t layer; };   // the first smem_bytes of the image go to shared memory

struct R1HostPlan {
    std::vector<uint8_t> bytes;                // the CTAs' images, each aligned to 128 bytes
    std::vector<R1Cta> ctas;
    std::vector<uint32_t> wmap[2][kMaxLayers]; // per exchange (0: state, 1: within the step) and layer: unit0 | units << 16 of every word
    size_t max_smem = 0, max_xg[2][2] = {{0, 0}, {0, 0}};   // largest shared-memory part of an image; gathered floats per product and part
    int layer_ctas[kMaxLayers] = {};
    double balance = 1.0;
};
inline int r1_gates(int cell, int op) {
    return cell == kR1Lstm || (cell == kR1Lstmp && op == 0) ? 4 : cell == kR1Gru ? 3 : cell == kR1Ligru || (cell == kR1GruRb && op == 0) ? 2 : 1;
}
constexpr int r1_ops(int cell) { return cell == kR1Lstmp || cell == kR1GruRb ? 2 : 1; }
// Pairs of a product's recurrent part in registers: 16 weight registers, as far as 128 per thread go.
constexpr int r1_reg_pairs(int cell, int val_bytes) { return (val_bytes == 2 ? 4 : 2) / r1_ops(cell); }
// W: per layer the gate matrix; Wp: LSTMP's projections.  in_size[l] + S columns (S the width of the
// recurrent state).  Returns CSB_OK, or 1 when the layout does not apply.
int plan_rnn1_host(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int n_ctas,
                   R1HostPlan* out);
// One call of the time loop at batch 1.  Returns 1 when the kernel does not take these matrices (nothing was done).
int rnn1_forward(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const float* const* bias, const float* x, int64_t T,
                 int H, int S, const int* in_size, const float* h0, const float* c0, float* y, float* hT, float* cT, unsigned flags, void* stream);
void drop_rnn1_plans(const csb_matrix* A);
void barrier_test_hook(unsigned int* extra, unsigned long long* ns);   // csb_rnn.cu

}  // namespace csb
