// Resident time loop (small batches): what its planner (csb_rnn1_plan.cpp) and its kernel (csb_rnn1.cu) share.
//
// A CTA owns a contiguous range of hidden units of one layer with all rows that produce them, and
// keeps their compressed weights in shared memory for the whole sequence.  The work of a product is
// cut into tasks, one per lane: a chunk of up to 8 kept columns of one block (4 in narrow tasks) times
// some of the block's kept rows.  A lane fetches the chunk's inputs once, straight from the staged
// vector through the column indices, and then takes the rows one after the other: 16 bytes of
// weights, eight products, one partial sum, stored to a place of its own.  So an input is read once per
// block instead of once per weight, nothing is gathered first, and nothing is scattered with a read
// behind it.  The partial sums of a row lie side by side and are added up when both parts are done.
// 32 tasks of about the same number of rows form a group, which a warp works through in lock-step.
// Columns are ordered inside a chunk, and partial sums inside a row, so that the lanes of a group meet
// different shared-memory banks as far as a greedy choice finds it.
#pragma once

#include "csb_internal.hpp"

namespace csb {

enum R1Cell { kR1Lstm = 0, kR1Gru = 1, kR1Lstmp = 2, kR1Ligru = 3, kR1GruRb = 4 };
enum { kR1Threads = 512, kR1Warps = kR1Threads / 32,
       kR1WarpUnits = 6,                       // states whose gates a warp applies at a time: four lanes each, two words of three
       kR1MaxUnits = 255,
       kR1MaxRows = 16,                        // rows of a task
       kR1Ring = 32, kR1Block = 8 };           // steps a published vector stays; steps between two looks at the readers' progress

// Columns of a wide task for a batch tile: its inputs stay in registers.
constexpr int r1_wide(int bt) { return bt >= 8 ? 4 : 8; }

// One group: 32 tasks.  Offsets are from the image's start.
struct R1Group {
    uint32_t cols_off;                         // [lane] u16 x width: indices into the staged vector (its length = a zero)
    uint32_t w_off;                            // [row][lane] width values
    uint32_t pos_off;                          // [row pair][lane] two u16: where the partial sums go
    uint16_t rows, narrow;                     // rows of the longest task; 1: half as many columns
};
static_assert(sizeof(R1Group) == 16, "one 16-byte word");
struct R1Row { uint16_t base[2]; uint16_t quads[2]; };   // a row's partial sums of the input and the recurrent part: start / 4, number / 4

// One product of a CTA: its rows' weights over an input part and a recurrent part (either may be empty).
struct R1Op {
    uint32_t rows_off;                         // R1Row per row, rows = gates * units, gate-major
    uint32_t groups_off;                       // R1Group per group: warp by warp, input part before recurrent part
    uint32_t warp_off;                         // u16[4] per warp: first group, groups of the input part, of the recurrent part, 0
    uint32_t partials;                         // partial sums (floats per batch column), places for idle lanes included
    uint16_t n_rows, units;
    uint32_t unit0;                            // first unit
    uint32_t word0;                            // first exchange word of the states this product publishes
    uint32_t pad;
};
static_assert(sizeof(R1Op) == 32, "two 16-byte words");
struct R1Header { R1Op op[2]; };               // start of a CTA's image
struct R1Cta { uint32_t off16, bytes; int32_t layer; uint32_t pad; };

struct R1HostPlan {
    std::vector<uint8_t> bytes;                // the CTAs' images, each aligned to 128 bytes
    std::vector<R1Cta> ctas;
    std::vector<uint32_t> wmap[2][kMaxLayers]; // per exchange (0: state, 1: within the step) and layer: first element | elements << 24 of every word
    size_t max_bytes = 0, max_partials[2] = {0, 0}, max_units = 0;   // largest over the CTAs
    int layer_ctas[kMaxLayers] = {};
};
inline int r1_gates(int cell, int op) {
    return cell == kR1Lstm || (cell == kR1Lstmp && op == 0) ? 4 : cell == kR1Gru ? 3 : cell == kR1Ligru || (cell == kR1GruRb && op == 0) ? 2 : 1;
}
inline int r1_ops(int cell) { return cell == kR1Lstmp || cell == kR1GruRb ? 2 : 1; }
// The kernel's shared memory behind a CTA's image: offsets in bytes, and all of it.
struct R1Carve {
    uint32_t vu[2], vr, vm, part[2], z[2], cs, bias0, bias1, misc;
    size_t total;
    R1Carve(const R1HostPlan& P, int cell, int max_in, int H, int S, int BT);
};
// W: per layer the gate matrix; Wp: LSTMP's projections.  in_size[l] + S columns (S the width of the
// recurrent state); B batch columns, BT of them in shared memory side by side.  Returns CSB_OK, or 1
// when the layout does not apply or a CTA needs more than smem_limit bytes of shared memory.
int plan_rnn1_host(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, int n_ctas,
                   size_t smem_limit, R1HostPlan* out);
// One call of the time loop.  Returns 1 when the kernel does not take these matrices or this batch (nothing was done).
int rnn1_forward(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const float* const* bias, const float* x, int64_t T, int B,
                 int H, int S, const int* in_size, const float* h0, const float* c0, float* y, float* hT, float* cT, unsigned flags, void* stream);
void drop_rnn1_plans(const csb_matrix* A);
void barrier_test_hook(unsigned int* extra, unsigned long long* ns);   // csb_rnn.cu

}  // namespace csb
