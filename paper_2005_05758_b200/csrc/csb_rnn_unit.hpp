// Resident time loop for small products (layout): every warp owns whole hidden units.
//
// Where a CTA has only a few thousand weights a step is a chain of latencies, not of traffic, and what
// counts is how few dependent steps and barriers lie between the arrival of h_{t-1} and the
// publication of h_t.  So a warp holds all rows of its units: `1 << lu` units at a time, a row on 32 >> lu
// lanes divided by the number of rows, and each lane a list of (column, weight) pairs of its row.  Pairs
// are multiplied straight with the staged vector in shared memory, a row's lanes meet in a few
// shuffles, the gates follow in the same warp: no partial sums in memory, one barrier per product.
// The GRU's candidate counts as two rows, one with the weights of the input part and one with those of
// the recurrent part.  The order of a row's pairs is free; it is chosen so that the lanes of a warp
// meet different shared-memory banks as far as a greedy choice finds it.
#pragma once

#include "csb_rnn1.hpp"

namespace csb {

// Rows (lane groups) of a unit in a product.
constexpr int ru_rows(int cell, int op) { return op == 1 ? 1 : cell == kR1Ligru || cell == kR1GruRb ? 2 : 4; }

// A warp's lists of one product, offsets from the image's start: [round][lane] 16 bytes, the input part's rounds
// followed by the recurrent part's.  fp16 values: four pairs (column u16, weight), fp32: two (column u32, weight).
struct RuWarp { uint32_t off; uint16_t n[2]; };
struct RuCta {
    uint32_t off16, bytes; int32_t layer;
    uint16_t units[2], lu[2]; uint32_t unit0[2];   // per product; a warp takes 1 << lu units
    uint32_t pad;
};
static_assert(sizeof(RuCta) == 32, "two 16-byte words");
// An image starts with RuWarp[2][kR1Warps].

struct RuHostPlan {
    std::vector<uint8_t> bytes;
    std::vector<RuCta> ctas;
    size_t max_bytes = 0;
    int layer_ctas[kMaxLayers] = {};
};
// Returns CSB_OK, or 1 when the layout does not apply (more units than the warps hold in one go).
int plan_unit_host(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, int n_ctas,
                   RuHostPlan* out);

}  // namespace csb
