// The batched product on tcgen05 tensor cores: layout shared by the planner (csb_umma_plan.cpp) and the
// kernel (csb_umma.cu).
//
// The matrix is cut into tiles of 128 output rows (four quadrants of 32, one per TMEM lane quarter) and
// windows of 64 columns.  A CTA takes MT tiles (a row group) over a range of windows; the S ranges of a row
// group are one thread-block cluster.  A tile-window is kept as four items, one per quadrant, each expanded by
// one warp, whose lanes are the rows, into the dense 32 x 64 operand:
//
//   header  uint4 per (row segment, column segment), row segments first:
//             x  bit l: lane l's row is kept (zero outside of the segment's rows, and where no column is kept)
//             y  where the segment's values start, bytes from the item
//             z, w  bit c: the segment's column c is kept
//   values  16 bytes per eight columns and kept row, [eight columns][row], binary16, zero where a column is not kept
//
// A row segment is the part of one block-row that lies in the quadrant, a column segment 16, 32 or 64 columns, the
// part of one block that lies in the window.  Rows are compact and columns are not: a lane then has its row of a window in
// eight 16-byte loads.  With the columns compact by pairs (1.5 instead of 2 times the compact size at 4x, 1.8 instead of
// 5 at 25x) it took a predicated load and add for every pair, and the expanding warps' instructions set the time.
//
// The tile-windows of a CTA go in rounds of four, one for each four of the sixteen expanding warps, in the order (group of
// `flush` windows, tile, window): the sums of a tile over such a group, a unit, come out of the tensor cores' accumulators
// before they grow further.  A round's items travel together, behind a table of where each warp's item starts.
// (Rounds, and not single tile-windows with a barrier each: the warp that issues the tensor instructions spent 530
// cycles on each with its waits and commits, 8192 x 8192 at batch 8 22 us.)
#pragma once

#include "csb_internal.hpp"

namespace csb {

enum { kUmmaWindow = 64, kUmmaImage = 64 * 256 /* bytes of a window of packed inputs, 64 batch columns */, kUmmaExpandWarps = 16, kUmmaMaxMT = 2, kUmmaMaxS = 8 };

struct UmmaQuad {             // 32 lanes of a tile
    int32_t row0, nrows;      // their rows of the matrix (none: nrows = 0)
    int32_t c0, c1;           // and the columns that count
    int32_t out0, pad[3];     // the first one's place in a product's output
};
static_assert(sizeof(UmmaQuad) == 32, "two 16-byte words");
// Bytes of packed inputs: the images of 64 batch columns, then 16 words per window (are there inputs that binary16 cannot hold?).
inline size_t umma_xp_bytes(int windows) { return (size_t)windows * (kUmmaImage + 64); }
struct UmmaCta {
    uint32_t off128;          // where its rounds start, 128-byte units
    int32_t table;            // its first entry in the table of rounds
    int32_t group, split;     // row group and which column range of it
    int32_t w0, nw;           // windows
    int32_t pad[2];
};
static_assert(sizeof(UmmaCta) == 32, "two 16-byte words");
struct UmmaRound { uint32_t off16, bytes; };   // a round of a CTA, from its start

struct UmmaHostPlan {
    int MT = 1, S = 1, flush = 1, n_groups = 0, windows = 0, seg_words = 32;   // seg_words: 32-bit words of a row of a column segment
    int threads = 16;                     // to plan with, at most
    std::vector<UmmaQuad> quads;          // [n_groups][MT][4]
    std::vector<UmmaCta> ctas;            // [n_groups][S]
    std::vector<UmmaRound> rounds;        // CTA after CTA
    std::vector<std::vector<uint8_t>> streams;   // per CTA
    uint32_t max_round = 0;               // bytes
    uint64_t total128 = 0;                // all streams, 128-byte units
};

// 32-bit words of a row of a column segment for blocks of this width; 0: the layout does not take them.
inline int umma_seg_words(int block_c) { return block_c == 16 ? 8 : block_c == 32 ? 16 : block_c % 64 == 0 ? 32 : 0; }
// Rows of the matrix in order, in groups of MT tiles.
std::vector<UmmaQuad> umma_row_quads(const csb_matrix* A, int MT);
// A layer of a recurrent stack: a tile is 32 hidden units, its quadrants the gates i, f, g, o or r, z and the input and the
// recurrent part of the candidate, whose sums stay apart (output rows 2H .. and 3H ..).
std::vector<UmmaQuad> umma_gate_quads(int gates, int in_size, int H, int MT);
// Tiles per CTA and column ranges per group for `tiles` tiles of `windows` windows on a device that holds clusters[S] clusters of S.
double umma_cost(int MT, int S, int windows);          // a CTA's modelled time, in tile-windows
void umma_shape(int tiles, int windows, const int* clusters, int* MT, int* S);
// Tile-window j of a round that has nj of them: which of the MT tiles, and which of the round's windows.  `len` is the
// number of windows of a unit.
struct UmmaPlace { int mt, window; };
#ifdef __CUDACC__
__host__ __device__
#endif
inline int umma_unit_len(int MT, int flush, int nj) { return MT == 2 && 2 * flush > nj ? nj >> 1 : flush; }
#ifdef __CUDACC__
__host__ __device__
#endif
inline UmmaPlace umma_place(int MT, int len, int j) {
    return MT == 1 ? UmmaPlace{0, j} : len == 2 ? UmmaPlace{j >> 1, j & 1} : UmmaPlace{j & 1, j >> 1};
}
// Windows per flush group.  The tensor cores truncate each sum, so the error follows the number of steps between two flushes.
// Two windows take 7 to 15 % less time from 4096 x 4096 on, and are taken where the error stays no larger than what
// mma.sync gave, whose chains grow with the number of blocks (they are a CTA's share of a block-row): from 6000 blocks on.
// 2-norm of the error against 64 bits, 1e-7, mma.sync / 1 / 2 windows, batch 8:
//   blocks of 64 x 64:  512 x 4096 at 4x 1.49 / 1.38 / 1.71, 4096 x 4096 at 25x 1.26 / 1.15 / 1.27, 8192 x 3072 at 25x (6144
//     blocks) 1.33 / 1.14 / 1.26, 8192 x 8192 at 4x 4.78 / 1.46 / 1.75, at 25x 1.70 / 1.20 / 1.32;
//   blocks of 32 x 32:  512 x 4096 at 9x 1.23 / 1.12 / 1.30, 2048 x 4096 at 4x (8192 blocks) 2.24 / 1.26 / 1.51;
//   of 64 x 128:  4096 x 4096 at 9x 1.70 / 1.28 / 1.87, 8192 x 8192 at 9x (8192 blocks) 2.87 / 1.36 / 1.91;
//   of 16 x 16:  512 x 2049 at 4x 1.41 / 1.14 / 1.37, 8192 x 8192 at 4x 24.8 / 1.43 / 1.54.
inline int umma_flush(int windows, int64_t blocks = 0x7fffffff) { return windows < 32 || blocks < 6000 ? 1 : 2; }
// Fills streams, rounds, ctas (the other members are set); throws std::bad_alloc.
void plan_umma_host(const csb_matrix* A, UmmaHostPlan* P);

}  // namespace csb
