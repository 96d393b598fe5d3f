// The block loop's planner turns a stack away before it emits anything.  What it turns away must be what does not fit:
// with the limit at a stack's need it plans, one byte below it refuses.  Prints a line per stack that breaks this.
#include <cstdio>

#include "../paper_2005_05758_b200/csrc/csb_rnn1.hpp"

using namespace csb;

static unsigned int state = 1;
static unsigned int draw() { return (state = state * 1664525u + 1013904223u) >> 16; }
static csb_matrix* matrix(int R, int C, int br, int bc, int dtype, unsigned int keep) {
    const size_t nblk = (size_t)((R + br - 1) / br) * ((C + bc - 1) / bc);
    std::vector<float> W((size_t)R * C, 0.5f);
    std::vector<uint8_t> rk(nblk * br), ck(nblk * bc);
    for (uint8_t& k : rk) k = draw() % 100 < keep;
    for (uint8_t& k : ck) k = draw() % 100 < keep;
    csb_matrix* A = nullptr;
    csb_encode(W.data(), R, C, C, br, bc, rk.data(), ck.data(), dtype, -1, nullptr, &A);
    return A;
}

int main() {
    struct Size { int I, H, br, bc, ctas; unsigned int keep; };
    const Size sizes[] = {{1, 24, 8, 8, 3, 100}, {39, 96, 16, 16, 20, 60}, {153, 160, 32, 32, 40, 30}, {70, 198, 33, 7, 12, 50}, {512, 512, 64, 64, 148, 35}};
    int bad = 0;
    for (const Size& z : sizes)
        for (int cell = 0; cell < 5; ++cell)
            for (int BT : {1, 4, 8}) {
                const int dtype = (z.I + cell + BT) & 1 ? CSB_F16 : CSB_F32, S = cell == kR1Lstmp ? z.H / 2 : z.H;
                const int G = r1_gates(cell, 0) + (cell == kR1GruRb ? 1 : 0), in[2] = {z.I, S};
                csb_matrix* W[2] = {matrix(G * z.H, z.I + S, z.br, z.bc, dtype, z.keep), matrix(G * z.H, 2 * S, z.br, z.bc, dtype, z.keep)};
                csb_matrix* P[2] = {matrix(S, z.H, z.br, z.bc, dtype, z.keep), matrix(S, z.H, z.br, z.bc, dtype, z.keep)};
                auto plan = [&](size_t limit, R1HostPlan* out) { return plan_rnn1_host(cell, 2, W, cell == kR1Lstmp ? P : nullptr, in, z.H, S, BT, z.ctas, limit, out); };
                R1HostPlan all, again;
                if (plan((size_t)1 << 40, &all) != CSB_OK) continue;
                const size_t need = R1Carve(all, cell, std::max(z.I, S), z.H, S, BT).total;
                size_t longest = 0;
                for (const R1Cta& c : all.ctas) longest = std::max(longest, (size_t)c.bytes);
                const int at = plan(need, &again), below = plan(need - 1, &again);
                if (at != CSB_OK || below != 1 || longest != all.max_bytes) { std::printf("input %d hidden %d cell %d tile %d: %d %d, image %zu of %zu\n", z.I, z.H, cell, BT, at, below, longest, all.max_bytes); ++bad; }
                for (csb_matrix* A : {W[0], W[1], P[0], P[1]}) csb_free(A);
            }
    return bad ? 1 : 0;
}
