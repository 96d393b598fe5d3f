// The tile-window layout of the batched product, walked with the kernel's addressing rules: round by round, per expanding
// warp its item, per lane its segment headers and words.  Every stored value must come back once, at its place.
// Prints the failures; exit code 1 on any.
#include <cstdarg>
#include <cstdio>
#include <random>

#include "../paper_2005_05758_b200/csrc/csb_umma.hpp"

using namespace csb;

namespace csb {
void set_error(const char* f, ...) { va_list a; va_start(a, f); vprintf(f, a); va_end(a); puts(""); }
void clear_error() {}
}

// Decodes P into `got` ([output row][column], binary16 bits); returns the number of broken rules.
static int decode(const csb_matrix& A, const UmmaHostPlan& P, std::vector<uint16_t>& got) {
    int bad = 0;
    for (size_t c = 0; c < P.ctas.size(); ++c) {
        const UmmaCta& me = P.ctas[c];
        const std::vector<uint8_t>& S = P.streams[c];
        const int segs = 32 / P.seg_words, ntw = me.nw * P.MT;
        for (int r = 0; 4 * r < ntw; ++r) {
            const UmmaRound round = P.rounds[(size_t)me.table + r];
            const size_t start = (size_t)round.off16 * 16;
            if (start + round.bytes > S.size() || round.bytes % 16 || round.bytes > P.max_round) return bad + 1;
            const int nj = std::min(4, ntw - 4 * r), len = umma_unit_len(P.MT, P.flush, nj);
            for (int warp = 0; warp < 4 * nj; ++warp) {
                uint32_t at;
                std::memcpy(&at, &S[start + 4 * (size_t)warp], 4);
                const size_t item = start + at;
                const UmmaPlace place = umma_place(P.MT, len, warp >> 2);
                const int window = me.w0 + r * 4 / P.MT + place.window;
                bad += item % 16 != 0 || window >= me.w0 + me.nw;
                const UmmaQuad q = P.quads[((size_t)me.group * P.MT + place.mt) * 4 + (warp & 3)];
                for (int lane = 0; lane < 32; ++lane) {
                    const int seg = lane < q.nrows ? (q.row0 + lane) / A.block_r - q.row0 / A.block_r : 0;
                    for (int s = 0; s < segs; ++s) {
                        uint32_t h[4];
                        std::memcpy(h, &S[item + 16 * (size_t)(seg * segs + s)], 16);
                        if (!((h[0] >> lane) & 1)) continue;
                        size_t p = item + h[1] + 16 * (size_t)__builtin_popcount(h[0] & ((1u << lane) - 1));
                        for (int j = 0; j < P.seg_words; j += 4, p += 16 * (size_t)__builtin_popcount(h[0])) {
                            if (p + 16 > start + round.bytes) return bad + 1;
                            uint16_t w[8];
                            std::memcpy(w, &S[p], 16);
                            for (int o = 0; o < 8; ++o) {
                                const int64_t col = (int64_t)window * kUmmaWindow + s * 2 * P.seg_words + 2 * j + o;
                                if (col >= A.cols || lane >= q.nrows) bad += w[o] != 0;
                                else if (w[o]) { bad += got[(size_t)(q.out0 + lane) * A.cols + col] != 0; got[(size_t)(q.out0 + lane) * A.cols + col] = w[o]; }
                            }
                        }
                    }
                }
            }
        }
    }
    return bad;
}

static int check(int R, int C, int br, int bc, double keep, int MT, int S, int gates, unsigned seed) {
    std::mt19937 gen(seed);
    std::uniform_real_distribution<float> uniform(0, 1);
    std::normal_distribution<float> normal(0, 1);
    std::vector<float> W((size_t)R * C);
    for (float& w : W) w = normal(gen);
    const int nbr = (R + br - 1) / br, nbc = (C + bc - 1) / bc;
    std::vector<uint8_t> rk((size_t)nbr * nbc * br), ck((size_t)nbr * nbc * bc);
    std::vector<float> f((size_t)nbr * nbc);
    for (float& x : f) x = (float)std::min(1.0, keep * (0.2 + 1.6 * uniform(gen)));
    for (size_t i = 0; i < rk.size(); ++i) rk[i] = uniform(gen) < f[i / br];
    for (size_t i = 0; i < ck.size(); ++i) ck[i] = uniform(gen) < f[i / bc];
    csb_matrix A;
    if (encode_host(W.data(), R, C, C, br, bc, rk.data(), ck.data(), CSB_F16, &A) != CSB_OK) return 1;
    UmmaHostPlan P;
    P.windows = (C + kUmmaWindow - 1) / kUmmaWindow;
    P.seg_words = umma_seg_words(bc);
    P.flush = umma_flush(P.windows);
    P.MT = MT;
    P.S = std::min(S, P.windows);
    const int H = gates ? R / gates : 0, I = gates ? C - H : 0;
    P.quads = gates ? umma_gate_quads(gates, I, H, MT) : umma_row_quads(&A, MT);
    P.n_groups = (int)(P.quads.size() / (4 * MT));
    plan_umma_host(&A, &P);
    const int out_rows = gates ? 4 * H : R;
    std::vector<uint16_t> want((size_t)out_rows * C, 0), got((size_t)out_rows * C, 0);
    const uint16_t* v = reinterpret_cast<const uint16_t*>(A.val.data());
    for (int b = 0; b < nbr * nbc; ++b)
        for (int i = 0; i < A.m[b]; ++i)
            for (int k = 0; k < A.n[b]; ++k) {
                int row = b / nbc * br + A.row_idx[A.ridx_off[b] + i];
                const int col = b % nbc * bc + A.col_idx[A.cidx_off[b] + k];
                if (gates == 3 && row >= 2 * H && col >= I) row += H;      // the candidate's recurrent part
                want[(size_t)row * C + col] = v[A.val_off[b] + (size_t)i * A.n[b] + k] & 0x7fff ? v[A.val_off[b] + (size_t)i * A.n[b] + k] : 0;
            }
    int bad = decode(A, P, got), diff = 0;
    for (size_t i = 0; i < want.size(); ++i) diff += want[i] != got[i];
    if (bad || diff) printf("%dx%d blocks %dx%d keep %.2f MT %d S %d gates %d: %d rules broken, %d values wrong\n", R, C, br, bc, keep, MT, S, gates, bad, diff);
    return bad || diff;
}

int main() {
    int failed = 0;
    unsigned seed = 1;
    const int shapes[][2] = {{300, 1177}, {512, 192}, {33, 70}, {129, 2049}, {1, 1}, {130, 64}};
    for (auto& s : shapes)
        for (int br : {16, 24, 32, 64, 100})
            for (int bc : {16, 32, 64, 128, 192})
                for (int MT = 1; MT <= 2; ++MT) failed |= check(s[0], s[1], br, bc, 0.5, MT, 1 + (int)(seed % 8), 0, seed), ++seed;
    for (int gates = 3; gates <= 4; ++gates)
        for (int H : {32, 48, 100, 160})
            for (int I : {1, 39, 64, 153})
                for (int bc : {16, 32, 64}) failed |= check(gates * H, I + H, bc, bc, 0.5, 1 + (int)(seed & 1), 1 + (int)(seed % 4), gates, seed), ++seed;
    failed |= check(512, 4096, 64, 64, 1.0, 2, 2, 0, seed) | check(512, 1024, 16, 16, 1.0, 1, 1, 0, seed + 1) | check(700, 3000, 64, 64, 0.05, 2, 3, 0, seed + 2);
    puts(failed ? "failed" : "ok");
    return failed;
}
