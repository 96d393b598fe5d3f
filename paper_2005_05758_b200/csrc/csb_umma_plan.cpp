// Planner of the batched product on tcgen05 tensor cores: the layout of csb_umma.hpp.
#include <algorithm>
#include <atomic>
#include <new>

#include "csb_host.hpp"
#include "csb_umma.hpp"

namespace csb {

std::vector<UmmaQuad> umma_row_quads(const csb_matrix* A, int MT) {
    const int64_t per = 128 * MT, groups = (A->rows + per - 1) / per;
    std::vector<UmmaQuad> q((size_t)(groups * MT * 4));
    for (size_t i = 0; i < q.size(); ++i) {
        const int64_t r0 = (int64_t)i * 32;
        q[i] = UmmaQuad{(int32_t)std::min(r0, A->rows), (int32_t)std::max<int64_t>(0, std::min<int64_t>(32, A->rows - r0)), 0, (int32_t)A->cols, (int32_t)r0, {}};
    }
    return q;
}

std::vector<UmmaQuad> umma_gate_quads(int gates, int in_size, int H, int MT) {
    const int per = 32 * MT, groups = (H + per - 1) / per;
    std::vector<UmmaQuad> q((size_t)groups * MT * 4);
    for (size_t i = 0; i < q.size(); ++i) {
        const int g = (int)(i & 3), u0 = (int)(i >> 2) * 32, row = gates == 3 && g == 3 ? 2 : g;
        q[i] = UmmaQuad{row * H + std::min(u0, H), std::max(0, std::min(32, H - u0)), gates == 3 && g == 3 ? in_size : 0,
                        gates == 3 && g == 2 ? in_size : in_size + H, g * H + u0, {}};
    }
    return q;
}

// A CTA's time follows its tile-windows (expansion and tensor instructions); the inputs of a window cost a CTA as
// much again as half a tile-window, whatever the number of tiles that use them; a cluster adds its barriers and sums.
double umma_cost(int MT, int S, int windows) { return ((windows + S - 1) / S) * (MT + 0.5) + (S > 1 ? 4.0 + 0.5 * S : 0.0); }

void umma_shape(int tiles, int windows, const int* clusters, int* MT, int* S) {
    double best = 1e300;
    for (int mt = kUmmaMaxMT; mt >= 1; --mt)
        for (int s = 1; s <= std::min<int>(kUmmaMaxS, windows); ++s) {
            if (clusters[s] < 1) continue;
            const int groups = (tiles + mt - 1) / mt;
            const double cost = ((groups + clusters[s] - 1) / clusters[s]) * umma_cost(mt, s, windows);
            if (cost < best) { best = cost; *MT = mt; *S = s; }
        }
}

namespace {

// One item: quadrant q over the window that starts at column w0.  Appends to `out`; `next` is filled in later.
struct ItemWriter {
    const csb_matrix* A;
    int seg_words;

    int segments(const UmmaQuad& q) const { return q.nrows ? (int)((q.row0 + q.nrows - 1) / A->block_r - q.row0 / A->block_r) + 1 : 1; }

    // One (row segment, column segment), the columns from `col` on: appends its values, returns the masks of its kept rows and columns.
    uint32_t segment(const UmmaQuad& q, int g, int64_t col, std::vector<uint8_t>& out, uint64_t* columns) const {
        if (!q.nrows || col >= A->cols) return 0;
        const int64_t bi = q.row0 / A->block_r + g, bj = col / A->block_c, b = bi * A->nbc + bj;
        const int m = A->m[b], n = A->n[b], base = (int)(col - bj * A->block_c);
        const uint8_t* ci = A->col_idx.data() + A->cidx_off[b];
        const int64_t c0 = std::max<int64_t>(0, q.c0 - bj * A->block_c), c1 = q.c1 - bj * A->block_c;   // in-block columns that count
        const int k0 = (int)(std::lower_bound(ci, ci + n, std::max<int64_t>(base, c0)) - ci);
        const int k1 = (int)(std::lower_bound(ci, ci + n, std::min<int64_t>(base + 2 * seg_words, std::max<int64_t>(0, c1))) - ci);
        if (k0 >= k1) return 0;
        const int64_t r0 = bi * A->block_r - q.row0;           // lane of the block-row's first row (may be negative)
        const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
        uint32_t rows = 0;
        int first = 0;
        for (int i = 0; i < m; ++i) {
            const int64_t lane = r0 + ri[i];
            if (lane < 0 || lane >= q.nrows) continue;
            if (!rows) first = i;
            rows |= 1u << lane;
        }
        if (!rows) return 0;
        const int kr = __builtin_popcount(rows);
        const size_t at = out.size();
        out.resize(at + (size_t)kr * seg_words * 4, 0);
        uint16_t* v = reinterpret_cast<uint16_t*>(out.data() + at);
        const uint16_t* src = reinterpret_cast<const uint16_t*>(A->val.data()) + A->val_off[b] + (size_t)first * n;
        uint16_t place[64];                                    // of the kept columns, in the first row
        for (int k = k0; k < k1; ++k) {
            const int c = ci[k] - base;
            place[k - k0] = (uint16_t)((c >> 3) * kr * 8 + (c & 7));
            *columns |= 1ull << c;
        }
        for (int i = 0; i < kr; ++i, src += n, v += 8)
            for (int k = k0; k < k1; ++k) v[place[k - k0]] = src[k];
        return rows;
    }

    void write(const UmmaQuad& q, int64_t w0, std::vector<uint8_t>& out) const {
        const size_t start = out.size();
        const int ng = segments(q), ns = 32 / seg_words;
        out.resize(start + (size_t)ng * ns * 16, 0);
        for (int g = 0; g < ng; ++g)
            for (int s = 0; s < ns; ++s) {
                uint32_t h[4] = {0u, (uint32_t)(out.size() - start), 0u, 0u};
                uint64_t columns = 0;
                h[0] = segment(q, g, w0 + (int64_t)s * 2 * seg_words, out, &columns);
                h[2] = (uint32_t)columns; h[3] = (uint32_t)(columns >> 32);
                std::memcpy(out.data() + start + (size_t)(g * ns + s) * 16, h, 16);
            }
    }
};

void plan_cta(const csb_matrix* A, const UmmaHostPlan& P, const UmmaCta& cta, UmmaRound* rounds, std::vector<uint8_t>* out) {
    const ItemWriter w{A, P.seg_words};
    const int ntw = cta.nw * P.MT, per = 4 / P.MT;         // windows of a round
    out->clear();
    for (int r = 0; 4 * r < ntw; ++r) {
        const int nj = std::min(4, ntw - 4 * r), len = umma_unit_len(P.MT, P.flush, nj);
        const size_t start = out->size();
        uint32_t table[kUmmaExpandWarps] = {};
        out->resize(start + sizeof table);
        for (int j = 0; j < nj; ++j) {
            const UmmaPlace at = umma_place(P.MT, len, j);
            for (int q = 0; q < 4; ++q) {
                table[j * 4 + q] = (uint32_t)(out->size() - start);
                w.write(P.quads[((size_t)cta.group * P.MT + at.mt) * 4 + q], (int64_t)(cta.w0 + r * per + at.window) * kUmmaWindow, *out);
            }
        }
        std::memcpy(out->data() + start, table, sizeof table);
        rounds[r] = UmmaRound{(uint32_t)(start / 16), (uint32_t)(out->size() - start)};
    }
}

}  // namespace

void plan_umma_host(const csb_matrix* A, UmmaHostPlan* P) {
    P->ctas.assign((size_t)P->n_groups * P->S, UmmaCta{});
    P->streams.assign(P->ctas.size(), {});
    P->rounds.clear();
    for (int g = 0; g < P->n_groups; ++g)
        for (int s = 0; s < P->S; ++s) {
            UmmaCta& c = P->ctas[(size_t)g * P->S + s];
            c.group = g; c.split = s;
            c.w0 = (int)((int64_t)P->windows * s / P->S);
            c.nw = (int)((int64_t)P->windows * (s + 1) / P->S) - c.w0;
            c.table = (int)P->rounds.size();
            P->rounds.resize(P->rounds.size() + (size_t)(c.nw * P->MT + 3) / 4);
        }
    // the CTAs' streams are independent of one another
    std::atomic<size_t> next{0};
    std::atomic<bool> failed{false};
    run_on_threads(A->nnz < 100000 ? 1 : (int)std::min<size_t>((size_t)P->threads, P->ctas.size()), [&]() {
        try {
            std::vector<uint8_t> scratch;                  // (room for the worst case for each CTA took a third to a half longer)
            for (size_t i; (i = next.fetch_add(1)) < P->ctas.size() && !failed;) {
                plan_cta(A, *P, P->ctas[i], P->rounds.data() + P->ctas[i].table, &scratch);
                P->streams[i].assign(scratch.begin(), scratch.end());
            }
        } catch (const std::bad_alloc&) { failed = true; }
    });
    if (failed) throw std::bad_alloc();
    P->total128 = 0;
    for (size_t i = 0; i < P->ctas.size(); ++i) {
        P->ctas[i].off128 = (uint32_t)P->total128;
        P->total128 += (P->streams[i].size() + 127) / 128;
    }
    P->max_round = 0;
    for (const UmmaRound& r : P->rounds) P->max_round = std::max(P->max_round, r.bytes);
}

}  // namespace csb
