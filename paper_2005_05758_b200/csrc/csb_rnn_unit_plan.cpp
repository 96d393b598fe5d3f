// Planner of the resident time loop for small products (layout: csb_rnn_unit.hpp).
#include <algorithm>
#include <atomic>
#include <new>

#include "csb_host.hpp"
#include "csb_rnn_unit.hpp"

namespace csb {

static inline size_t pad_to(size_t v, size_t a) { return (v + a - 1) / a * a; }

namespace {

// Rows of a CTA's part of a product (gate by gate, units [u0, u0 + units)), and which columns are the input part (< split).
struct Source { const csb_matrix* A; int64_t row0, stride; int gates, u0, units, split, zero[2]; };

// The pairs of a CTA's rows, part by part and row by row: where row r of part p starts, the columns (counted from the
// part's first) and the values.
struct Pairs {
    std::vector<uint32_t> first[2], fill;
    std::vector<uint16_t> col[2];
    std::vector<uint32_t> val[2];              // the bits of the value
};
// Every (block, kept row of the source): f(row, block's kept columns before the split, block, place among the kept rows).
template <typename F>
void for_rows(const Source& s, F f) {
    const csb_matrix* A = s.A;
    const int BR = A->block_r, BC = A->block_c;
    for (int g = 0; g < s.gates; ++g) {
        const int64_t lo = s.row0 + g * s.stride + s.u0, hi = lo + s.units;
        for (int64_t bi = lo / BR; bi * BR < hi; ++bi) {
            const int a = (int)std::max<int64_t>(0, lo - bi * BR), z = (int)std::min<int64_t>(BR, hi - bi * BR);
            for (int64_t bj = 0; bj < A->nbc; ++bj) {
                const int64_t b = bi * A->nbc + bj, c0 = bj * BC;
                const int m = A->m[b], n = A->n[b];
                if (!m || !n) continue;
                const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
                const uint8_t* ci = A->col_idx.data() + A->cidx_off[b];
                int at = (int)(std::lower_bound(ri, ri + m, a) - ri);
                if (at == m || ri[at] >= z) continue;
                const int cut = c0 >= s.split ? 0 : c0 + BC <= s.split ? n : (int)(std::lower_bound(ci, ci + n, (int)(s.split - c0)) - ci);
                for (; at < m && ri[at] < z; ++at) f((int)(g * s.units + bi * BR + ri[at] - lo), cut, b, at);
            }
        }
    }
}
// (a pass that counts and one that fills: a binary search per block, not per row and block)
void collect(const Source& s, Pairs* P) {
    const csb_matrix* A = s.A;
    const int vs = val_size(A->val_dtype), BC = A->block_c;
    const size_t rows = (size_t)s.gates * s.units;
    for (auto& f : P->first) f.assign(rows + 1, 0);
    for_rows(s, [&](int r, int cut, int64_t b, int) { P->first[0][r + 1] += cut; P->first[1][r + 1] += A->n[b] - cut; });
    for (int p = 0; p < 2; ++p) {
        for (size_t r = 0; r < rows; ++r) P->first[p][r + 1] += P->first[p][r];
        P->col[p].resize(P->first[p][rows]); P->val[p].resize(P->first[p][rows]);
    }
    P->fill.assign(2 * rows, 0);
    for_rows(s, [&](int r, int cut, int64_t b, int place) {
        const uint8_t* ci = A->col_idx.data() + A->cidx_off[b];
        const int n = A->n[b], c0 = (int)(b % A->nbc) * BC;
        const uint8_t* v = A->val.data() + (A->val_off[b] + (uint64_t)place * n) * vs;
        for (int p = 0; p < 2; ++p) {
            const int from = p ? cut : 0, to = p ? n : cut, base = p ? c0 - s.split : c0;
            uint32_t at = P->first[p][r] + P->fill[2 * r + p];
            for (int k = from; k < to; ++k, ++at) { P->col[p][at] = (uint16_t)(base + ci[k]); P->val[p][at] = 0; std::memcpy(&P->val[p][at], v + (size_t)k * vs, vs); }
            P->fill[2 * r + p] += (uint32_t)(to - from);
        }
    });
}

std::vector<double> row_weights(const csb_matrix* A) {
    std::vector<double> w((size_t)A->rows, 0.0);
    for (int64_t b = 0; b < A->nblk; ++b) {
        const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
        for (int r = 0; r < A->m[b]; ++r) w[(b / A->nbc) * A->block_r + ri[r]] += A->n[b];
    }
    return w;
}

// Contiguous ranges of units, at most `parts` of them and `most` units each, of about equal cost.
std::vector<int> cut_units(const std::vector<double>& cost, int parts, int most) {
    const int n = (int)cost.size();
    auto pack = [&](double T, std::vector<int>* cut) {
        int used = 1, start = 0;
        double cur = 0;
        if (cut) cut->assign(1, 0);
        for (int u = 0; u < n; ++u) {
            if (u > start && (cur + cost[u] > T || u - start >= most)) { if (cut) cut->push_back(u); start = u; cur = 0; ++used; }
            cur += cost[u];
        }
        if (cut) cut->push_back(n);
        return used;
    };
    double lo = 0, hi = 1;
    for (double c : cost) hi += c;
    for (int i = 0; i < 40; ++i) { const double mid = 0.5 * (lo + hi); if (pack(mid, nullptr) <= parts) hi = mid; else lo = mid; }
    std::vector<int> cut;
    pack(hi, &cut);
    return cut;
}

// The lists of one warp: units [w0, w0 + n) of the CTA's on 1 << lu unit slots.  Takes the pairs out of P.
void emit_warp(const Source& s, Pairs& P, int cell, int op, int lu, int w0, int n, int BT, std::vector<uint8_t>& out, RuWarp* d) {
    const int rows = ru_rows(cell, op), LR = (32 / rows) >> lu, lr_log = __builtin_ctz(LR), vs = val_size(s.A->val_dtype);
    const int per_log = vs == 2 ? 2 : 1, per = 1 << per_log;                  // pairs in 16 bytes
    const int banks = std::max(32 / BT, 4), pass = BT == 1 ? 32 : 8;          // lanes that share a pass over the banks
    out.resize(pad_to(out.size(), 16), 0);
    d->off = (uint32_t)out.size();
    for (int p = 0; p < 2; ++p) {
        uint32_t from[32] = {}, left[32] = {};                                // per row on the warp's lanes
        size_t steps = 0;
        for (int i = 0; i < n; ++i)
            for (int g = 0; g < rows; ++g) {
                // GRU: rows 2 and 3 are the candidate's input and recurrent part
                if (cell == kR1Gru && g >= 2 && g - 2 != p) continue;
                const int r = (cell == kR1Gru ? std::min(g, 2) : g) * s.units + w0 + i;
                from[i * rows + g] = P.first[p][r]; left[i * rows + g] = P.first[p][r + 1] - P.first[p][r];
                steps = std::max(steps, ((size_t)left[i * rows + g] + LR - 1) / LR);
            }
        const size_t rounds = (steps + per - 1) / per, base = out.size();
        d->n[p] = (uint16_t)rounds;
        out.resize(base + rounds * 512, 0);
        for (size_t k = 0; k < rounds * per; ++k) {
            uint8_t* to = out.data() + base + (k >> per_log) * 512 + (k & (per - 1)) * (vs == 2 ? 4 : 8);
            for (int l0 = 0; l0 < 32; l0 += pass) {
                uint32_t used = 0u;
                uint16_t used_col[32];
                for (int i = 0; i < pass; ++i) {
                    const int l = l0 + ((i + 11 * (int)k) & (pass - 1)), row = l >> lr_log;       // another lane chooses first in every step
                    uint32_t c = (uint32_t)s.zero[p], bits = 0u;
                    if (left[row]) {
                        // the last pair whose bank no lane of the pass reads, or whose column one reads already
                        uint16_t* col = P.col[p].data() + from[row];
                        uint32_t* val = P.val[p].data() + from[row];
                        const uint32_t last = --left[row];
                        uint32_t best = last;
                        for (uint32_t q = last + 1, end = q > 24 ? q - 24 : 0; q-- > end;) {
                            const uint32_t b = col[q] & (uint32_t)(banks - 1);
                            if (!(used >> b & 1u) || used_col[b] == col[q]) { best = q; break; }
                        }
                        c = col[best]; bits = val[best];
                        col[best] = col[last]; val[best] = val[last];
                        used |= 1u << (c & (uint32_t)(banks - 1));
                        used_col[c & (uint32_t)(banks - 1)] = (uint16_t)c;
                    }
                    if (vs == 2) { const uint32_t w = c | bits << 16; std::memcpy(to + l * 16, &w, 4); }
                    else { std::memcpy(to + l * 16, &c, 4); std::memcpy(to + l * 16 + 4, &bits, 4); }
                }
            }
        }
    }
}

}  // namespace

int plan_unit_host(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, int n_ctas,
                   RuHostPlan* out) {
    *out = RuHostPlan{};
    const int ops = r1_ops(cell);
    for (int l = 0; l < L; ++l) if (in_size[l] >= 65535 || S >= 65535 || H >= 65535) return 1;
    if (n_ctas < L) return 1;
    // units a warp may take: a row needs at least as many lanes as there are batch columns
    int max_lu[2];
    for (int op = 0; op < 2; ++op) { max_lu[op] = 0; while (max_lu[op] < 2 && ((32 / ru_rows(cell, op)) >> (max_lu[op] + 1)) >= BT) ++max_lu[op]; }
    const int G = r1_gates(cell, 0) + (cell == kR1GruRb ? 1 : 0);
    std::vector<std::vector<double>> unit_cost(L), proj_cost(L);
    std::vector<double> layer_cost(L, 0.0);
    for (int l = 0; l < L; ++l) {
        const std::vector<double> w = row_weights(W[l]);
        unit_cost[l].assign(H, 32.0);
        for (int g = 0; g < G; ++g) for (int u = 0; u < H; ++u) unit_cost[l][u] += w[(size_t)g * H + u];
        if (cell == kR1Lstmp) { proj_cost[l] = row_weights(Wp[l]); for (double& c : proj_cost[l]) c += 32.0; }
        for (double c : unit_cost[l]) layer_cost[l] += c;
        for (double c : proj_cost[l]) layer_cost[l] += c;
    }
    std::vector<int> per(L, 1);
    for (int used = L; used < n_ctas; ++used) {
        int best = 0;
        for (int l = 1; l < L; ++l) if (layer_cost[l] / per[l] > layer_cost[best] / per[best]) best = l;
        ++per[best];
    }
    struct Job { int layer, u0[2], units[2]; };
    std::vector<Job> jobs;
    for (int l = 0; l < L; ++l) {
        // as few units per warp as the CTAs allow
        auto most = [&](int units, int op) { int lu = 0; while (lu < max_lu[op] && (int64_t)per[l] * (kR1Warps << lu) < units) ++lu; return kR1Warps << lu; };
        const std::vector<int> cu = cut_units(unit_cost[l], per[l], most(H, 0));
        std::vector<int> cp;
        if (cell == kR1Lstmp) cp = cut_units(proj_cost[l], per[l], most(S, 1));
        const int n = std::max((int)cu.size(), (int)cp.size()) - 1;
        if (n > per[l]) return 1;
        for (int i = 0; i < n; ++i) {
            Job j{l, {0, 0}, {0, 0}};
            if (i + 1 < (int)cu.size()) { j.u0[0] = cu[i]; j.units[0] = cu[i + 1] - cu[i]; }
            if (cell == kR1GruRb) { j.u0[1] = j.u0[0]; j.units[1] = j.units[0]; }
            if (i + 1 < (int)cp.size()) { j.u0[1] = cp[i]; j.units[1] = cp[i + 1] - cp[i]; }
            if (ops == 2 && j.units[1] > kR1Warps << max_lu[1]) return 1;
            jobs.push_back(j);
        }
        out->layer_ctas[l] = n;
    }
    std::vector<std::vector<uint8_t>> img(jobs.size());
    std::vector<RuCta> ctas(jobs.size());
    std::atomic<int> next{0}, status{CSB_OK};
    auto work = [&]() {
        Pairs P;
        for (int c; status.load() == CSB_OK && (c = next.fetch_add(1)) < (int)jobs.size();) {
            try {
                const Job& j = jobs[c];
                RuCta& ct = ctas[c];
                ct = RuCta{};
                ct.layer = j.layer;
                std::vector<uint8_t>& b = img[c];
                b.assign(2 * kR1Warps * sizeof(RuWarp), 0);
                for (int op = 0; op < ops; ++op) {
                    const bool proj = cell == kR1Lstmp && op == 1;
                    const Source s{proj ? Wp[j.layer] : W[j.layer], op == 1 && !proj ? 2 * (int64_t)H : 0, H, op == 1 ? 1 : r1_gates(cell, 0), j.u0[op],
                                   j.units[op], proj ? 0 : in_size[j.layer], {in_size[j.layer], op == 1 ? H : S}};
                    collect(s, &P);
                    int lu = 0;
                    while (kR1Warps << lu < j.units[op]) ++lu;
                    ct.units[op] = (uint16_t)j.units[op]; ct.unit0[op] = (uint32_t)j.u0[op]; ct.lu[op] = (uint16_t)lu;
                    for (int w = 0; w << lu < j.units[op]; ++w) {
                        RuWarp d{};
                        emit_warp(s, P, cell, op, lu, w << lu, std::min(1 << lu, j.units[op] - (w << lu)), BT, b, &d);
                        std::memcpy(b.data() + (op * kR1Warps + w) * sizeof(RuWarp), &d, sizeof d);
                    }
                }
                b.resize(pad_to(b.size(), 128), 0);
            } catch (const std::bad_alloc&) { status.store(CSB_ERR_ALLOC); }
        }
    };
    run_on_threads((int)std::min<size_t>(16, std::max<size_t>(1, jobs.size() / 4)), work);
    if (status.load() == CSB_ERR_ALLOC) throw std::bad_alloc();
    size_t base = 0;
    for (size_t c = 0; c < jobs.size(); ++c) {
        ctas[c].off16 = (uint32_t)(base / 16); ctas[c].bytes = (uint32_t)img[c].size();
        base += img[c].size();
        out->max_bytes = std::max(out->max_bytes, img[c].size());
    }
    out->bytes.reserve(base);
    for (auto& i : img) { out->bytes.insert(out->bytes.end(), i.begin(), i.end()); std::vector<uint8_t>().swap(i); }
    out->ctas = std::move(ctas);
    return CSB_OK;
}

}  // namespace csb
