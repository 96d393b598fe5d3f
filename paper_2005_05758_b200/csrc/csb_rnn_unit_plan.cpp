// Planner of the resident time loop for small products (layout: csb_rnn_unit.hpp).
#include <algorithm>
#include <atomic>
#include <new>

#include "csb_host.hpp"
#include "csb_rnn_unit.hpp"

namespace csb {

static inline size_t pad_to(size_t v, size_t a) { return (v + a - 1) / a * a; }

namespace {

struct Pair { uint16_t col; const uint8_t* v; };

// The kept weights of matrix row `row` whose columns lie in [c0, c1), as pairs with column - c0.
void row_pairs(const csb_matrix* A, int64_t row, int64_t c0, int64_t c1, std::vector<Pair>* out) {
    const int BR = A->block_r, BC = A->block_c, vs = val_size(A->val_dtype), r = (int)(row % BR);
    for (int64_t bj = c0 / BC; bj < A->nbc && bj * BC < c1; ++bj) {
        const int64_t b = row / BR * A->nbc + bj, base = bj * BC;
        const int m = A->m[b], n = A->n[b];
        const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
        const uint8_t* at = std::lower_bound(ri, ri + m, (uint8_t)r);
        if (at == ri + m || *at != r) continue;
        const uint8_t* ci = A->col_idx.data() + A->cidx_off[b];
        const uint8_t* v = A->val.data() + (A->val_off[b] + (uint64_t)(at - ri) * n) * vs;
        for (int k = 0; k < n; ++k) {
            const int64_t c = base + ci[k];
            if (c >= c0 && c < c1) out->push_back({(uint16_t)(c - c0), v + (size_t)k * vs});
        }
    }
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

struct Source { const csb_matrix* A; int64_t row0, stride; int split, zero[2]; };   // columns < split: input part

// The lists of one warp: units [u0, u0 + n) on 1 << lu unit slots.
void emit_warp(const Source& s, int cell, int op, int lu, int u0, int n, int BT, std::vector<uint8_t>& out, RuWarp* d) {
    const int rows = ru_rows(cell, op), LR = (32 / rows) >> lu, vs = val_size(s.A->val_dtype), per = vs == 2 ? 4 : 2;
    const int banks = std::max(32 / BT, 4), pass = BT == 1 ? 32 : 8;          // lanes that share a pass over the banks
    out.resize(pad_to(out.size(), 16), 0);
    d->off = (uint32_t)out.size();
    for (int p = 0; p < 2; ++p) {
        std::vector<std::vector<Pair>> pool((size_t)rows << lu);
        size_t steps = 0;
        for (int i = 0; i < n; ++i)
            for (int g = 0; g < rows; ++g) {
                // GRU: rows 2 and 3 are the candidate's input and recurrent part
                if (cell == kR1Gru && g >= 2 && g - 2 != p) continue;
                std::vector<Pair>& v = pool[(size_t)i * rows + g];
                row_pairs(s.A, s.row0 + (cell == kR1Gru ? std::min(g, 2) : g) * s.stride + u0 + i, p ? s.split : 0, p ? s.A->cols : s.split, &v);
                steps = std::max(steps, (v.size() + LR - 1) / LR);
            }
        const size_t rounds = (steps + per - 1) / per;
        d->n[p] = (uint16_t)rounds;
        const size_t base = out.size();
        out.resize(base + rounds * 512, 0);
        std::vector<int> used((size_t)banks);
        for (size_t k = 0; k < rounds * per; ++k)
            for (int l0 = 0; l0 < 32; l0 += pass) {
                std::fill(used.begin(), used.end(), -1);
                for (int i = 0; i < pass; ++i) {
                    const int l = l0 + (i + 11 * (int)k) % pass, row = l / LR;        // another lane chooses first in every step
                    std::vector<Pair>& v = pool[row];
                    uint16_t col = (uint16_t)s.zero[p];
                    const uint8_t* val = nullptr;
                    if (!v.empty()) {
                        size_t best = v.size() - 1;
                        for (size_t q = v.size(), end = q > 24 ? q - 24 : 0; q-- > end;) { const int u = used[v[q].col % banks]; if (u < 0 || u == v[q].col) { best = q; break; } }
                        col = v[best].col; val = v[best].v;
                        v[best] = v.back();
                        v.pop_back();
                        used[col % banks] = col;
                    }
                    uint8_t* q = out.data() + base + (k / per) * 512 + (size_t)l * 16 + (k % per) * (vs == 2 ? 4 : 8);
                    if (vs == 2) { std::memcpy(q, &col, 2); if (val) std::memcpy(q + 2, val, 2); }
                    else { const uint32_t c = col; std::memcpy(q, &c, 4); if (val) std::memcpy(q + 4, val, 4); }
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
                    const Source s{proj ? Wp[j.layer] : W[j.layer], op == 1 && !proj ? 2 * (int64_t)H : 0, H, proj ? 0 : in_size[j.layer],
                                   {in_size[j.layer], op == 1 ? H : S}};
                    int lu = 0;
                    while (kR1Warps << lu < j.units[op]) ++lu;
                    ct.units[op] = (uint16_t)j.units[op]; ct.unit0[op] = (uint32_t)j.u0[op]; ct.lu[op] = (uint16_t)lu;
                    for (int w = 0; w << lu < j.units[op]; ++w) {
                        RuWarp d{};
                        emit_warp(s, cell, op, lu, j.u0[op] + (w << lu), std::min(1 << lu, j.units[op] - (w << lu)), BT, b, &d);
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
    out->bytes.resize(base);
    base = 0;
    for (auto& i : img) { std::memcpy(out->bytes.data() + base, i.data(), i.size()); base += i.size(); std::vector<uint8_t>().swap(i); }
    out->ctas = std::move(ctas);
    return CSB_OK;
}

}  // namespace csb
