// Planner of the resident time loop (layout: csb_rnn1.hpp).
//
// Hidden units are cut into one contiguous range per CTA, the CTAs dealt to the layers in proportion to
// their weights.  A range that ends inside a block-row makes two CTAs fetch the inputs of its blocks,
// so the cut is tried at several granularities (units one by one up to whole block-rows) and the one
// whose longest CTA is modelled shortest is taken.
#include <algorithm>
#include <atomic>
#include <new>

#include "csb_host.hpp"
#include "csb_rnn1.hpp"

namespace csb {

static inline size_t pad_to(size_t v, size_t a) { return (v + a - 1) / a * a; }

namespace {

struct OpSource { const csb_matrix* A; int64_t row0, gate_stride; int gates, unit0, units, split; };   // columns < split: input part

// A chunk of a block's kept columns times some of its kept rows.
struct Task {
    const csb_matrix* A;
    int64_t block;
    int k0, k1, r0, r1;          // ranges into the block's kept-column and kept-row lists
    int row_base;                // local row of in-block row 0 (may be negative)
    int col_base;                // index in the staged vector of in-block column 0 (may be negative)
};

// Every (block, kept rows of the CTA, columns of a part): f(part, block, ra, rz, k0, k1, row_base, col_base)
template <typename F>
void for_pieces(const OpSource& s, F f) {
    const csb_matrix* A = s.A;
    const int BR = A->block_r, BC = A->block_c;
    for (int g = 0; g < s.gates; ++g) {
        const int64_t lo = s.row0 + g * s.gate_stride + s.unit0, hi = lo + s.units;
        for (int64_t bi = lo / BR; bi * BR < hi; ++bi) {
            const int a = (int)std::max<int64_t>(0, lo - bi * BR), z = (int)std::min<int64_t>(BR, hi - bi * BR);
            for (int64_t bj = 0; bj < A->nbc; ++bj) {
                const int64_t b = bi * A->nbc + bj, c0 = bj * BC;
                const int m = A->m[b], n = A->n[b];
                if (!m || !n) continue;
                const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
                const uint8_t* ci = A->col_idx.data() + A->cidx_off[b];
                const int ra = (int)(std::lower_bound(ri, ri + m, a) - ri), rz = (int)(std::lower_bound(ri, ri + m, z) - ri);
                if (ra == rz) continue;
                const int cut = c0 >= s.split ? 0 : c0 + BC <= s.split ? n : (int)(std::lower_bound(ci, ci + n, (int)(s.split - c0)) - ci);
                const int row_base = (int)(bi * BR - lo) + g * s.units;
                if (cut > 0) f(0, b, ra, rz, 0, cut, row_base, (int)c0);
                if (cut < n) f(1, b, ra, rz, cut, n, row_base, (int)(c0 - s.split));
            }
        }
    }
}

// What a lane pays, in shared-memory passes: fetching a chunk's inputs, and a row of it.
constexpr double kTaskCost = 14.0, kRowCost = 6.0;

double range_cost(const OpSource& s, int wide) {
    double c = 0;
    for_pieces(s, [&](int, int64_t, int ra, int rz, int k0, int k1, int, int) { c += ((k1 - k0 + wide - 1) / wide) * (kTaskCost + kRowCost * (rz - ra)); });
    return c;
}

template <typename V>
uint32_t append(std::vector<uint8_t>& b, const V* p, size_t n) {
    b.resize(pad_to(b.size(), 16), 0);
    const uint32_t at = (uint32_t)b.size();
    b.resize(at + pad_to(n * sizeof(V), 16), 0);
    if (n) std::memcpy(b.data() + at, p, n * sizeof(V));
    return at;
}

struct Image { std::vector<uint8_t> bytes; size_t partials[2] = {0, 0}, rows = 0; };

// Lays one product out behind the image; returns 1 when it does not fit the layout.
int emit_op(const OpSource& s, const int zero[2], int op, int BT, Image* img) {
    const int wide = r1_wide(BT), vs = val_size(s.A->val_dtype);
    const size_t n_rows = (size_t)s.gates * s.units;
    // lanes that share a pass over the banks, and the banks (in units of BT floats) they must keep apart
    const int pass = BT == 1 ? 32 : BT == 2 ? 16 : 8, banks = std::max(32 / BT, 4);
    // ---- tasks: rows at most so many that there is about one group for every warp
    std::vector<Task> tasks[2][2];             // [part][narrow]
    std::vector<uint32_t> count[2];            // partial sums per row and part
    for (int p = 0; p < 2; ++p) {
        int limit = kR1MaxRows;
        for (;; limit = std::max(1, limit / 2)) {
            for (auto& v : tasks[p]) v.clear();
            count[p].assign(n_rows, 0);
            for_pieces(s, [&](int part, int64_t b, int ra, int rz, int k0, int k1, int row_base, int col_base) {
                if (part != p) return;
                const int splits = (rz - ra + limit - 1) / limit;
                for (int k = k0; k < k1; k += wide) {
                    const int ke = std::min(k1, k + wide);
                    for (int i = 0; i < splits; ++i) {
                        const int x = ra + (rz - ra) * i / splits, y = ra + (rz - ra) * (i + 1) / splits;
                        tasks[p][ke - k <= wide / 2].push_back({s.A, b, k, ke, x, y, row_base, col_base});
                    }
                    for (int r = ra; r < rz; ++r) ++count[p][row_base + s.A->row_idx[s.A->ridx_off[b] + r]];
                }
            });
            // halving the rows must not make more groups than there are warps
            const size_t groups = (tasks[p][0].size() + 31) / 32 + (tasks[p][1].size() + 31) / 32;
            if (limit == 1 || groups * 2 > (size_t)kR1Warps) break;
        }
    }
    // ---- places of the partial sums: row by row, input part then recurrent part, in quads; then one per lane for idle lanes
    std::vector<R1Row> rows(std::max<size_t>(n_rows, 1));
    std::vector<uint32_t> first[2] = {std::vector<uint32_t>(n_rows), std::vector<uint32_t>(n_rows)};
    size_t at = 0;
    for (size_t r = 0; r < n_rows; ++r)
        for (int p = 0; p < 2; ++p) {
            const size_t q = (count[p][r] + 3) / 4;
            rows[r].base[p] = (uint16_t)(at / 4); rows[r].quads[p] = (uint16_t)q;
            first[p][r] = (uint32_t)at;
            at += 4 * q;
        }
    const size_t idle = at;
    at += 32;
    if (at > 65535) return 1;
    img->partials[op] = at;
    img->rows = std::max(img->rows, n_rows);
    std::vector<std::vector<uint16_t>> free_places[2];
    for (int p = 0; p < 2; ++p) {
        free_places[p].resize(n_rows);
        for (size_t r = 0; r < n_rows; ++r) for (uint32_t i = 0; i < count[p][r]; ++i) free_places[p][r].push_back((uint16_t)(first[p][r] + i));
    }
    // ---- groups: 32 tasks of about the same number of rows, longest first to the warp with the least work
    std::vector<R1Group> groups[kR1Warps][2];
    double load[kR1Warps] = {};
    for (int p = 0; p < 2; ++p) {
        struct G { size_t from; int narrow, rows; };
        std::vector<G> order;
        for (int nw = 0; nw < 2; ++nw) {
            std::vector<Task>& v = tasks[p][nw];
            std::stable_sort(v.begin(), v.end(), [](const Task& a, const Task& b) { return a.r1 - a.r0 > b.r1 - b.r0; });
            for (size_t i = 0; i < v.size(); i += 32) order.push_back({i, nw, v[i].r1 - v[i].r0});
        }
        std::stable_sort(order.begin(), order.end(), [](const G& a, const G& b) { return a.rows > b.rows; });
        double part_load[kR1Warps] = {};
        for (const G& g : order) {
            int w = 0;
            for (int i = 1; i < kR1Warps; ++i) if (part_load[i] < part_load[w] || (part_load[i] == part_load[w] && load[i] < load[w])) w = i;
            const double cost = kTaskCost + kRowCost * g.rows;
            part_load[w] += cost; load[w] += cost;
            const std::vector<Task>& v = tasks[p][g.narrow];
            const size_t lanes = std::min<size_t>(32, v.size() - g.from);
            const int width = g.narrow ? wide / 2 : wide;
            // order of the columns inside each lane's chunk: in each step different banks within a pass
            std::vector<uint16_t> cols((size_t)32 * width, (uint16_t)zero[p]);
            std::vector<int> pick((size_t)32 * width, -1);
            std::vector<uint32_t> left(32, 0);
            for (size_t l = 0; l < lanes; ++l) left[l] = (1u << (v[g.from + l].k1 - v[g.from + l].k0)) - 1u;
            for (int k = 0; k < width; ++k)
                for (int l0 = 0; l0 < 32; l0 += pass) {
                    std::vector<int> used((size_t)banks, -1);
                    for (int l = l0; l < l0 + pass; ++l) {
                        if (!left[l]) continue;
                        const Task& t = v[g.from + l];
                        const uint8_t* ci = t.A->col_idx.data() + t.A->cidx_off[t.block] + t.k0;
                        int best = -1, col = 0;
                        for (int i = 0; i < t.k1 - t.k0; ++i) {
                            if (!(left[l] >> i & 1u)) continue;
                            const int c = t.col_base + ci[i], u = used[c % banks];
                            if (best < 0) { best = i; col = c; }
                            if (u < 0 || u == c) { best = i; col = c; break; }
                        }
                        used[col % banks] = col;
                        left[l] &= ~(1u << best);
                        cols[(size_t)l * width + k] = (uint16_t)col;
                        pick[(size_t)l * width + k] = best;
                    }
                }
            std::vector<uint8_t> w_bytes((size_t)g.rows * 32 * width * vs, 0);
            std::vector<uint16_t> pos((size_t)((g.rows + 1) / 2) * 64, 0);
            for (int r = 0; r < (g.rows + 1) / 2 * 2; ++r)
                for (int l0 = 0; l0 < 32; l0 += pass) {
                    std::vector<uint8_t> used((size_t)banks, 0);
                    for (int l = l0; l < l0 + pass; ++l) {
                        uint16_t place = (uint16_t)(idle + l);
                        if ((size_t)l < lanes && r < v[g.from + l].r1 - v[g.from + l].r0) {
                            const Task& t = v[g.from + l];
                            const int row = t.row_base + t.A->row_idx[t.A->ridx_off[t.block] + t.r0 + r];
                            std::vector<uint16_t>& fp = free_places[p][row];
                            size_t best = fp.size() - 1;
                            for (size_t i = fp.size(); i-- > 0;) if (!used[fp[i] % banks]) { best = i; break; }
                            place = fp[best];
                            fp[best] = fp.back();
                            fp.pop_back();
                            const uint8_t* src = t.A->val.data() + (t.A->val_off[t.block] + (uint64_t)(t.r0 + r) * t.A->n[t.block] + t.k0) * vs;
                            uint8_t* dst = w_bytes.data() + ((size_t)r * 32 + l) * width * vs;
                            // fp32 values, eight columns: two halves of 16 bytes per lane, [half][lane]
                            for (int k = 0; k < width; ++k) {
                                const int i = pick[(size_t)l * width + k];
                                if (i < 0) continue;
                                uint8_t* d = width * vs == 32 ? w_bytes.data() + (((size_t)r * 2 + k / 4) * 32 + l) * 16 + (k % 4) * 4 : dst + (size_t)k * vs;
                                std::memcpy(d, src + (size_t)i * vs, vs);
                            }
                        }
                        used[place % banks] = 1;
                        pos[((size_t)(r / 2) * 32 + l) * 2 + (r & 1)] = place;
                    }
                }
            R1Group d{};
            d.cols_off = append(img->bytes, cols.data(), cols.size());
            d.w_off = append(img->bytes, w_bytes.data(), w_bytes.size());
            d.pos_off = append(img->bytes, pos.data(), pos.size());
            d.rows = (uint16_t)g.rows; d.narrow = (uint16_t)g.narrow;
            groups[w][p].push_back(d);
        }
    }
    std::vector<R1Group> all;
    std::vector<uint16_t> warp_desc;
    for (int w = 0; w < kR1Warps; ++w) {
        warp_desc.push_back((uint16_t)all.size());
        for (int p = 0; p < 2; ++p) { warp_desc.push_back((uint16_t)groups[w][p].size()); all.insert(all.end(), groups[w][p].begin(), groups[w][p].end()); }
        warp_desc.push_back(0);
    }
    R1Op d{};
    d.n_rows = (uint16_t)n_rows; d.units = (uint16_t)s.units; d.unit0 = (uint32_t)s.unit0; d.partials = (uint32_t)at;
    d.rows_off = append(img->bytes, rows.data(), n_rows);
    d.groups_off = append(img->bytes, all.data(), all.size());
    d.warp_off = append(img->bytes, warp_desc.data(), warp_desc.size());
    std::memcpy(img->bytes.data() + op * sizeof(R1Op), &d, sizeof d);
    return CSB_OK;
}

// Contiguous ranges of units, at most `parts` of them, of about equal cost; cuts at multiples of `grain`.
std::vector<int> cut_units(const std::vector<double>& cost, int parts, int grain, int max_units) {
    const int n = (int)cost.size();
    std::vector<double> atom;
    for (int u = 0; u < n; ++u) { if (u % grain == 0) atom.push_back(0); atom.back() += cost[u]; }
    const int na = (int)atom.size(), max_atoms = std::max(1, max_units / grain);
    auto pack = [&](double T, std::vector<int>* cut) {
        int used = 1, start = 0;
        double cur = 0;
        if (cut) cut->assign(1, 0);
        for (int u = 0; u < na; ++u) {
            if (u > start && (cur + atom[u] > T || u - start >= max_atoms)) { if (cut) cut->push_back(u * grain); start = u; cur = 0; ++used; }
            cur += atom[u];
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

std::vector<double> row_weights(const csb_matrix* A) {
    std::vector<double> w((size_t)A->rows, 0.0);
    for (int64_t b = 0; b < A->nblk; ++b) {
        const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
        const double chunks = (A->n[b] + 7) / 8;
        for (int r = 0; r < A->m[b]; ++r) w[(b / A->nbc) * A->block_r + ri[r]] += chunks;
    }
    return w;
}

}  // namespace

int plan_rnn1_host(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, int n_ctas,
                   R1HostPlan* out) {
    *out = R1HostPlan{};
    const int G = r1_gates(cell, 0) + (cell == kR1GruRb ? 1 : 0);
    for (int l = 0; l < L; ++l) if (in_size[l] >= 65535 || S >= 65535 || H >= 65535) return 1;
    // ---- CTAs per layer in proportion to the weights
    std::vector<std::vector<double>> unit_cost(L), proj_cost(L);
    std::vector<double> layer_cost(L, 0.0);
    for (int l = 0; l < L; ++l) {
        const std::vector<double> w = row_weights(W[l]);
        unit_cost[l].assign(H, 4.0);                         // the gate arithmetic of a unit
        for (int g = 0; g < G; ++g) for (int u = 0; u < H; ++u) unit_cost[l][u] += w[(size_t)g * H + u];
        if (cell == kR1Lstmp) { proj_cost[l] = row_weights(Wp[l]); for (double& c : proj_cost[l]) c += 2.0; }
        for (double c : unit_cost[l]) layer_cost[l] += c;
        for (double c : proj_cost[l]) layer_cost[l] += c;
    }
    if (n_ctas < L) return 1;
    std::vector<int> per(L, 1);
    for (int used = L; used < n_ctas; ++used) {              // the next CTA goes to the layer with the most work per CTA
        int best = 0;
        for (int l = 1; l < L; ++l) if (layer_cost[l] / per[l] > layer_cost[best] / per[best]) best = l;
        ++per[best];
    }
    // ---- unit ranges: the granularity with the shortest longest CTA
    const int wide = r1_wide(BT);
    auto best_cut = [&](const csb_matrix* A, const std::vector<double>& cost, int parts, int gates, int64_t stride, int split) {
        std::vector<int> best;
        double best_cost = 0;
        for (int grain = 1; grain <= A->block_r; grain = grain == 1 ? std::max(2, A->block_r / 8) : grain * 2) {
            if (grain > 1 && A->block_r % grain) continue;
            const std::vector<int> cut = cut_units(cost, parts, grain, kR1MaxUnits);
            if ((int)cut.size() - 1 > parts) continue;
            double worst = 0;
            for (size_t i = 0; i + 1 < cut.size(); ++i) worst = std::max(worst, range_cost({A, 0, stride, gates, cut[i], cut[i + 1] - cut[i], split}, wide));
            if (best.empty() || worst < best_cost) { best = cut; best_cost = worst; }
        }
        return best;
    };
    struct Job { int layer, u0, units, p0, punits; };
    std::vector<Job> jobs;
    for (int l = 0; l < L; ++l) {
        const std::vector<int> cu = best_cut(W[l], unit_cost[l], per[l], G, H, in_size[l]);
        std::vector<int> cp;
        if (cell == kR1Lstmp) cp = best_cut(Wp[l], proj_cost[l], per[l], 1, S, 0);
        if (cu.empty() || (cell == kR1Lstmp && cp.empty())) return 1;
        const int n = std::max((int)cu.size(), (int)cp.size()) - 1;
        for (int i = 0; i < n; ++i) {
            Job j{l, 0, 0, 0, 0};
            if (i + 1 < (int)cu.size()) { j.u0 = cu[i]; j.units = cu[i + 1] - cu[i]; }
            if (i + 1 < (int)cp.size()) { j.p0 = cp[i]; j.punits = cp[i + 1] - cp[i]; }
            jobs.push_back(j);
        }
        out->layer_ctas[l] = n;
    }
    // ---- the CTAs' images, on a few host threads
    std::vector<Image> img(jobs.size());
    std::atomic<int> next{0}, status{CSB_OK};
    auto work = [&]() {
        for (int c; status.load() == CSB_OK && (c = next.fetch_add(1)) < (int)jobs.size();) {
            int rc = CSB_OK;
            try {
                const Job& j = jobs[c];
                Image& I = img[c];
                I.bytes.assign(sizeof(R1Header), 0);
                const int zero[2] = {in_size[j.layer], S};
                rc = emit_op({W[j.layer], 0, H, r1_gates(cell, 0), j.u0, j.units, in_size[j.layer]}, zero, 0, BT, &I);
                if (rc == CSB_OK && cell == kR1GruRb) rc = emit_op({W[j.layer], 2 * (int64_t)H, H, 1, j.u0, j.units, in_size[j.layer]}, zero, 1, BT, &I);
                if (rc == CSB_OK && cell == kR1Lstmp) {
                    const int zero_m[2] = {0, H};
                    rc = emit_op({Wp[j.layer], 0, S, 1, j.p0, j.punits, 0}, zero_m, 1, BT, &I);
                }
            } catch (const std::bad_alloc&) { rc = CSB_ERR_ALLOC; }
            if (rc != CSB_OK) status.store(rc);
        }
    };
    run_on_threads((int)std::min<size_t>(8, std::max<size_t>(1, jobs.size() / 8)), work);
    if (status.load() == CSB_ERR_ALLOC) throw std::bad_alloc();
    if (status.load() != CSB_OK) return status.load();
    // ---- exchange words: three elements each (unit by unit, the batch columns of a unit side by side), CTA by CTA
    size_t base = 0, sum = 0;
    const int last = r1_ops(cell) - 1;
    if ((size_t)std::max(H, S) * BT >= (1u << 24)) return 1;
    for (size_t c = 0; c < jobs.size(); ++c) {
        const Job& j = jobs[c];
        R1Header* h = reinterpret_cast<R1Header*>(img[c].bytes.data());
        for (int op = 0; op <= last; ++op) {
            std::vector<uint32_t>& map = out->wmap[op == last ? 0 : 1][j.layer];   // the last product of a step makes the state
            h->op[op].word0 = (uint32_t)map.size();
            const bool proj = cell == kR1Lstmp && op == 1;
            const int e0 = (proj ? j.p0 : j.u0) * BT, n = (proj ? j.punits : j.units) * BT;
            for (int e = 0; e < n; e += 3) map.push_back((uint32_t)(e0 + e) | ((uint32_t)std::min(3, n - e) << 24));
            out->max_units = std::max(out->max_units, (size_t)(proj ? j.punits : j.units));
            out->max_partials[op] = std::max(out->max_partials[op], img[c].partials[op]);
        }
        img[c].bytes.resize(pad_to(img[c].bytes.size(), 128), 0);
        out->ctas.push_back({(uint32_t)(base / 16), (uint32_t)img[c].bytes.size(), j.layer, 0});
        base += img[c].bytes.size();
        sum += img[c].bytes.size();
        out->max_bytes = std::max(out->max_bytes, img[c].bytes.size());
        out->max_rows = std::max(out->max_rows, img[c].rows);
    }
    out->balance = out->max_bytes ? (double)sum / jobs.size() / out->max_bytes : 1.0;
    out->bytes.resize(base);
    base = 0;
    for (Image& i : img) { std::memcpy(out->bytes.data() + base, i.bytes.data(), i.bytes.size()); base += i.bytes.size(); std::vector<uint8_t>().swap(i.bytes); }
    return CSB_OK;
}

}  // namespace csb
