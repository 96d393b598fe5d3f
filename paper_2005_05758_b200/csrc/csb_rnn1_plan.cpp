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

// One product of a CTA before anything is emitted: its tasks and groups, where the partial sums lie, and how long it gets.
struct GroupRef { int part, narrow, rows, warp; size_t from; };
struct OpLayout {
    std::vector<Task> tasks[2][2];             // [part][narrow], longest first
    std::vector<uint32_t> count[2], first[2];  // partial sums of a row and part: how many, where
    std::vector<R1Row> rows;
    std::vector<GroupRef> groups;              // in the order in which they are emitted
    size_t n_rows = 0, partials = 0, bytes = 0;
};
struct Image { std::vector<uint8_t> bytes; OpLayout op[2]; };

// Returns 1 when the product does not fit the layout.
int lay_out_op(const OpSource& s, int BT, OpLayout* o) {
    const int wide = r1_wide(BT), vs = val_size(s.A->val_dtype);
    const size_t n_rows = o->n_rows = (size_t)s.gates * s.units;
    // ---- tasks: rows at most so many that there is about one group for every warp
    for (int p = 0; p < 2; ++p) {
        int limit = kR1MaxRows;
        for (;; limit = std::max(1, limit / 2)) {
            for (auto& v : o->tasks[p]) v.clear();
            o->count[p].assign(n_rows, 0);
            for_pieces(s, [&](int part, int64_t b, int ra, int rz, int k0, int k1, int row_base, int col_base) {
                if (part != p) return;
                const int splits = (rz - ra + limit - 1) / limit;
                for (int k = k0; k < k1; k += wide) {
                    const int ke = std::min(k1, k + wide);
                    for (int i = 0; i < splits; ++i) {
                        const int x = ra + (rz - ra) * i / splits, y = ra + (rz - ra) * (i + 1) / splits;
                        o->tasks[p][ke - k <= wide / 2].push_back({s.A, b, k, ke, x, y, row_base, col_base});
                    }
                    for (int r = ra; r < rz; ++r) ++o->count[p][row_base + s.A->row_idx[s.A->ridx_off[b] + r]];
                }
            });
            // halving the rows must not make more groups than there are warps
            const size_t groups = (o->tasks[p][0].size() + 31) / 32 + (o->tasks[p][1].size() + 31) / 32;
            if (limit == 1 || groups * 2 > (size_t)kR1Warps) break;
        }
    }
    // ---- places of the partial sums: row by row, input part then recurrent part, in quads; then one per lane for idle lanes
    o->rows.assign(std::max<size_t>(n_rows, 1), R1Row{});
    size_t at = 0;
    for (auto& f : o->first) f.assign(n_rows, 0);
    for (size_t r = 0; r < n_rows; ++r)
        for (int p = 0; p < 2; ++p) {
            const size_t q = (o->count[p][r] + 3) / 4;
            o->rows[r].base[p] = (uint16_t)(at / 4); o->rows[r].quads[p] = (uint16_t)q;
            o->first[p][r] = (uint32_t)at;
            at += 4 * q;
        }
    at += 32;
    if (at > 65535) return 1;
    o->partials = at;
    // ---- groups: 32 tasks of about the same number of rows, longest first to the warp with the least work
    double load[kR1Warps] = {};
    for (int p = 0; p < 2; ++p) {
        std::vector<GroupRef> order;
        for (int nw = 0; nw < 2; ++nw) {
            std::vector<Task>& v = o->tasks[p][nw];
            std::stable_sort(v.begin(), v.end(), [](const Task& a, const Task& b) { return a.r1 - a.r0 > b.r1 - b.r0; });
            for (size_t i = 0; i < v.size(); i += 32) order.push_back({p, nw, v[i].r1 - v[i].r0, 0, i});
        }
        std::stable_sort(order.begin(), order.end(), [](const GroupRef& a, const GroupRef& b) { return a.rows > b.rows; });
        double part_load[kR1Warps] = {};
        for (GroupRef& g : order) {
            for (int i = 1; i < kR1Warps; ++i) if (part_load[i] < part_load[g.warp] || (part_load[i] == part_load[g.warp] && load[i] < load[g.warp])) g.warp = i;
            const double cost = kTaskCost + kRowCost * g.rows;
            part_load[g.warp] += cost; load[g.warp] += cost;
            const size_t width = g.narrow ? wide / 2 : wide;
            o->bytes += 64 * width + (size_t)g.rows * 32 * width * vs + (size_t)((g.rows + 1) / 2) * 128;
        }
        o->groups.insert(o->groups.end(), order.begin(), order.end());
    }
    o->bytes += pad_to(n_rows * sizeof(R1Row), 16) + o->groups.size() * sizeof(R1Group) + (size_t)kR1Warps * 8;
    return CSB_OK;
}

// Lays one product out behind the image.
void emit_op(const OpSource& s, const OpLayout& o, const int zero[2], int op, int BT, std::vector<uint8_t>& out) {
    const int wide = r1_wide(BT), vs = val_size(s.A->val_dtype);
    // lanes that share a pass over the banks, and the banks (in units of BT floats) they must keep apart
    const int pass = BT == 1 ? 32 : 8, banks = std::max(32 / BT, 4);
    const size_t idle = o.partials - 32;
    std::vector<std::vector<uint16_t>> free_places[2];
    for (int p = 0; p < 2; ++p) {
        free_places[p].resize(o.n_rows);
        for (size_t r = 0; r < o.n_rows; ++r) for (uint32_t i = 0; i < o.count[p][r]; ++i) free_places[p][r].push_back((uint16_t)(o.first[p][r] + i));
    }
    std::vector<R1Group> groups[kR1Warps][2];
    for (const GroupRef& g : o.groups) {
        const int p = g.part;
        const std::vector<Task>& v = o.tasks[p][g.narrow];
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
        d.cols_off = append(out, cols.data(), cols.size());
        d.w_off = append(out, w_bytes.data(), w_bytes.size());
        d.pos_off = append(out, pos.data(), pos.size());
        d.rows = (uint16_t)g.rows; d.narrow = (uint16_t)g.narrow;
        groups[g.warp][p].push_back(d);
    }
    std::vector<R1Group> all;
    std::vector<uint16_t> warp_desc;
    for (int w = 0; w < kR1Warps; ++w) {
        warp_desc.push_back((uint16_t)all.size());
        for (int p = 0; p < 2; ++p) { warp_desc.push_back((uint16_t)groups[w][p].size()); all.insert(all.end(), groups[w][p].begin(), groups[w][p].end()); }
        warp_desc.push_back(0);
    }
    R1Op d{};
    d.n_rows = (uint16_t)o.n_rows; d.units = (uint16_t)s.units; d.unit0 = (uint32_t)s.unit0; d.partials = (uint32_t)o.partials;
    d.rows_off = append(out, o.rows.data(), o.n_rows);
    d.groups_off = append(out, all.data(), all.size());
    d.warp_off = append(out, warp_desc.data(), warp_desc.size());
    std::memcpy(out.data() + op * sizeof(R1Op), &d, sizeof d);
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

R1Carve::R1Carve(const R1HostPlan& P, int cell, int max_in, int H, int S, int BT) {
    size_t at = P.max_bytes;
    auto room = [&](size_t floats) { const size_t o = at; at = (at + floats * 4 + 15) & ~(size_t)15; return (uint32_t)o; };
    for (uint32_t& v : vu) v = room((size_t)(max_in + 1) * BT);
    vr = room((size_t)(S + 1) * BT); vm = room(r1_ops(cell) == 2 ? (size_t)(H + 1) * BT : 0);
    for (int op = 0; op < 2; ++op) part[op] = room(P.max_partials[op] * BT);
    z[0] = room(4 * P.max_units * BT); z[1] = room(r1_ops(cell) == 2 ? P.max_units * BT : 0);
    cs = room(P.max_units * BT); bias0 = room(4 * P.max_units); bias1 = room(P.max_units);
    misc = room(4);
    total = at;
}

int plan_rnn1_host(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int BT, int n_ctas,
                   size_t smem_limit, R1HostPlan* out) {
    *out = R1HostPlan{};
    // ---- What the weights take at least, whichever way they are dealt: their chunks' rows (values and a position) and
    // partial sums.  If the CTAs' mean is past the limit already, nothing need be planned (two 2048-unit LSTM layers at
    // 4x: 0.15 ms instead of 67; at 8x, where only the layouts below show it, 4.6 instead of 38).
    {
        const size_t wide = (size_t)r1_wide(BT);
        double least = 0;
        auto add = [&](const csb_matrix* A) {
            for (int64_t b = 0; b < A->nblk; ++b) {
                const size_t n = A->n[b], tail = n % wide, width = n / wide * wide + (tail == 0 ? 0 : tail <= wide / 2 ? wide / 2 : wide);
                least += (double)A->m[b] * (double)(width * val_size(A->val_dtype) + (n + wide - 1) / wide * (2 + 4 * (size_t)BT));
            }
        };
        int max_in = 0;
        for (int l = 0; l < L; ++l) { add(W[l]); if (cell == kR1Lstmp) add(Wp[l]); max_in = std::max(max_in, in_size[l]); }
        if (least / std::max(n_ctas, 1) + (double)R1Carve(*out, cell, max_in, H, S, BT).total > (double)smem_limit) return 1;
    }
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
    struct Cut { const csb_matrix* A; const std::vector<double>* cost; int parts, gates; int64_t stride; int split, grain; std::vector<int> cut; double worst; };
    std::vector<Cut> cuts;                                   // of every matrix, the granularities ascending
    auto add_cuts = [&](const csb_matrix* A, const std::vector<double>& cost, int parts, int gates, int64_t stride, int split) {
        for (int grain = 1; grain <= A->block_r; grain = grain == 1 ? std::max(2, A->block_r / 8) : grain * 2)
            if (grain == 1 || A->block_r % grain == 0) cuts.push_back({A, &cost, parts, gates, stride, split, grain, {}, 0.0});
    };
    for (int l = 0; l < L; ++l) {
        add_cuts(W[l], unit_cost[l], per[l], G, H, in_size[l]);
        if (cell == kR1Lstmp) add_cuts(Wp[l], proj_cost[l], per[l], 1, S, 0);
    }
    std::atomic<int> next{0}, status{CSB_OK};
    // items of work taken from a counter by a few host threads
    auto in_parallel = [&](int n, auto&& item) {
        next.store(0);
        run_on_threads(std::max(1, std::min(8, n / 2)), [&]() {
            for (int c; status.load() == CSB_OK && (c = next.fetch_add(1)) < n;) {
                int rc;
                try { rc = item(c); } catch (const std::bad_alloc&) { rc = CSB_ERR_ALLOC; }
                if (rc != CSB_OK) status.store(rc);
            }
        });
        if (status.load() == CSB_ERR_ALLOC) throw std::bad_alloc();
        return status.load();
    };
    in_parallel((int)cuts.size(), [&](int i) {
        Cut& c = cuts[i];
        c.cut = cut_units(*c.cost, c.parts, c.grain, kR1MaxUnits);
        if ((int)c.cut.size() - 1 > c.parts) { c.cut.clear(); return (int)CSB_OK; }
        for (size_t k = 0; k + 1 < c.cut.size(); ++k)
            c.worst = std::max(c.worst, range_cost({c.A, 0, c.stride, c.gates, c.cut[k], c.cut[k + 1] - c.cut[k], c.split}, wide));
        return (int)CSB_OK;
    });
    auto best_cut = [&](const csb_matrix* A, const std::vector<double>& cost) {
        const Cut* best = nullptr;
        for (const Cut& c : cuts) if (c.A == A && c.cost == &cost && !c.cut.empty() && (!best || c.worst < best->worst)) best = &c;
        return best ? best->cut : std::vector<int>();
    };
    struct Job { int layer, u0, units, p0, punits; };
    std::vector<Job> jobs;
    for (int l = 0; l < L; ++l) {
        const std::vector<int> cu = best_cut(W[l], unit_cost[l]);
        std::vector<int> cp;
        if (cell == kR1Lstmp) cp = best_cut(Wp[l], proj_cost[l]);
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
    // ---- the CTAs' layouts; what they take of shared memory; only then their images
    std::vector<Image> img(jobs.size());
    auto source = [&](const Job& j, int op) -> OpSource {
        if (op == 0) return {W[j.layer], 0, H, r1_gates(cell, 0), j.u0, j.units, in_size[j.layer]};
        if (cell == kR1GruRb) return {W[j.layer], 2 * (int64_t)H, H, 1, j.u0, j.units, in_size[j.layer]};
        return {Wp[j.layer], 0, S, 1, j.p0, j.punits, 0};
    };
    const int ops = r1_ops(cell);
    if (in_parallel((int)jobs.size(), [&](int c) {
            int rc = CSB_OK;
            for (int op = 0; op < ops && rc == CSB_OK; ++op) rc = lay_out_op(source(jobs[c], op), BT, &img[c].op[op]);
            return rc;
        }) != CSB_OK) return status.load();
    for (size_t c = 0; c < jobs.size(); ++c) {
        size_t bytes = sizeof(R1Header);
        for (int op = 0; op < ops; ++op) {
            bytes += img[c].op[op].bytes;
            out->max_partials[op] = std::max(out->max_partials[op], img[c].op[op].partials);
        }
        out->max_bytes = std::max(out->max_bytes, pad_to(bytes, 128));
        out->max_units = std::max(out->max_units, (size_t)std::max(jobs[c].units, cell == kR1Lstmp ? jobs[c].punits : 0));
    }
    int max_in = 0;
    for (int l = 0; l < L; ++l) max_in = std::max(max_in, in_size[l]);
    if (R1Carve(*out, cell, max_in, H, S, BT).total > smem_limit) return 1;
    if (in_parallel((int)jobs.size(), [&](int c) {
            const Job& j = jobs[c];
            std::vector<uint8_t>& bytes = img[c].bytes;
            bytes.reserve(out->max_bytes);
            bytes.assign(sizeof(R1Header), 0);
            const int zero[2] = {in_size[j.layer], S}, zero_m[2] = {0, H};
            for (int op = 0; op < ops; ++op) emit_op(source(j, op), img[c].op[op], cell == kR1Lstmp && op == 1 ? zero_m : zero, op, BT, bytes);
            return (int)CSB_OK;
        }) != CSB_OK) return status.load();
    // ---- exchange words: three elements each (unit by unit, the batch columns of a unit side by side), CTA by CTA
    size_t base = 0;
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
        }
        img[c].bytes.resize(pad_to(img[c].bytes.size(), 128), 0);
        out->ctas.push_back({(uint32_t)(base / 16), (uint32_t)img[c].bytes.size(), j.layer, 0});
        base += img[c].bytes.size();
    }
    out->bytes.reserve(base);
    for (Image& i : img) { out->bytes.insert(out->bytes.end(), i.bytes.begin(), i.bytes.end()); std::vector<uint8_t>().swap(i.bytes); }
    return CSB_OK;
}

}  // namespace csb
