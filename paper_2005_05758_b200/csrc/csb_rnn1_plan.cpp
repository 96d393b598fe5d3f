// Planner of the batch-1 time loop (layout: csb_rnn1.hpp).
//
// Hidden units are cut into one contiguous range per CTA, the CTAs dealt to the layers in proportion
// to their weights.  Inside a CTA every row gets a number of threads in proportion to its slots; the
// order of a thread's slots is free (fp32 sums of one thread in any order), and it is chosen so that
// the eight lanes of a quarter-warp, whose 16-byte reads of gathered inputs share one pass over the
// shared-memory banks, fall into different bank groups or onto the same address.
#include <algorithm>
#include <atomic>
#include <new>
#include <system_error>
#include <thread>

#include "csb_rnn1.hpp"

namespace csb {

static inline size_t pad_to(size_t v, size_t a) { return (v + a - 1) / a * a; }

namespace {

struct Slot { const uint8_t* v; uint16_t place; uint8_t cnt; };      // `cnt` values at v, gathered inputs at 16 * place bytes
struct Rows { std::vector<std::vector<Slot>> part[2]; };              // [part][row] slots

struct OpSource { const csb_matrix* A; int64_t row0, gate_stride; int gates, unit0, units, split; };   // columns < split: input part

// Collects the rows of one product and the lists of columns it gathers.
void collect(const OpSource& s, Rows* R, std::vector<uint16_t>* gather, const int zero[2]) {
    const csb_matrix* A = s.A;
    const int BR = A->block_r, BC = A->block_c, vs = val_size(A->val_dtype);
    for (int p = 0; p < 2; ++p) {
        R->part[p].assign((size_t)s.gates * s.units, {});
        gather[p].assign(4, (uint16_t)zero[p]);            // place 0 holds zeros: where lanes without work read
    }
    for (int g = 0; g < s.gates; ++g) {
        const int64_t lo = s.row0 + g * s.gate_stride + s.unit0, hi = lo + s.units;
        for (int64_t bi = lo / BR; bi * BR < hi; ++bi) {
            const int a = (int)std::max<int64_t>(0, lo - bi * BR), z = (int)std::min<int64_t>(BR, hi - bi * BR);
            for (int64_t bj = 0; bj < A->nbc; ++bj) {
                const int64_t b = bi * A->nbc + bj;
                const int m = A->m[b], n = A->n[b];
                if (!m || !n) continue;
                const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
                const uint8_t* ci = A->col_idx.data() + A->cidx_off[b];
                const int ra = (int)(std::lower_bound(ri, ri + m, a) - ri), rz = (int)(std::lower_bound(ri, ri + m, z) - ri);
                if (ra == rz) continue;
                const int64_t c0 = bj * BC;
                const int cut = c0 >= s.split ? 0 : c0 + BC <= s.split ? n : (int)(std::lower_bound(ci, ci + n, (int)(s.split - c0)) - ci);
                for (int p = 0; p < 2; ++p) {
                    const int k0 = p ? cut : 0, k1 = p ? n : cut;
                    if (k0 == k1) continue;
                    const size_t at = gather[p].size();
                    for (int k = k0; k < k1; ++k) gather[p].push_back((uint16_t)(c0 + ci[k] - (p ? s.split : 0)));
                    while (gather[p].size() & 3) gather[p].push_back((uint16_t)zero[p]);
                    for (int r = ra; r < rz; ++r) {
                        const uint8_t* v = A->val.data() + (A->val_off[b] + (uint64_t)r * n) * vs;
                        std::vector<Slot>& list = R->part[p][(size_t)g * s.units + (bi * BR + ri[r] - lo)];
                        for (int k = k0; k < k1; k += 4)
                            list.push_back({v + (size_t)k * vs, (uint16_t)((at + (k - k0)) / 4), (uint8_t)std::min(4, k1 - k)});
                    }
                }
            }
        }
    }
}

// Orders the slots of eight lanes so that in each step they meet different bank groups (16 bytes of
// the 128 that one pass serves) or the same address, as far as a greedy choice finds it: the lane
// with the fewest free choices goes first and takes from the bank group it has most of.
void order_quarter(std::vector<Slot>* lane) {
    std::vector<Slot> out[8];
    size_t steps = 0;
    for (int l = 0; l < 8; ++l) steps = std::max(steps, lane[l].size());
    for (size_t st = 0; st < steps; ++st) {
        int used[8];                           // place read in this step per bank group, -1: none
        std::fill(used, used + 8, -1);
        bool done[8] = {};
        for (int turn = 0; turn < 8; ++turn) {
            int best_l = -1, best_free = 1 << 30;
            size_t best_k = 0;
            bool best_ok = false;
            for (int l = 0; l < 8; ++l) {
                if (done[l] || lane[l].empty()) continue;
                int have[8] = {}, free_slots = 0;
                for (const Slot& s : lane[l]) ++have[s.place & 7];
                size_t pick = 0;
                int score = -1;
                for (size_t k = 0; k < lane[l].size(); ++k) {
                    const int p = lane[l][k].place, g = p & 7;
                    const bool ok = used[g] < 0 || used[g] == p;
                    free_slots += ok;
                    const int sc = ok ? (used[g] == p ? 1000 : 0) + have[g] + 1 : 0;
                    if (sc > score) { score = sc; pick = k; }
                }
                // a lane that is ahead of the others in length must not fall behind: longest list breaks ties
                const int key = free_slots * 64 - (int)std::min<size_t>(lane[l].size(), 63);
                if (key < best_free) { best_free = key; best_l = l; best_k = pick; best_ok = score > 0; }
            }
            if (best_l < 0) break;
            const Slot s = lane[best_l][best_k];
            if (best_ok && used[s.place & 7] < 0) used[s.place & 7] = s.place;
            out[best_l].push_back(s);
            lane[best_l][best_k] = lane[best_l].back();
            lane[best_l].pop_back();
            done[best_l] = true;
        }
    }
    for (int l = 0; l < 8; ++l) lane[l].swap(out[l]);
}

struct Image { std::vector<uint8_t> bytes, reg[2]; std::vector<uint32_t> reg_places[2]; size_t smem_bytes = 0; size_t xg[2][2] = {{0, 0}, {0, 0}}; };

template <typename V>
uint32_t append(std::vector<uint8_t>& b, const V* p, size_t n) {
    b.resize(pad_to(b.size(), 16), 0);
    const uint32_t at = (uint32_t)b.size();
    b.resize(at + pad_to(n * sizeof(V), 16), 0);
    if (n) std::memcpy(b.data() + at, p, n * sizeof(V));
    return at;
}

// Lays one product out behind the image; returns 1 when it does not fit the layout.
int emit_op(const OpSource& s, const int zero[2], int op, size_t reg_pairs, Image* img) {
    Rows R;
    std::vector<uint16_t> gather[2];
    collect(s, &R, gather, zero);
    const size_t n_rows = (size_t)s.gates * s.units;
    const int vs = val_size(s.A->val_dtype);
    // threads per row: the smallest K with sum over rows of ceil(slots / K) <= threads
    std::vector<uint32_t> slots(n_rows), rows(n_rows);
    size_t total = 0, longest = 0;
    for (size_t r = 0; r < n_rows; ++r) {
        slots[r] = (uint32_t)(R.part[0][r].size() + R.part[1][r].size());
        total += slots[r];
        longest = std::max<size_t>(longest, slots[r]);
    }
    auto threads_for = [&](size_t K) { size_t n = 0; for (uint32_t v : slots) n += (v + K - 1) / K; return n; };
    size_t lo = std::max<size_t>(1, total / kR1Threads), hi = std::max<size_t>(longest, 1);
    if (threads_for(hi) > (size_t)kR1Threads) return 1;      // more rows than threads
    while (lo < hi) { const size_t mid = (lo + hi) / 2; if (threads_for(mid) <= (size_t)kR1Threads) hi = mid; else lo = mid + 1; }
    const size_t K = hi;
    std::vector<Slot> lists[2][kR1Threads];
    uint32_t t = 0;
    for (size_t r = 0; r < n_rows; ++r) {
        const uint32_t k = (uint32_t)((slots[r] + K - 1) / K);
        rows[r] = t | (k << 16);
        for (int p = 0; p < 2; ++p) {
            const std::vector<Slot>& src = R.part[p][r];
            for (uint32_t j = 0; j < k; ++j) lists[p][t + j].assign(src.begin() + src.size() * j / k, src.begin() + src.size() * (j + 1) / k);
        }
        t += k;
    }
    for (int p = 0; p < 2; ++p)
        for (int q = 0; q < kR1Threads; q += 8) order_quarter(&lists[p][q]);
    // emit, warp by warp
    std::vector<uint8_t> w, o;
    struct WarpDesc { uint32_t w16, o, n_in, n_rec; } wd[kR1Warps];
    auto emit_pair = [&](int p, int wp, size_t it, uint8_t* wdst, uint8_t* odst) {
        for (int h = 0; h < 2; ++h)
            for (int l = 0; l < 32; ++l) {
                const std::vector<Slot>& list = lists[p][wp * 32 + l];
                const size_t k = 2 * it + h;
                uint16_t bytes = 0;
                if (k < list.size()) {
                    bytes = (uint16_t)(list[k].place * 16u);
                    // fp16: both slots of a pair in 16 bytes per lane; fp32: 16 bytes per slot, [slot][lane]
                    std::memcpy(wdst + (vs == 2 ? (size_t)l * 16 + h * 8 : (size_t)(h * 32 + l) * 16), list[k].v, (size_t)list[k].cnt * vs);
                }
                std::memcpy(odst + (size_t)l * 4 + h * 2, &bytes, 2);
            }
    };
    const size_t pair_bytes = 32 * 8 * vs;
    img->reg[op].assign(kR1Warps * reg_pairs * pair_bytes, 0);
    img->reg_places[op].assign(kR1Warps * reg_pairs * 32, 0);
    for (int wp = 0; wp < kR1Warps; ++wp) {
        wd[wp].w16 = (uint32_t)(w.size() / 16); wd[wp].o = (uint32_t)o.size();
        for (int p = 0; p < 2; ++p) {
            size_t most = 0;
            for (int l = 0; l < 32; ++l) most = std::max(most, lists[p][wp * 32 + l].size());
            const size_t pairs = (most + 1) / 2, first = p ? std::min(reg_pairs, pairs) : 0;
            for (size_t it = 0; it < first; ++it)
                emit_pair(p, wp, it, img->reg[op].data() + (wp * reg_pairs + it) * pair_bytes, (uint8_t*)(img->reg_places[op].data() + (wp * reg_pairs + it) * 32));
            (p ? wd[wp].n_rec : wd[wp].n_in) = (uint32_t)(pairs - first);
            for (size_t it = first; it < pairs; ++it) {
                const size_t wb = w.size(), ob = o.size();
                w.resize(wb + pair_bytes, 0);
                o.resize(ob + 32 * 4, 0);
                emit_pair(p, wp, it, w.data() + wb, o.data() + ob);
            }
        }
    }
    for (int p = 0; p < 2; ++p) if (gather[p].size() * 4 > 65536) return 1;      // places are 16-bit byte offsets
    R1Op d{};
    d.n_rows = (uint16_t)n_rows; d.units = (uint16_t)s.units; d.unit0 = (uint32_t)s.unit0;
    d.rows_off = append(img->bytes, rows.data(), rows.size());
    const uint32_t w_at = append(img->bytes, w.data(), w.size()), o_at = append(img->bytes, o.data(), o.size());
    for (WarpDesc& x : wd) { x.w16 += w_at / 16; x.o += o_at; }
    d.warp_off = append(img->bytes, wd, kR1Warps);
    for (int p = 0; p < 2; ++p) {
        d.gather_off[p] = append(img->bytes, gather[p].data(), gather[p].size());
        d.quads[p] = (uint16_t)(gather[p].size() / 4);
        img->xg[op][p] = gather[p].size();
    }
    std::memcpy(img->bytes.data() + op * sizeof(R1Op), &d, sizeof d);
    return CSB_OK;
}

// Contiguous ranges of units, `parts` of them, of about equal cost.
std::vector<int> cut_units(const std::vector<double>& cost, int parts, int max_units) {
    const int n = (int)cost.size();
    parts = std::max(1, std::min(parts, n));
    auto pack = [&](double T, std::vector<int>* cut) {
        int used = 1, start = 0;
        double cur = 0;
        if (cut) cut->assign(1, 0);
        for (int u = 0; u < n; ++u) {
            if (u > start && (cur + cost[u] > T || u - start >= max_units)) { if (cut) cut->push_back(u); start = u; cur = 0; ++used; }
            cur += cost[u];
        }
        if (cut) cut->push_back(n);
        return used;
    };
    double lo = 0, hi = 1;
    for (double c : cost) hi += c;
    for (int i = 0; i < 50; ++i) { const double mid = 0.5 * (lo + hi); if (pack(mid, nullptr) <= parts) hi = mid; else lo = mid; }
    std::vector<int> cut;
    pack(hi, &cut);
    return cut;
}

std::vector<double> row_weights(const csb_matrix* A) {
    std::vector<double> w((size_t)A->rows, 0.0);
    for (int64_t b = 0; b < A->nblk; ++b) {
        const uint8_t* ri = A->row_idx.data() + A->ridx_off[b];
        const double slots = (A->n[b] + 3) / 4;
        for (int r = 0; r < A->m[b]; ++r) w[(b / A->nbc) * A->block_r + ri[r]] += slots;
    }
    return w;
}

}  // namespace

int plan_rnn1_host(int cell, int L, const csb_matrix* const* W, const csb_matrix* const* Wp, const int* in_size, int H, int S, int n_ctas,
                   R1HostPlan* out) {
    *out = R1HostPlan{};
    const int G = r1_gates(cell, 0) + (cell == kR1GruRb ? 1 : 0);
    for (int l = 0; l < L; ++l) if (in_size[l] >= 65535 || S >= 65535 || H >= 65535) return 1;
    // ---- CTAs per layer in proportion to the slots, unit ranges of equal cost inside a layer
    std::vector<std::vector<double>> unit_cost(L), proj_cost(L);
    std::vector<double> layer_cost(L, 0.0);
    double total = 0;
    for (int l = 0; l < L; ++l) {
        const std::vector<double> w = row_weights(W[l]);
        unit_cost[l].assign(H, 8.0);                         // the gate arithmetic of a unit
        for (int g = 0; g < G; ++g) for (int u = 0; u < H; ++u) unit_cost[l][u] += w[(size_t)g * H + u];
        if (cell == kR1Lstmp) { proj_cost[l] = row_weights(Wp[l]); for (double& c : proj_cost[l]) c += 4.0; }
        for (double c : unit_cost[l]) layer_cost[l] += c;
        for (double c : proj_cost[l]) layer_cost[l] += c;
        total += layer_cost[l];
    }
    if (n_ctas < L) return 1;
    std::vector<int> per(L, 1);
    for (int used = L; used < n_ctas; ++used) {              // the next CTA goes to the layer with the most work per CTA
        int best = 0;
        for (int l = 1; l < L; ++l) if (layer_cost[l] / per[l] > layer_cost[best] / per[best]) best = l;
        ++per[best];
    }
    struct Job { int layer, u0, units, p0, punits; };
    std::vector<Job> jobs;
    double worst = 0;
    for (int l = 0; l < L; ++l) {
        const std::vector<int> cu = cut_units(unit_cost[l], per[l], kR1MaxUnits);
        std::vector<int> cp;
        if (cell == kR1Lstmp) cp = cut_units(proj_cost[l], std::min<int>(per[l], std::max<int>((int)cu.size() - 1, 1)), kR1MaxUnits);
        const int n = std::max((int)cu.size(), (int)cp.size()) - 1;
        if (n > per[l]) return 1;                            // more units than the CTAs' gate lanes take
        for (int i = 0; i < n; ++i) {
            Job j{l, 0, 0, 0, 0};
            if (i + 1 < (int)cu.size()) { j.u0 = cu[i]; j.units = cu[i + 1] - cu[i]; }
            if (i + 1 < (int)cp.size()) { j.p0 = cp[i]; j.punits = cp[i + 1] - cp[i]; }
            double c = 0;
            for (int u = j.u0; u < j.u0 + j.units; ++u) c += unit_cost[l][u];
            for (int u = j.p0; u < j.p0 + j.punits; ++u) c += proj_cost[l][u];
            worst = std::max(worst, c);
            jobs.push_back(j);
        }
        out->layer_ctas[l] = n;
    }
    out->balance = worst > 0 ? total / jobs.size() / worst : 1.0;
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
                const OpSource a{W[j.layer], 0, H, r1_gates(cell, 0), j.u0, j.units, in_size[j.layer]};
                const size_t regs = r1_reg_pairs(cell, val_size(W[j.layer]->val_dtype));
                rc = emit_op(a, zero, 0, regs, &I);
                if (rc == CSB_OK && cell == kR1GruRb) {
                    const OpSource b{W[j.layer], 2 * (int64_t)H, H, 1, j.u0, j.units, in_size[j.layer]};
                    rc = emit_op(b, zero, 1, regs, &I);
                }
                if (rc == CSB_OK && cell == kR1Lstmp) {
                    const int zero_m[2] = {0, H};
                    const OpSource b{Wp[j.layer], 0, S, 1, j.p0, j.punits, 0};
                    rc = emit_op(b, zero_m, 1, regs, &I);
                }
                if (rc == CSB_OK) {
                    // what stays in registers goes behind what is copied to shared memory
                    I.bytes.resize(pad_to(I.bytes.size(), 16), 0);
                    I.smem_bytes = I.bytes.size();
                    for (int op = 0; op < r1_ops(cell); ++op) {
                        const uint32_t r = append(I.bytes, I.reg[op].data(), I.reg[op].size()), q = append(I.bytes, I.reg_places[op].data(), I.reg_places[op].size());
                        R1Op* d = &reinterpret_cast<R1Header*>(I.bytes.data())->op[op];
                        d->reg_off = r; d->reg_places = q;
                        std::vector<uint8_t>().swap(I.reg[op]);
                        std::vector<uint32_t>().swap(I.reg_places[op]);
                    }
                }
            } catch (const std::bad_alloc&) { rc = CSB_ERR_ALLOC; }
            if (rc != CSB_OK) status.store(rc);
        }
    };
    {
        const unsigned hw = std::thread::hardware_concurrency();
        std::vector<std::thread> pool;
        try { for (unsigned t = 1; t < std::min<unsigned>(hw ? hw : 1, 8) && t < jobs.size() / 8; ++t) pool.emplace_back(work); } catch (const std::system_error&) {}
        work();
        for (auto& t : pool) t.join();
    }
    if (status.load() == CSB_ERR_ALLOC) throw std::bad_alloc();
    if (status.load() != CSB_OK) return status.load();
    // ---- exchange words: three units each, CTA by CTA
    size_t base = 0;
    for (size_t c = 0; c < jobs.size(); ++c) {
        const Job& j = jobs[c];
        R1Header* h = reinterpret_cast<R1Header*>(img[c].bytes.data());
        const int last = r1_ops(cell) - 1;
        for (int op = 0; op <= last; ++op) {
            std::vector<uint32_t>& map = out->wmap[op == last ? 0 : 1][j.layer];   // the last product of a step makes the state
            h->op[op].word0 = (uint32_t)map.size();
            const int u0 = cell == kR1Lstmp && op == 1 ? j.p0 : j.u0, n = cell == kR1Lstmp && op == 1 ? j.punits : j.units;
            for (int u = 0; u < n; u += 3) map.push_back((uint32_t)(u0 + u) | ((uint32_t)std::min(3, n - u) << 16));
            if (map.size() > (size_t)kR1Words * kR1Threads) return 1;
        }
        img[c].bytes.resize(pad_to(img[c].bytes.size(), 128), 0);
        out->ctas.push_back({(uint32_t)(base / 16), (uint32_t)img[c].bytes.size(), (uint32_t)img[c].smem_bytes, j.layer});
        base += img[c].bytes.size();
        out->max_smem = std::max(out->max_smem, img[c].smem_bytes);
        for (int op = 0; op < 2; ++op) for (int p = 0; p < 2; ++p) out->max_xg[op][p] = std::max(out->max_xg[op][p], img[c].xg[op][p]);
    }
    out->bytes.resize(base);
    base = 0;
    for (Image& i : img) { std::memcpy(out->bytes.data() + base, i.bytes.data(), i.bytes.size()); base += i.bytes.size(); std::vector<uint8_t>().swap(i.bytes); }
    return CSB_OK;
}

}  // namespace csb
