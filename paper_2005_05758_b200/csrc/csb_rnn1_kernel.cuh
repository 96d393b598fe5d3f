// Resident time loop of the recurrent cells (LSTM, GRU, LSTMP, Li-GRU, reset-before GRU) for small
// batches, where the matrices leave no room for the lists of csb_rnn_unit_kernel.cuh: one cooperative launch per sequence (Section 2.1 of the paper: per step a CSB product with
// [u_t ; h_{t-1}], then the element-wise gate arithmetic, the c / h "context link" feeding the next step).
//
// A CTA owns a range of hidden units of one layer (csb_rnn1.hpp); its weights stay in shared memory.
// What bounds a step is latency: the exchange of h_t between CTAs, then product, sums and gates, and
// inside the product the traffic of shared memory.  So
//   * a vector crosses CTAs as 16-byte words of three values and the number of their step, written
//     and read with single 16-byte accesses (relaxed, 128-bit atomic): a reader that sees the step
//     it waits for also holds the values.  No fence, no counter, no grid barrier; layers run as a
//     dataflow pipeline.  Step numbers go on from call to call (a word per CTA keeps the count), so
//     nothing is cleared between calls.  A vector stays for 32 steps; every 8 steps a layer checks
//     that the layer above has read what it is about to overwrite;
//   * the product over the input part [u_t] is done while h_{t-1} is on its way, and u_{t+1} is fetched
//     into the other of two buffers meanwhile;
//   * a lane of the product fetches up to 8 inputs through the column indices into registers and
//     multiplies them with the rows of its task one after the other; partial sums go to places of
//     their own, ordered by row.  Measured at 2 x 2048 units, 10x pruned, batch 1: a step takes 4.2 us
//     (6.7 with indices and weights read row by row), of which the two walks are about half;
//   * three barriers a step: inputs complete, partial sums complete, row sums complete.
// LSTMP and the reset-before GRU have a second product in the step (the projection; the candidate's):
// what it reads (o * tanh(c); r * h) crosses the CTAs of the layer in the same way.
//
// Initial states, bias, x, y and final states are read and written in place, so a call is one launch.
#pragma once

#include "csb_rnn_exchange.cuh"
#include "csb_rnn1_args.hpp"

namespace csb {

typedef unsigned __int128 Word;                // three values and a step number
__device__ __forceinline__ Word ld_word(const uint4* p) {
    Word w;
    asm volatile("ld.relaxed.gpu.global.b128 %0, [%1];" : "=q"(w) : "l"(p) : "memory");
    return w;
}
__device__ __forceinline__ void st_word(uint4* p, float a, float b, float c, uint32_t tag) {
    const Word w = (Word)__float_as_uint(a) | ((Word)__float_as_uint(b) << 32) | ((Word)__float_as_uint(c) << 64) | ((Word)tag << 96);
    asm volatile("st.relaxed.gpu.global.b128 [%0], %1;" ::"l"(p), "q"(w) : "memory");
}
__device__ __forceinline__ uint32_t word_tag(Word w) { return (uint32_t)(w >> 96); }
// N consecutive 32-bit words of shared memory.
template <int N> struct Regs { uint32_t v[N]; };
template <int N>
__device__ __forceinline__ Regs<N> ld_regs(const uint8_t* p) {
    Regs<N> r;
    if (N == 1) r.v[0] = *reinterpret_cast<const uint32_t*>(p);
    if (N == 2) { const uint2 t = *reinterpret_cast<const uint2*>(p); r.v[0] = t.x; r.v[N > 1 ? 1 : 0] = t.y; }
#pragma unroll
    for (int i = 0; i + 4 <= N; i += 4) {
        const uint4 t = *reinterpret_cast<const uint4*>(p + 4 * i);
        r.v[i] = t.x; r.v[i + 1 < N ? i + 1 : 0] = t.y; r.v[i + 2 < N ? i + 2 : 0] = t.z; r.v[i + 3 < N ? i + 3 : 0] = t.w;
    }
    return r;
}

// One group of tasks with K columns: inputs into registers, then row after row.
template <typename T, int BT, int K>
__device__ __forceinline__ void walk_group(const uint8_t* img, const R1Group& g, int lane, const float* v, float* partials) {
    constexpr int kWords = K * (int)sizeof(T) / 4;         // weight words of a row
    const Regs<K / 2> c = ld_regs<K / 2>(img + g.cols_off + lane * (K * 2));
    float x[K][BT];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float* p = v + (size_t)((c.v[k / 2] >> (16 * (k & 1))) & 0xffffu) * BT;
        if (BT == 1) x[k][0] = *p;
#pragma unroll
        for (int b = 0; b + 4 <= BT; b += 4) {
            const float4 t = *reinterpret_cast<const float4*>(p + b);
            x[k][b] = t.x; x[k][b + 1 < BT ? b + 1 : 0] = t.y; x[k][b + 2 < BT ? b + 2 : 0] = t.z; x[k][b + 3 < BT ? b + 3 : 0] = t.w;
        }
    }
    const uint8_t* w = img + g.w_off + lane * (kWords == 8 ? 16 : kWords * 4);
    const uint32_t* pos = reinterpret_cast<const uint32_t*>(img + g.pos_off) + lane;
    auto row = [&](const Regs<kWords>& q, uint32_t place) {
        float wf[K];
#pragma unroll
        for (int i = 0; i < kWords; ++i) {
            if (sizeof(T) == 2) { const float2 t = half2_to_float2(q.v[i]); wf[(2 * i) % K] = t.x; wf[(2 * i + 1) % K] = t.y; }
            else wf[i % K] = __uint_as_float(q.v[i]);
        }
        float* out = partials + place * BT;
        if (BT == 1) {
            float2 a = make_float2(wf[0] * x[0][0], wf[1] * x[1][0]);
#pragma unroll
            for (int k = 2; k < K; k += 2) a = fma2(make_float2(wf[k], wf[k + 1]), make_float2(x[k][0], x[k + 1][0]), a);
            *out = a.x + a.y;
        } else {
            float2 a[BT / 2 > 0 ? BT / 2 : 1];
#pragma unroll
            for (int b = 0; b < BT / 2; ++b) a[b] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; ++k)
#pragma unroll
                for (int b = 0; b < BT / 2; ++b) a[b] = fma2(make_float2(wf[k], wf[k]), make_float2(x[k][2 * b], x[k][(2 * b + 1) % BT]), a[b]);
#pragma unroll
            for (int b = 0; b + 1 < BT / 2; b += 2)
                *reinterpret_cast<float4*>(out + 2 * b) = make_float4(a[b].x, a[b].y, a[(b + 1) % (BT / 2 > 0 ? BT / 2 : 1)].x, a[(b + 1) % (BT / 2 > 0 ? BT / 2 : 1)].y);
        }
    };
    auto load = [&](int r) {
        if (kWords == 8) {                                 // fp32, eight columns: [half][lane]
            const Regs<4> lo = ld_regs<4>(w + (size_t)r * 1024), hi = ld_regs<4>(w + (size_t)r * 1024 + 512);
            Regs<kWords> q;
#pragma unroll
            for (int i = 0; i < 4; ++i) { q.v[i % kWords] = lo.v[i]; q.v[(4 + i) % kWords] = hi.v[i]; }
            return q;
        }
        return ld_regs<kWords>(w + (size_t)r * (32 * kWords * 4));
    };
    int r = 0;
    // batch 1, fp16: the next two rows' weights are on their way while two are multiplied (2 x 2048 GRU units, 10x: 4.33
    // to 4.13 us a step, LSTM 4.29 to 4.23; more batch columns have no registers for it)
    if (BT == 1 && sizeof(T) == 2 && g.rows >= 2) {
        uint32_t p = pos[0];
        Regs<kWords> a = load(0), b = load(1);
#pragma unroll 2
        for (; r + 4 <= g.rows; r += 2) {
            const uint32_t pn = pos[(r / 2 + 1) * 32];
            const Regs<kWords> an = load(r + 2), bn = load(r + 3);
            row(a, p & 0xffffu);
            row(b, p >> 16);
            a = an; b = bn; p = pn;
        }
        row(a, p & 0xffffu);
        row(b, p >> 16);
        r += 2;
    }
    for (; r + 2 <= g.rows; r += 2) {
        const uint32_t p = pos[(r / 2) * 32];
        const Regs<kWords> a = load(r), b = load(r + 1);
        row(a, p & 0xffffu);
        row(b, p >> 16);
    }
    if (r < g.rows) row(load(r), pos[(r / 2) * 32] & 0xffffu);
}

// A warp's groups [g0, g0 + n) of one product.
template <typename T, int BT>
__device__ __forceinline__ void walk(const uint8_t* img, const R1Group* groups, int n, int lane, const float* v, float* partials) {
    constexpr int kWide = BT >= 8 ? 4 : 8;                 // r1_wide()
    for (int i = 0; i < n; ++i) {
        const R1Group g = groups[i];
        if (g.narrow) walk_group<T, BT, kWide / 2>(img, g, lane, v, partials);
        else walk_group<T, BT, kWide>(img, g, lane, v, partials);
    }
}

template <typename T, int CELL, int BT>
__global__ void __launch_bounds__(kR1Threads, 1) csb_rnn1_kernel(const __grid_constant__ R1Args a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr int OPS = CELL == kR1Lstmp || CELL == kR1GruRb ? 2 : 1;
    constexpr int G0 = CELL == kR1Lstm || CELL == kR1Lstmp ? 4 : CELL == kR1Gru ? 3 : 2;
    constexpr int kW = BT >= 8 ? 4 : BT >= 4 ? 3 : 2;      // exchange words a thread asks for ahead
    constexpr bool kHasC = CELL == kR1Lstm || CELL == kR1Lstmp;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const R1Cta me = a.ctas[blockIdx.x];
    const int layer = me.layer, below = layer - 1, I = a.in_size[layer], S = a.S, H = a.H, T_ = a.T, B = a.B;
    const uint8_t* img = smem;
    auto f32 = [&](uint32_t off) { return reinterpret_cast<float*>(smem + off); };
    float* vr = f32(a.vr);
    float* vm = f32(a.vm);
    float* cs = f32(a.cs);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + a.misc);
    volatile int* s_ok = reinterpret_cast<volatile int*>(smem + a.misc + 8);

    // ---- weights; initial state; first input.  A staged vector holds BT values per column and ends in zeros.
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
        mbar_expect_tx(bar, me.bytes);
        const uint8_t* src = a.images + (size_t)me.off16 * 16;
        for (uint32_t off = 0; off < me.bytes; off += 16384u) bulk_g2s(smem + off, src + off, min(16384u, me.bytes - off), bar);
        *s_ok = 1;
    }
    auto stage = [&](float* dst, const float* src, int n) {      // [B][n] in global memory
        for (int b = 0; b < BT; ++b)
            for (int i = tid; i < n; i += kR1Threads) dst[i * BT + b] = src && b < B ? __ldg(src + (size_t)b * n + i) : 0.f;
    };
    stage(vr, a.h0 ? a.h0 + (size_t)layer * B * S : nullptr, S);
    if (layer == 0) stage(f32(a.vu[0]), a.x, I);
    if (tid < BT) { vr[S * BT + tid] = 0.f; f32(a.vu[0])[I * BT + tid] = 0.f; f32(a.vu[1])[I * BT + tid] = 0.f; if (OPS == 2) vm[H * BT + tid] = 0.f; }
    if (layer == 0 && BT > 1)                                    // batch columns past B stay zero
        for (int i = tid; i < I * BT; i += kR1Threads) if (i % BT >= B) f32(a.vu[1])[i] = 0.f;
    const uint32_t base = a.epoch[blockIdx.x] + 1u;        // the step number of step 0
    uint32_t above0 = 0;                                   // the progress of the layer above when this call began
    if (layer + 1 < a.L) above0 = ld_relaxed(a.progress + layer + 1);
    __syncthreads();
    bool ok = mbar_wait_bounded(bar, 0);
    if (!ok) *(volatile uint32_t*)a.status = (uint32_t)kDevCopyTimeout;
    if (!__syncthreads_and(ok)) {
        if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
        return;
    }
    const R1Header* hd = reinterpret_cast<const R1Header*>(img);
    const int U0 = hd->op[0].units, U1 = OPS == 2 ? hd->op[OPS - 1].units : 0;
    // places of partial sums that no task writes stay zero; cell state and bias of the CTA's units
#pragma unroll
    for (int op = 0; op < OPS; ++op) for (int i = tid; i < (int)hd->op[op].partials * BT; i += kR1Threads) f32(a.part[op])[i] = 0.f;
    if (kHasC)
        for (int i = tid; i < U0 * BT; i += kR1Threads) {
            const int u = i / BT, b = i % BT;
            cs[i] = a.c0 && b < B ? __ldg(a.c0 + ((size_t)layer * B + b) * H + hd->op[0].unit0 + u) : 0.f;
        }
    const float* bl = a.bias[layer];
    for (int i = tid; i < 4 * U0; i += kR1Threads) {
        const int g = i / U0, u = i % U0;
        f32(a.bias0)[i] = bl && g < (CELL == kR1Gru ? 4 : G0) ? __ldg(bl + (size_t)g * H + hd->op[0].unit0 + u) : 0.f;
    }
    if (OPS == 2)
        for (int u = tid; u < U1; u += kR1Threads) f32(a.bias1)[u] = bl && CELL == kR1GruRb ? __ldg(bl + (size_t)2 * H + hd->op[OPS - 1].unit0 + u) : 0.f;
    struct Walk { const R1Group* g; int n[2]; } wk[OPS];
#pragma unroll
    for (int op = 0; op < OPS; ++op) {
        const uint16_t* wd = reinterpret_cast<const uint16_t*>(img + hd->op[op].warp_off) + warp * 4;
        wk[op].g = reinterpret_cast<const R1Group*>(img + hd->op[op].groups_off) + wd[0];
        wk[op].n[0] = wd[1]; wk[op].n[1] = wd[2];
    }
    // row sums: 2^lp neighbouring lanes per row
    int lp[OPS];
#pragma unroll
    for (int op = 0; op < OPS; ++op) { lp[op] = 0; while (lp[op] < 5 && (hd->op[op].n_rows << (lp[op] + 1)) <= kR1Threads) ++lp[op]; }

    // ---- the exchange.  The first words are asked for early (poll_issue), all are taken in poll_take.
    uint4* ex_state = a.ex[0][layer];
    const int n_state = a.words[0][layer];
    const uint32_t* map_state = a.wmap[0][layer];
    uint4* ex_mid = OPS == 2 ? a.ex[1][layer] : nullptr;
    const int n_mid = OPS == 2 ? a.words[1][layer] : 0;
    const uint32_t* map_mid = OPS == 2 ? a.wmap[1][layer] : nullptr;
    const uint4* ex_below = layer > 0 ? a.ex[0][below] : nullptr;
    const int n_below = layer > 0 ? a.words[0][below] : 0;
    const uint32_t* map_below = layer > 0 ? a.wmap[0][below] : nullptr;
    auto poll_issue = [&](Word (&w)[kW], const uint4* src, int n) {
#pragma unroll
        for (int q = 0; q < kW; ++q) if (tid + q * kR1Threads < n) w[q] = ld_word(src + tid + q * kR1Threads);
    };
    auto take_word = [&](Word w, const uint4* src, const uint32_t* map, int i, uint32_t want, float* dst) {
        unsigned long long t0 = 0;
        unsigned int spins = 0;
        while (word_tag(w) != want) {
            if (*s_ok == 0) { ok = false; break; }         // another thread has given up
            if ((++spins & 63u) == 0) {
                const unsigned long long now = global_ns();
                if (t0 == 0) t0 = now;
                else if (now - t0 > a.limit_ns) { *(volatile uint32_t*)a.status = (uint32_t)kDevBarrierTimeout; *s_ok = 0; ok = false; break; }
            }
            w = ld_word(src + i);
        }
        const uint32_t m = __ldg(map + i);
        float* p = dst + (m & 0xffffffu);
        p[0] = __uint_as_float((uint32_t)w);
        if ((m >> 24) > 1) p[1] = __uint_as_float((uint32_t)(w >> 32));
        if ((m >> 24) > 2) p[2] = __uint_as_float((uint32_t)(w >> 64));
    };
    auto poll_take = [&](Word (&w)[kW], const uint4* src, int n, const uint32_t* map, uint32_t want, float* dst) {
        want += a.never;
#pragma unroll
        for (int q = 0; q < kW; ++q) if (tid + q * kR1Threads < n) take_word(w[q], src, map, tid + q * kR1Threads, want, dst);
        for (int i0 = kW * kR1Threads; i0 < n; i0 += kW * kR1Threads) {
            poll_issue(w, src + i0, n - i0);
#pragma unroll
            for (int q = 0; q < kW; ++q) if (i0 + tid + q * kR1Threads < n) take_word(w[q], src, map, i0 + tid + q * kR1Threads, want, dst);
        }
    };
    // The sums of a product's rows over their partial sums (GRU: input and recurrent part apart).
    auto row_sums = [&](int op) {
        const R1Row* rows = reinterpret_cast<const R1Row*>(img + hd->op[op].rows_off);
        const float* P = f32(a.part[op]);
        float* z = f32(a.z[op]);
        const int n = hd->op[op].n_rows, lanes = 1 << lp[op], s = tid & (lanes - 1);
        for (int r0 = 0; r0 < n; r0 += kR1Threads >> lp[op]) {
            const int r = r0 + (tid >> lp[op]);
            float sum[2][BT];
#pragma unroll
            for (int b = 0; b < BT; ++b) { sum[0][b] = 0.f; sum[1][b] = 0.f; }
            if (r < n) {
                const R1Row d = rows[r];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const float* q = P + (size_t)d.base[p] * 4 * BT;
                    for (int i = s; i < d.quads[p]; i += lanes)
#pragma unroll
                        for (int k = 0; k < BT; ++k) {     // BT float4: four places of BT values
                            const float4 t = *reinterpret_cast<const float4*>(q + ((size_t)i * BT + k) * 4);
                            const float e[4] = {t.x, t.y, t.z, t.w};
                            float* acc = sum[CELL == kR1Gru ? p : 0];
                            if (BT == 1) acc[0] += (e[0] + e[1]) + (e[2] + e[3]);
                            else
#pragma unroll
                                for (int j = 0; j < 4; ++j) acc[(4 * k + j) % BT] += e[j];
                        }
                }
            }
            for (int off = lanes >> 1; off >= 1; off >>= 1)
#pragma unroll
                for (int b = 0; b < BT; ++b) {
                    sum[0][b] += __shfl_xor_sync(0xffffffffu, sum[0][b], off);
                    if (CELL == kR1Gru) sum[1][b] += __shfl_xor_sync(0xffffffffu, sum[1][b], off);
                }
            if (r < n && s == 0)
#pragma unroll
                for (int b = 0; b < BT; ++b) {
                    if (CELL == kR1Gru) {
                        const bool cand = r >= 2 * U0;     // the candidate's two parts stay apart: slots 2 and 3
                        z[r * BT + b] = cand ? sum[0][b] : sum[0][b] + sum[1][b];
                        if (cand) z[(r + U0) * BT + b] = sum[1][b];
                    } else z[r * BT + b] = sum[0][b];
                }
        }
    };
    Word wr[kW] = {}, wi[kW] = {};
    if (layer > 0) {
        poll_issue(wi, ex_below, n_below);
        poll_take(wi, ex_below, n_below, map_below, base, f32(a.vu[0]));
    }
    if (!__syncthreads_and(ok)) {
        if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
        return;
    }
#ifdef CSB_PHASE_CLOCKS
    long long lap[8] = {0, 0, 0, 0, 0, 0, 0, 0}, lap_at = clock64();
#endif
    const int j = lane >> 2, g = lane & 3;                 // gate lanes: four per state, six states per warp and round
    for (int t = 0; t < T_; ++t) {
        const bool more = t + 1 < T_;
        const float* vu = f32(a.vu[t & 1]);
        float* vu_next = f32(a.vu[(t + 1) & 1]);
        // ---- u_t lies in vu: its part of the product, while h_{t-1} and u_{t+1} are on their way
        const uint4* rec_src = ex_state + (size_t)((t - 1) & (kR1Ring - 1)) * n_state;
        const uint4* next_src = ex_below + (size_t)((t + 1) & (kR1Ring - 1)) * n_below;
        if (layer == 0 && more)
            for (int b = 0; b < B; ++b)
                for (int i = tid; i < I; i += kR1Threads) cp_async4(vu_next + i * BT + b, a.x + ((size_t)(t + 1) * B + b) * I + i);
        if (t > 0) poll_issue(wr, rec_src, n_state);
        walk<T, BT>(img, wk[0].g, wk[0].n[0], lane, vu, f32(a.part[0]));
        if (CELL == kR1GruRb) walk<T, BT>(img, wk[OPS - 1].g, wk[OPS - 1].n[0], lane, vu, f32(a.part[1]));
        R1_LAP(0);                                         // product of the input part
        if (t > 0) poll_take(wr, rec_src, n_state, map_state, base + (uint32_t)(t - 1), vr);
        if (layer > 0 && more) poll_issue(wi, next_src, n_below);
        R1_LAP(1);                                         // the state of the step before
        if (!__syncthreads_and(ok)) break;
        R1_LAP(2);
        if (layer > 0 && tid == 0 && (t & (kR1Block - 1)) == kR1Block - 1) atomicAdd(a.progress + layer, 1u);   // u up to step t has been read
        walk<T, BT>(img, wk[0].g + wk[0].n[0], wk[0].n[1], lane, vr, f32(a.part[0]));
        R1_LAP(3);                                         // product of the recurrent part
        if (layer > 0 && more) poll_take(wi, next_src, n_below, map_below, base + (uint32_t)(t + 1), vu_next);
        if (layer == 0 && more) cp_async_wait();
        // before the slots of steps t .. t + 7 are overwritten, the layer above must have read what they
        // hold, steps up to t - 25.  Only the sum over its CTAs of the blocks of 8 they have read is kept:
        // CTAs of one layer are never more than two steps apart, so while one has not finished block k
        // none of the others has finished block k + 1, and the sum is below n k.
        if (layer + 1 < a.L && t >= kR1Ring && (t & (kR1Block - 1)) == 0 && tid == 0) {
            const uint32_t need = (uint32_t)a.layer_ctas[layer + 1] * (uint32_t)((t - kR1Ring + kR1Block) / kR1Block);
            unsigned long long t0 = 0;
            unsigned int spins = 0;
            while (ld_relaxed(a.progress + layer + 1) - above0 < need) {
                if ((++spins & 63u) == 0) {
                    const unsigned long long now = global_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > a.limit_ns) { *(volatile uint32_t*)a.status = (uint32_t)kDevBarrierTimeout; *s_ok = 0; ok = false; break; }
                }
            }
        }
        if (!__syncthreads_and(ok)) break;
        row_sums(0);
        __syncthreads();
        R1_LAP(4);                                         // row sums
        // ---- gates: lane g of a state's four applies gate g
        const int E0 = U0 * BT;
        for (int e0 = warp * kR1WarpUnits; e0 < E0; e0 += kR1Warps * kR1WarpUnits) {
            const int e = e0 + j, l0 = lane & ~3;
            const bool on = j < kR1WarpUnits && e < E0;
            const int u = on ? e / BT : 0, b = on ? e % BT : 0;
            float z = on && g < (CELL == kR1Gru ? 4 : G0) ? f32(a.z[0])[g * E0 + e] + f32(a.bias0)[g * U0 + u] : 0.f;
            const int at = ((int)hd->op[0].unit0 + u) * BT + b;      // the state's element in the staged vectors
            const float hp = CELL == kR1Gru || CELL == kR1Ligru || CELL == kR1GruRb ? vr[at] : 0.f;
            float h, c = 0.f;
            if (kHasC) {
                c = on ? cs[e] : 0.f;
                z = activation(z, g == 2);
                const float zi = __shfl_sync(0xffffffffu, z, l0), zf = __shfl_sync(0xffffffffu, z, l0 + 1);
                const float zc = __shfl_sync(0xffffffffu, z, l0 + 2), zo = __shfl_sync(0xffffffffu, z, l0 + 3);
                c = zf * c + zi * zc;
                h = zo * activation(c, true);
                if (on && g == 0) cs[e] = c;
            } else if (CELL == kR1Gru) {
                if (g < 2) z = activation(z, false);
                const float r = __shfl_sync(0xffffffffu, z, l0), zz = __shfl_sync(0xffffffffu, z, l0 + 1);
                const float ni = __shfl_sync(0xffffffffu, z, l0 + 2), nh = __shfl_sync(0xffffffffu, z, l0 + 3);
                h = (1.f - zz) * activation(ni + r * nh, true) + zz * hp;
            } else if (CELL == kR1Ligru) {
                if (g == 0) z = activation(z, false);
                const float zz = __shfl_sync(0xffffffffu, z, l0), cand = fmaxf(__shfl_sync(0xffffffffu, z, l0 + 1), 0.f);
                h = zz * hp + (1.f - zz) * cand;
            } else {
                z = activation(z, false);
                if (on && g == 1) cs[e] = z;               // the update gate, for the second half of the step
                h = __shfl_sync(0xffffffffu, z, l0) * hp;  // r * h_{t-1}
            }
            const float h1 = __shfl_down_sync(0xffffffffu, h, 4), h2 = __shfl_down_sync(0xffffffffu, h, 8);
            uint4* ex = OPS == 2 ? ex_mid + (size_t)(t & (kR1Ring - 1)) * n_mid : ex_state + (size_t)(t & (kR1Ring - 1)) * n_state;
            if (on && g == 0 && (j == 0 || j == 3) && (OPS == 2 || more || layer + 1 < a.L)) st_word(ex + hd->op[0].word0 + e / 3, h, h1, h2, base + (uint32_t)t);
            if (on && g == 0 && b < B) {
                if (OPS == 1) {
                    if (layer == a.L - 1 && a.y) a.y[((size_t)t * B + b) * S + at / BT] = h;
                    if (!more && a.hT) a.hT[((size_t)layer * B + b) * S + at / BT] = h;
                }
                if (kHasC && !more && a.cT) a.cT[((size_t)layer * B + b) * H + at / BT] = c;
            }
        }
        R1_LAP(5);                                         // gates
        if (OPS == 2) {
            // ---- second product of the step: what the first one gave, from every CTA of the layer
            const uint4* src = ex_mid + (size_t)(t & (kR1Ring - 1)) * n_mid;
            poll_issue(wr, src, n_mid);
            poll_take(wr, src, n_mid, map_mid, base + (uint32_t)t, vm);
            if (!__syncthreads_and(ok)) break;
            R1_LAP(6);                                     // exchange inside the step
            walk<T, BT>(img, wk[OPS - 1].g + wk[OPS - 1].n[0], wk[OPS - 1].n[1], lane, vm, f32(a.part[1]));
            __syncthreads();
            row_sums(OPS - 1);
            __syncthreads();
            const int E1 = U1 * BT;
            for (int e0 = warp * kR1WarpUnits; e0 < E1; e0 += kR1Warps * kR1WarpUnits) {
                const int e = e0 + j;
                const bool on = j < kR1WarpUnits && e < E1;
                const int u = on ? e / BT : 0, b = on ? e % BT : 0, at = ((int)hd->op[OPS - 1].unit0 + u) * BT + b;
                float h = on ? f32(a.z[1])[e] + f32(a.bias1)[u] : 0.f;
                if (CELL == kR1GruRb && on) { const float zz = cs[e]; h = (1.f - zz) * activation(h, true) + zz * vr[at]; }
                const float h1 = __shfl_down_sync(0xffffffffu, h, 4), h2 = __shfl_down_sync(0xffffffffu, h, 8);
                if (on && g == 0 && (j == 0 || j == 3) && (more || layer + 1 < a.L))
                    st_word(ex_state + (size_t)(t & (kR1Ring - 1)) * n_state + hd->op[OPS - 1].word0 + e / 3, h, h1, h2, base + (uint32_t)t);
                if (on && g == 0 && b < B) {
                    if (layer == a.L - 1 && a.y) a.y[((size_t)t * B + b) * S + at / BT] = h;
                    if (!more && a.hT) a.hT[((size_t)layer * B + b) * S + at / BT] = h;
                }
            }
            R1_LAP(7);                                     // second product, its sums and gates
        }
    }
#ifdef CSB_PHASE_CLOCKS
    if (tid == 0) for (int i = 0; i < 8; ++i) a.clocks[(size_t)blockIdx.x * 8 + i] = lap[i];
#endif
    if (tid == 0) a.epoch[blockIdx.x] = base - 1u + (uint32_t)T_;
}

template <typename T, int BT>
static const void* pick_kernel(int cell) {
    switch (cell) {
        case kR1Lstm: return (const void*)csb_rnn1_kernel<T, kR1Lstm, BT>;
        case kR1Gru: return (const void*)csb_rnn1_kernel<T, kR1Gru, BT>;
        case kR1Lstmp: return (const void*)csb_rnn1_kernel<T, kR1Lstmp, BT>;
        case kR1Ligru: return (const void*)csb_rnn1_kernel<T, kR1Ligru, BT>;
        default: return (const void*)csb_rnn1_kernel<T, kR1GruRb, BT>;
    }
}

}  // namespace csb
